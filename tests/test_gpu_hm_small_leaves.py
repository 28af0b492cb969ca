"""The compressed product on tiles of at most 8 and 16 rows, whose entries share warps two and four at a time where there
are more of them than warps.

Against the product with the exported matrix: 3 eps, as the other tests of the compressed form.  The same bits on every run.
"""

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1803_08333_gb300 as rf  # noqa: E402


@pytest.mark.parametrize("level,leaf,eps,cols", [(7, 8, 1e-4, 13), (11, 8, 1e-4, 1), (11, 12, 1e-6, 3), (10, 16, 1e-4, 22),
                                                 (10, 24, 1e-4, 40)])
def test_product(level, leaf, eps, cols):
    from paper_1803_08333_gb300 import build

    build.build()
    m = synth.geodesic_sphere(level)
    op = rf.Operator(rf.Context(0), m.verts, m.tris, 0.5, scaling="k")
    H = rf.Compressed(op, eps=eps, leaf=leaf)
    rng = np.random.default_rng(cols)
    for which, n in (("T_A", op.N), ("V", op.nc)):
        M = op.export(which).to(torch.complex128)
        x = torch.from_numpy(rng.standard_normal((cols, n)) + 1j * rng.standard_normal((cols, n))).cuda()
        y, ref = H.apply(which, x), x @ M.T
        err = (torch.linalg.norm(y - ref, dim=1) / torch.linalg.norm(ref, dim=1)).max().item()
        assert err <= max(3 * eps, 1e-6), (which, err)
        assert torch.equal(y, H.apply(which, x))
    H.close()
