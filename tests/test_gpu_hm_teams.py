"""The compressed product with 8, 4, 2 and 1 CTAs a row tile.

Against the product with the exported matrix: 3 eps, as the other tests of the compressed form, and 1e-12 where one dense
block holds all (n products in FP64).  The same bits on every run.
"""

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1803_08333_gb300 as rf  # noqa: E402


@pytest.mark.parametrize("level,leaf,eps,cols", [(3, 8, 1e-4, 1), (5, 1000, 1e-4, 5), (6, 32, 1e-10, 4), (10, 32, 1e-4, 4),
                                                 (10, 32, 1e-4, 9), (12, 16, 1e-8, 16)])
def test_product_of_teams(level, leaf, eps, cols):
    from paper_1803_08333_gb300 import build

    build.build()
    m = synth.geodesic_sphere(level)
    op = rf.Operator(rf.Context(0), m.verts, m.tris, 0.5, scaling="k")
    H = rf.Compressed(op, eps=eps, leaf=leaf, max_rank=128)
    rng = np.random.default_rng(cols)
    for which, n in (("T_A", op.N), ("V", op.nc)):
        M = op.export(which).to(torch.complex128)
        x = torch.from_numpy(rng.standard_normal((cols, n)) + 1j * rng.standard_normal((cols, n))).cuda()
        y, ref = H.apply(which, x), x @ M.T
        tol = 1e-12 if leaf >= n else max(3 * eps, 1e-6)  # the crosses are stored in 32 bits
        err = (torch.linalg.norm(y - ref, dim=1) / torch.linalg.norm(ref, dim=1)).max().item()
        assert err <= tol, (which, err)
        assert torch.equal(y, H.apply(which, x))
    H.close()
