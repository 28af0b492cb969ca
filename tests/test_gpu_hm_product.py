"""The compressed product over its row tiles and cross items: ragged tiles, groups of one to four
columns, clusters smaller and larger than a tile, and blocks that all stay dense.

With a leaf size of at least n the compressed matrix is one dense block, so the product is an FP64
sum of n products of the exported entries: error at most about n 2^-53 of the sum of absolute
terms, held to 1e-12.  With crosses it is held to 3 eps, as the other tests of the compressed form.
"""

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1803_08333_gb300 as rf  # noqa: E402

EPS = 1e-4


@pytest.mark.parametrize("mesh,leaf,cols", [("f5", 1024, 1), ("f5", 1024, 6), ("f5", 8, 2), ("plate", 33, 7),
                                            ("plate", 40, 3), ("plate", 8, 4), ("f8", 64, 9)])
def test_product_over_tiles_and_column_groups(mesh, leaf, cols):
    from paper_1803_08333_gb300 import build

    build.build()
    m = {"f5": lambda: synth.geodesic_sphere(5), "f8": lambda: synth.geodesic_sphere(8),
         "plate": lambda: synth.plate(17)}[mesh]()
    op = rf.Operator(rf.Context(0), m.verts, m.tris, 0.5, scaling="k")
    H = rf.Compressed(op, eps=EPS, leaf=leaf)
    rng = np.random.default_rng(cols)
    for which, n in (("T_A", op.N), ("V", op.nc)):
        M = op.export(which).to(torch.complex128)
        x = torch.from_numpy(rng.standard_normal((cols, n)) + 1j * rng.standard_normal((cols, n))).cuda()
        y, ref = H.apply(which, x), x @ M.T
        tol = 1e-12 if leaf >= n else 3 * EPS
        err = (torch.linalg.norm(y - ref, dim=1) / torch.linalg.norm(ref, dim=1)).max().item()
        assert err <= tol, (which, err)
        assert torch.equal(y, H.apply(which, x))  # no sum depends on the order CTAs run in
        one = torch.cat([H.apply(which, x[c]) for c in range(cols)])
        assert torch.linalg.norm(one - y) <= 1e-12 * torch.linalg.norm(y)
    H.close()
