"""Inner products of 4 to 65 columns on the split-BF16 GEMM with the K blocks of all row tiles dealt out in equal
shares: fewer and more row tiles than SMs, ragged tiles, one to many slots a tile, each tile width.

Against the accurate products: a BF16x3 product is good to about 2^-16, and A chains nine of them: 1e-3.
Against the same products with whole tiles a CTA (a column tile of 32 gives several column tiles, which are not
shared out): the FP32 sums differ in order only, nine times: 1e-4.
"""

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1803_08333_gb300 as rf  # noqa: E402


@pytest.mark.parametrize("level,cols", [(2, 4), (4, 4), (4, 24), (7, 16), (9, 17), (9, 32), (9, 33), (16, 8), (16, 64),
                                        (18, 24), (20, 20), (20, 65)])
def test_inner_products(level, cols):
    from paper_1803_08333_gb300 import build

    build.build()
    m = synth.geodesic_sphere(level)
    op = rf.Operator(rf.Context(0), m.verts, m.tris, 0.7, scaling="k")
    x = torch.from_numpy(np.random.default_rng(cols).standard_normal((cols, op.N, 2)).view(np.complex128)[..., 0])
    x = x.cuda()
    op.set_plan({"mrhs_min": 1})
    got = op.apply("A_INNER", x)
    ref = op.apply("A", x)
    rel = torch.linalg.norm(got - ref, dim=1) / torch.linalg.norm(ref, dim=1)
    assert rel.max().item() <= 1e-3
    if cols > 16:
        op.set_plan({"mrhs_min": 1, "gemm_bn": 32})
        whole = op.apply("A_INNER", x)
        rel = torch.linalg.norm(got - whole, dim=1) / torch.linalg.norm(whole, dim=1)
        assert rel.max().item() <= 1e-4
