"""Compressed products of so many columns that their cross sums take several passes (256 MB each), the last one ragged.

Against the same columns in narrow blocks: sums of FP64 products in another order, 1e-12 of a column.
"""

import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1803_08333_gb300 as rf  # noqa: E402


@pytest.mark.parametrize("which,cols", [("T_A", 6003), ("V", 9001)])
def test_passes(which, cols):
    from paper_1803_08333_gb300 import build

    build.build()
    m = synth.geodesic_sphere(10)
    op = rf.Operator(rf.Context(0), m.verts, m.tris, 0.5, scaling="k")
    H = rf.Compressed(op, eps=1e-6, leaf=16)
    n = op.N if which == "T_A" else op.nc
    g = torch.Generator(device="cuda").manual_seed(cols)
    x = torch.complex(torch.randn(cols, n, dtype=torch.float64, device="cuda", generator=g),
                      torch.randn(cols, n, dtype=torch.float64, device="cuda", generator=g))
    launched = rf.launch_count()
    y = H.apply(which, x)
    assert rf.launch_count() - launched >= 6  # three kernels a pass
    for c in list(range(0, cols, 997)) + [cols - 4, cols - 3, cols - 1]:
        ref = H.apply(which, x[c : c + 3])
        got = y[c : c + 3]
        assert (torch.linalg.norm(got - ref, dim=1) <= 1e-12 * torch.linalg.norm(ref, dim=1)).all(), c
    H.close()
