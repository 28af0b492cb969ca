"""(Sigma^T Sigma)^+ from the fixed-point residual: odd cell counts, cells with fewer than three neighbours,
and a row of more than 14000 cells (twice the threads).

Both sides are the pseudo-inverse to rounding; held to 1e-11 as the other factor parity test.
"""

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1803_08333_gb300 as rf  # noqa: E402


def _cut(level, cells):  # a sphere with its last cells left out: boundary, odd counts
    m = synth.geodesic_sphere(level)
    return m.verts, m.tris[: len(m.tris) - cells]


@pytest.mark.parametrize("mesh", ["sphere", "odd", "plate", "long"])
def test_laplacian_factor(mesh):
    from paper_1803_08333_gb300 import build

    build.build()
    if mesh == "sphere":
        m = synth.geodesic_sphere(4)
        v, t = m.verts, m.tris
    elif mesh == "odd":
        v, t = _cut(5, 1)
    elif mesh == "plate":
        m = synth.plate(13)
        v, t = m.verts, m.tris
    else:
        m = synth.torus(170, 43)  # 14620 cells
        v, t = m.verts, m.tris
    op = rf.Operator(rf.Context(0), v, t, 1.0, scaling="k")
    X = op.export("LPLUS")
    _, ec = op.edges()
    L = torch.zeros((op.nc, op.nc), dtype=torch.float64, device="cuda")
    a, b = (torch.from_numpy(ec[:, i].astype(np.int64)).cuda() for i in (0, 1))
    one = torch.ones(op.N, dtype=torch.float64, device="cuda")
    for r, c, w in ((a, a, one), (b, b, one), (a, b, -one), (b, a, -one)):
        L.index_put_((r, c), w, accumulate=True)
    M = L + 1.0 / op.nc
    if mesh == "long":  # M X - I on some rows
        rows = torch.arange(0, op.nc, 997, device="cuda")
        R = M[rows] @ (X + 1.0 / op.nc)
        R[torch.arange(len(rows), device="cuda"), rows] -= 1.0
        assert R.abs().max().item() <= 1e-11
    else:
        ref = torch.linalg.inv(M) - 1.0 / op.nc
        assert (torch.linalg.norm(X - ref) / torch.linalg.norm(ref)).item() <= 1e-11
    assert torch.equal(X, X.T)
