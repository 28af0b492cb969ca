"""Accurate products of 4 to 33 columns (integer sums up to 32, FP64 ones above) against
FP64 products of the library's own stored matrices.

Six digits of 8 bits under a power-of-two scale per row and per column truncate each term at about
2^-48 of the row and column maxima; over n terms that stays below 1e-11 of the product.  The shapes
hit one and several row tiles, ragged rows and K, one and two column tiles (16 and 32 wide), and
split and unsplit K ranges.
"""

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1803_08333_gb300 as rf  # noqa: E402

MESHES = {"torus": lambda: synth.torus(3, 5, jitter=0.02), "f5": lambda: synth.geodesic_sphere(5),
          "plate": lambda: synth.plate(27), "f13": lambda: synth.geodesic_sphere(13)}


def _rel(a, b):
    big = b.abs().max()  # the squares of the smallest and largest columns leave the FP64 range
    a, b = a / big, b / big
    return (torch.linalg.norm(a - b) / torch.linalg.norm(b)).item()


@pytest.mark.parametrize("mesh,cols", [("torus", 4), ("torus", 8), ("f5", 5), ("f5", 8), ("f5", 9), ("plate", 16),
                                       ("plate", 17), ("f13", 4), ("f13", 8), ("f13", 24), ("f13", 32), ("f5", 33)])
def test_narrow_accurate_products(mesh, cols):
    from paper_1803_08333_gb300 import build

    build.build()
    m = MESHES[mesh]()
    op = rf.Operator(rf.Context(0), m.verts, m.tris, 0.7, scaling="k")
    rng = np.random.default_rng(cols)
    # columns of very different sizes, one of them zero
    x = rng.standard_normal((cols, op.N)) + 1j * rng.standard_normal((cols, op.N))
    x *= 10.0 ** rng.uniform(-200, 200, (cols, 1))
    x[cols // 2] = 0
    x = torch.from_numpy(x).cuda()
    TA, V, Lp = (op.export(w).to(torch.complex128) for w in ("T_A", "V", "LPLUS"))
    _, ec = op.edges()
    S = torch.zeros((op.N, op.nc), dtype=torch.complex128, device="cuda")
    at = torch.arange(op.N, device="cuda")
    S[at, torch.from_numpy(ec[:, 0].astype(np.int64)).cuda()] = 1
    S[at, torch.from_numpy(ec[:, 1].astype(np.int64)).cuda()] = -1
    k = 0.7
    s = x @ S
    want = {"T_A": x @ TA.T, "T_PHI": s @ V.T @ S.T,
            "T_ADJ": -1j * k * (x @ TA.conj().T) + 1j / k * (s @ V.conj().T @ S.T)}
    got = {w: op.apply(w, x) for w in want}
    want["P_SIGMA"], got["P_SIGMA"] = s @ Lp.T @ S.T, op.precondition("P_SIGMA", x)
    for w in want:
        assert torch.count_nonzero(got[w][cols // 2]) == 0
        for c in range(cols):
            if c != cols // 2:
                assert _rel(got[w][c], want[w][c]) <= 1e-11, (w, c, _rel(got[w][c], want[w][c]))
