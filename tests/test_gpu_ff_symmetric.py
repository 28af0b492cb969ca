"""Accurate products of 1 to 4 columns on the float-float GEMV, which reads the upper triangle of a symmetric
matrix, against FP64 products of the library's own stored matrices.

A product's terms carry 48 bits and its partial sums meet in FP64 after at most 128 of them: below
1e-12 of the norm over the sizes here.  They hit one tile, ragged rows and segments (512 complex entries, 1024 of
a factor), several segments and several columns.
"""

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1803_08333_gb300 as rf  # noqa: E402

MESHES = {"torus": lambda: synth.torus(3, 5, jitter=0.02), "f4": lambda: synth.geodesic_sphere(4),
          "f5": lambda: synth.geodesic_sphere(5), "plate": lambda: synth.plate(19),
          "f9": lambda: synth.geodesic_sphere(9)}


@pytest.mark.parametrize("mesh,cols", [("torus", 1), ("torus", 2), ("f4", 3), ("f5", 1), ("f5", 2), ("plate", 2),
                                       ("plate", 4), ("f9", 1), ("f9", 3)])
def test_accurate_gemv(mesh, cols):
    from paper_1803_08333_gb300 import build

    build.build()
    m = MESHES[mesh]()
    k = 0.7
    outer = "sigma" if mesh == "plate" else "gsigma"
    op = rf.Operator(rf.Context(0), m.verts, m.tris, k, scaling="k", outer=outer)
    op.set_plan({"mrhs_min": 65536, "exact_min": 65536})
    x = torch.from_numpy(np.random.default_rng(cols).standard_normal((cols, op.N, 2)).view(np.complex128)[..., 0])
    x = x.cuda()
    for f in ["T_A", "V", "LPLUS", "GLL_INV"] + ["GTP_INV"] * (outer == "gsigma"):  # what half of a matrix relies on
        M = op.export(f)
        assert torch.equal(M, M.T), f
    TA, V, Lp = (op.export(w).to(torch.complex128) for w in ("T_A", "V", "LPLUS"))
    _, ec = op.edges()
    S = torch.zeros((op.N, op.nc), dtype=torch.complex128, device="cuda")
    at = torch.arange(op.N, device="cuda")
    S[at, torch.from_numpy(ec[:, 0].astype(np.int64)).cuda()] = 1
    S[at, torch.from_numpy(ec[:, 1].astype(np.int64)).cuda()] = -1
    s = x @ S
    want = {"T_A": x @ TA.T, "T_PHI": s @ V.T @ S.T,
            "T_ADJ": -1j * k * (x @ TA.conj().T) + 1j / k * (s @ V.conj().T @ S.T)}
    got = {w: op.apply(w, x) for w in want}
    want["P_SIGMA"], got["P_SIGMA"] = s @ Lp.T @ S.T, op.precondition("P_SIGMA", x)
    for w in want:
        for c in range(cols):
            assert (torch.linalg.norm(got[w][c] - want[w][c]) / torch.linalg.norm(want[w][c])).item() <= 1e-12, (w, c)
