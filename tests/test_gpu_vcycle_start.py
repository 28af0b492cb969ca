"""(Sigma^T Sigma)^+ from the V-cycle built as a matrix: one to several levels, rows in groups of four and (a coarse level
of more than 7040 rows) of two, ragged last groups, open and closed surfaces.

The result must not need the conjugate-gradient start (factor_iterations_lplus counts its steps), is exactly symmetric,
and rows of (L + J) (X + J) - I vanish to rounding: 1e-11 as the other factor tests.
"""

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1803_08333_gb300 as rf  # noqa: E402

MESHES = {"f4": lambda: synth.geodesic_sphere(4), "f11": lambda: synth.geodesic_sphere(11),
          "plate": lambda: synth.plate(31), "torus": lambda: synth.torus(60, 7), "f40": lambda: synth.geodesic_sphere(40)}


@pytest.mark.parametrize("mesh,cut", [("f4", 0), ("f4", 1), ("f11", 3), ("plate", 0), ("torus", 0), ("f40", 1)])
def test_start(mesh, cut):
    from paper_1803_08333_gb300 import build

    build.build()
    m = MESHES[mesh]()
    op = rf.Operator(rf.Context(0), m.verts, m.tris[: len(m.tris) - cut], 1.0, scaling="k")
    assert op.info().factor_iterations_lplus == 0
    X = op.export("LPLUS")
    assert torch.equal(X, X.T)
    _, ec = op.edges()
    n = op.nc
    a, b = (ec[:, i].astype(np.int64) for i in (0, 1))
    rows = np.arange(0, n, max(1, n // 40))
    M = torch.full((len(rows), n), 1.0 / n, dtype=torch.float64)
    at = {c: r for r, c in enumerate(rows)}
    for p, q in zip(np.concatenate([a, b]), np.concatenate([b, a])):
        if p in at:
            M[at[p], p] += 1.0
            M[at[p], q] -= 1.0
    R = M.cuda() @ X  # (L + J) X = (L + J) (X + J) - J = I - J
    R += 1.0 / n
    R[torch.arange(len(rows), device="cuda"), torch.from_numpy(rows).cuda()] -= 1.0
    assert R.abs().max().item() <= 1e-11
