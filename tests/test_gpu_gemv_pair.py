"""T_A and V in one launch: T and T^H of one column against FP64 products of the stored matrices (1e-12, as the single
products in float-float), and the inner form of A of one and two columns against the accurate one (nine FP32 products in
a chain: 1e-4).  From fewer work units than CTAs (45 functions) to many a CTA."""

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1803_08333_gb300 as rf  # noqa: E402

MESHES = {"torus": lambda: synth.torus(3, 5, jitter=0.02), "f4": lambda: synth.geodesic_sphere(4),
          "f5": lambda: synth.geodesic_sphere(5), "plate": lambda: synth.plate(19),
          "f13": lambda: synth.geodesic_sphere(13)}


@pytest.mark.parametrize("mesh", list(MESHES))
def test_pairs(mesh):
    from paper_1803_08333_gb300 import build

    build.build()
    m = MESHES[mesh]()
    k = 0.7
    op = rf.Operator(rf.Context(0), m.verts, m.tris, k, scaling="k")
    rng = np.random.default_rng(3)
    x = torch.from_numpy(rng.standard_normal((2, op.N)) + 1j * rng.standard_normal((2, op.N))).cuda()
    TA, V = (op.export(w).to(torch.complex128) for w in ("T_A", "V"))
    _, ec = op.edges()
    S = torch.zeros((op.N, op.nc), dtype=torch.complex128, device="cuda")
    at = torch.arange(op.N, device="cuda")
    S[at, torch.from_numpy(ec[:, 0].astype(np.int64)).cuda()] = 1
    S[at, torch.from_numpy(ec[:, 1].astype(np.int64)).cuda()] = -1
    s = x[0] @ S
    want = {"T": 1j * k * (TA @ x[0]) - 1j / k * (S @ (V @ s)),
            "T_ADJ": -1j * k * (TA.conj() @ x[0]) + 1j / k * (S @ (V.conj() @ s))}
    for w in want:
        got = op.apply(w, x[0])[0]
        assert (torch.linalg.norm(got - want[w]) / torch.linalg.norm(want[w])).item() <= 1e-12, w
    for cols in (1, 2):
        ref, got = op.apply("A", x[:cols]), op.apply("A_INNER", x[:cols])
        assert (torch.linalg.norm(got - ref, dim=1) / torch.linalg.norm(ref, dim=1)).max().item() <= 1e-4
