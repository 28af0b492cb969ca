"""Near-pair entries of V where the closed-form integrals meet their special cases: coplanar cells (no
solid angle, points on the extension of an edge), slivers, sharp edges, a count of pairs that is no
multiple of a block's.

The integrals are FP64 and the entries are stored as FP32: relative 1e-6 entrywise, the tolerance of the
other near-entry parity test.
"""

import numpy as np
import pytest

import synth
from oracle import efie

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1803_08333_gb300 as rf  # noqa: E402

MESHES = {"flat": lambda: synth.plate(4, jitter=0.0), "plate": lambda: synth.plate(5),
          "sliver": lambda: synth.ellipsoid(3, axes=(1.0, 0.9, 0.02)), "cube": lambda: synth.cube(2, jitter=0.0),
          "torus": lambda: synth.torus(9, 3)}


@pytest.mark.parametrize("mesh,k", [("flat", 1.0), ("plate", 1e-4), ("sliver", 0.5), ("cube", 2.0), ("torus", 1e-3)])
def test_near_entries(mesh, k):
    from paper_1803_08333_gb300 import build

    build.build()
    m = MESHES[mesh]()
    D = efie.discretize(m.verts, m.tris)
    TA, V = efie.assemble(D, k)
    op = rf.Operator(rf.Context(0), m.verts, m.tris, k, scaling="k")
    gV = op.export("V").cpu().numpy().astype(np.complex128)
    a, b = D.near[:, 0], D.near[:, 1]
    assert np.isfinite(gV).all()
    assert (np.abs(gV[a, b] - V[a, b]) / np.abs(V[a, b])).max() <= 1e-6
    gT = op.export("T_A").cpu().numpy().astype(np.complex128)
    assert np.linalg.norm(gT - TA) <= 1e-5 * np.linalg.norm(TA)
