"""Near pairs whose outer quadrature point is a corner of the source cell: a closed flat body with one cell on one side
and three on the other, which meet at its centroid (the rule's first point).

On an edge's line every term with the edge's logarithm has a vanishing factor, so the entries are finite; FP64 integrals
stored as FP32, 1e-6 entrywise and 1e-5 in the norm as in the other near-entry tests.
"""

import numpy as np
import pytest

from oracle import efie

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1803_08333_gb300 as rf  # noqa: E402

TRIS = np.array([[0, 1, 2], [1, 0, 3], [2, 1, 3], [0, 2, 3]], np.int32)


@pytest.mark.parametrize("k,turn", [(1.0, 0), (1e-3, 1), (0.3, 2)])
def test_corner_at_a_quadrature_point(k, turn):
    from paper_1803_08333_gb300 import build

    build.build()
    v = np.roll(np.array([[0, 0, 0], [3, 0, 0], [0, 3, 0], [1, 1, 0]], np.float64), turn, axis=1)
    D = efie.discretize(v, TRIS)
    assert (D.qp[0, 0] == v[3]).all()
    TA, V = efie.assemble(D, k)
    op = rf.Operator(rf.Context(0), v, TRIS, k, scaling="k")
    gV = op.export("V").cpu().numpy().astype(np.complex128)
    gT = op.export("T_A").cpu().numpy().astype(np.complex128)
    assert np.isfinite(gV).all() and np.isfinite(gT).all()
    assert (np.abs(gV - V) / np.abs(V)).max() <= 1e-6
    assert np.linalg.norm(gT - TA) <= 1e-5 * np.linalg.norm(TA)
