"""The start of (Sigma^T Sigma)^+ with groups of four, two and one rows of the V-cycle built as a matrix, and with the cycle
on columns, which operators take by size: the same matrix.

FP64 sums of up to some 10^4 terms in another order: 1e-11 of the largest entry, as the other factor tests.
"""

import ctypes

import numpy as np
import pytest

import synth
from oracle import efie

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1803_08333_gb300 as rf  # noqa: E402

MESHES = {"f2": lambda: synth.geodesic_sphere(2), "f11": lambda: synth.geodesic_sphere(11), "plate": lambda: synth.plate(31),
          "torus": lambda: synth.torus(60, 7)}


@pytest.mark.parametrize("mesh,cut", [("f2", 0), ("f2", 1), ("f11", 3), ("plate", 0), ("torus", 0)])
def test_groups_of_rows(mesh, cut):
    from paper_1803_08333_gb300 import build

    build.build()
    m = MESHES[mesh]()
    S = efie.discretize(m.verts, m.tris[: len(m.tris) - cut]).Sigma
    A = (S.T @ S).tocsr()
    A.sort_indices()
    n = A.shape[0]
    ptr, col, val = A.indptr.astype(np.int32), A.indices.astype(np.int32), A.data.astype(np.float64)
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    X = {}
    for rows in (0, 1, 2, 4):
        X[rows] = torch.full((n, n), float("nan"), dtype=torch.float64, device="cuda")
        assert rf.lib().rfcmp_vcycle_start(p(ptr), p(col), p(val), n, rows, X[rows].data_ptr()) == 0
    big = X[0].abs().max().item()
    for rows in (1, 2, 4):
        assert torch.equal(X[rows], X[rows].T)
        assert (X[rows] - X[0]).abs().max().item() <= 1e-11 * big
    # an approximate inverse: the cycle contracts
    D = torch.from_numpy(A.toarray()).cuda() + 1.0 / n
    E = torch.eye(n, dtype=torch.float64, device="cuda") - X[4] @ D
    v = E.clone()
    for _ in range(6):
        v = v @ v
        v /= v.abs().max()
    assert (torch.linalg.norm(E @ v) / torch.linalg.norm(v)).item() < 1.0
