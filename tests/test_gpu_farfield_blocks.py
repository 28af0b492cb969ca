"""The radiation vector over its column groups (one, four, eight, a second pass beyond 64), chunks of
cells (fewer than a block, ragged, several) and phase branches (short polynomials, general series),
against the oracle's radiation integral of the same currents.

Both sides are FP64 sums of the same terms; the RCS agrees to 1e-6 dB within 40 dB of its peak, the
tolerance of the other far-field parity tests.
"""

import numpy as np
import pytest

import synth
from oracle import efie, farfield

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1803_08333_gb300 as rf  # noqa: E402

MESHES = {"ico": lambda: synth.geodesic_sphere(1, seed=9), "f5": lambda: synth.geodesic_sphere(5),
          "plate": lambda: synth.plate(9)}


@pytest.mark.parametrize("mesh,k,cols,ndir", [("ico", 2.5, 1, 1), ("ico", 30.0, 3, 7), ("f5", 1e-4, 4, 5),
                                              ("f5", 0.6, 5, 181), ("plate", 2.0, 8, 13), ("f5", 12.0, 9, 6),
                                              ("plate", 0.2, 66, 3)])
def test_radiation_over_groups_and_chunks(mesh, k, cols, ndir):
    from paper_1803_08333_gb300 import build

    build.build()
    m = MESHES[mesh]()
    D = efie.discretize(m.verts, m.tris)
    op = rf.Operator(rf.Context(0), m.verts, m.tris, k, scaling="k")
    e = op.rhs_planewave(*synth.random_plane_waves(cols, seed=cols))
    dirs = farfield.cut_directions(np.linspace(0.1, 3.0, ndir), 0.3)
    got = op.farfield(e, dirs)
    assert got.shape == (cols, ndir)
    for c in range(cols):
        ref = farfield.bistatic_rcs(D, e[c].cpu().numpy(), k, dirs)
        keep = ref > ref.max() * 1e-4
        assert np.abs(got[c][keep] - 10 * np.log10(ref[keep])).max() <= 1e-6
    assert np.array_equal(got, op.farfield(e, dirs))  # fixed-order sums
