"""RCS of so many currents that their cell sums take two passes (256 MB each), the last one ragged and of other groups.

Against the same currents in narrow calls: FP64 sums in another order, 1e-9 dB off the nulls.
"""

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1803_08333_gb300 as rf  # noqa: E402


@pytest.mark.parametrize("cols,ndir", [(437, 3), (866, 1)])
def test_passes(cols, ndir):
    from paper_1803_08333_gb300 import build

    build.build()
    m = synth.geodesic_sphere(22)
    op = rf.Operator(rf.Context(0), m.verts, m.tris, 1.0, scaling="k")
    j = op.rhs_planewave(*synth.random_plane_waves(cols, seed=3))
    u = np.random.default_rng(ndir).standard_normal((ndir, 3))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    got = op.farfield(j, u)
    for c in (0, 61, 428, 432, cols - 2):
        ref = op.farfield(j[c : c + 2], u)
        keep = ref > ref.max() - 40.0
        assert np.abs(got[c : c + 2] - ref)[keep].max() <= 1e-9
