"""Accurate products of blocks with a NaN, an infinite and a huge column: 5 to 32 columns take the integer sums, 33 and more the
FP64 ones.

A column with a value that is not finite has no digits: its products are NaN; the others are what they are without it,
to the last bit.
"""

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1803_08333_gb300 as rf  # noqa: E402


@pytest.mark.parametrize("cols", [5, 8, 32, 33, 40])
def test_columns_that_are_not_finite(cols):
    from paper_1803_08333_gb300 import build

    build.build()
    m = synth.geodesic_sphere(5)
    op = rf.Operator(rf.Context(0), m.verts, m.tris, 0.7, scaling="k")
    rng = np.random.default_rng(cols)
    x = rng.standard_normal((cols, op.N)) + 1j * rng.standard_normal((cols, op.N))
    x[0] *= 1e-200  # scales of both signs
    x[3] *= 1e200
    x = torch.from_numpy(x).cuda()
    y = x.clone()
    y[1, 7] = complex(float("nan"), 0.0)
    y[cols - 1, op.N - 1] = complex(0.0, float("-inf"))
    keep = [c for c in range(cols) if c not in (1, cols - 1)]
    got, want = op.apply("T_A", y), op.apply("T_A", x)
    assert torch.equal(torch.view_as_real(got[keep]), torch.view_as_real(want[keep]))
    assert torch.isfinite(torch.view_as_real(want)).all()
    # T_A mixes the real and the imaginary part of a column
    assert torch.isnan(torch.view_as_real(got[1])).all() and torch.isnan(torch.view_as_real(got[cols - 1])).all()
