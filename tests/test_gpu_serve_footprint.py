"""The bytes the server reserves for an operator and its solves bound what they take from the device's pool."""

import gc

import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1803_08333_gb300 as rf  # noqa: E402
from paper_1803_08333_gb300 import serve  # noqa: E402


@pytest.mark.parametrize("level", [4, 8, 16])
@pytest.mark.parametrize("cols,session", [(1, 0), (4, 0), (16, 0), (32, 0), (64, 0), (64, 1)])
def test_bound(level, cols, session):
    from paper_1803_08333_gb300 import build

    build.build()
    m = synth.geodesic_sphere(level)
    ctx = rf.Context(0)
    gc.collect()
    rf.pool_trim()
    rf.pool_reset_high()
    before = rf.pool_stats()["used"]
    op = rf.Operator(ctx, m.verts, m.tris, 1.0)
    torch.cuda.synchronize()
    assert rf.pool_stats()["used_high"] - before <= serve.op_footprint(op.nv, op.nc, 1, with_factors=True)
    op.solve(op.rhs_planewave(*synth.random_plane_waves(1, seed=1)))
    kh, pol = synth.random_plane_waves(cols, seed=2)
    e = op.rhs_planewave(kh, pol)
    torch.cuda.synchronize()
    rf.pool_trim()  # earlier frees are counted
    rf.pool_reset_high()
    before = rf.pool_stats()["used"]
    if session:
        b = op.batch(cols)
        b.admit(e)
        b.step()
    else:
        op.solve(e)
    torch.cuda.synchronize()
    grown = rf.pool_stats()["used_high"] - before
    if session:
        b.close()
    assert grown <= serve.op_footprint(op.nv, op.nc, cols, with_factors=True, widest=1)
