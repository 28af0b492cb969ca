"""Device memory of a compression: what the build holds at its peak is what it says it needs, with a budget and without.

The smallest budget that a build accepts is found from its own refusals, which name the bytes they lack.
"""

import gc
import re

import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1803_08333_gb300 as rf  # noqa: E402


def _peak(op, **opts):
    gc.collect()
    rf.pool_trim()  # earlier frees are counted
    rf.pool_reset_high()
    before = rf.pool_stats()["used"]
    h = rf.Compressed(op, **opts)
    torch.cuda.synchronize()
    s = rf.pool_stats()
    h.close()
    return s["used_high"] - before, s["used"] - before


# slots of many crosses; of one; no admissible block at all
@pytest.mark.parametrize("level,leaf,max_rank", [(10, 32, 256), (8, 8, 64), (7, 16, 1), (4, 1000, 64), (9, 600, 64)])
def test_peak_is_the_stated_one(level, leaf, max_rank):
    from paper_1803_08333_gb300 import build

    build.build()
    m = synth.geodesic_sphere(level)
    opts = {"leaf": leaf, "max_rank": max_rank}
    free = rf.Context(0)
    op = rf.Operator(free, m.verts, m.tris, 0.5, scaling="k")
    base = free.bytes_in_use()
    unbounded, held = _peak(op, **opts)
    budget = base + 4096
    for _ in range(3):  # T_A's refusal, V's, none
        ctx = rf.Context(0, hbm_budget_bytes=budget)
        op = rf.Operator(ctx, m.verts, m.tris, 0.5, scaling="k")
        assert ctx.bytes_in_use() == base
        try:
            bounded, _ = _peak(op, **opts)
            break
        except rf.RfcmpError as e:
            need, left = map(int, re.search(r"up to (\d+) bytes, budget has (\d+)", str(e)).groups())
            budget += need - left
    else:
        pytest.fail("the build refuses the bytes that it asked for")
    assert held <= bounded <= budget - base
    assert unbounded <= budget - base
