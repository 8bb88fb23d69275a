"""The ordered projection at the edges of its tiles (8192 rows) and of the 64
tiles one sum covers, from no match to every row, and past its capacity.  Rows
are copies of table rows and must equal the oracle's, in table order."""
import numpy as np
import pytest

from paper_1709_00700_gb300 import datagen, pv, workloads
from tests.gpu_util import assert_same, register, want

pytestmark = pytest.mark.gpu

SUPER = 64 * 8192


@pytest.mark.parametrize("n", [1, 31, 8191, 8192, 8193, SUPER - 1, SUPER, SUPER + 8193])
@pytest.mark.parametrize("items", [1, 2, 4])
def test_tile_edges(n, items):
    ctx = pv.Context(0)
    tables = {"t": datagen.table_filter_agg(n, seed=n + items)}
    register(ctx, tables)
    for a_lt, hi in ((0, 99), (10, 40), (100, 99)):
        plan = workloads.filter_project_plan(a_lt, 0, hi)
        for pred in ("branch", "predicated"):
            got = ctx.query(plan, pv.variant(exec="multi", pred=pred, items_per_thread=items, block=64 * items))
            assert_same(got, want(plan, tables), ctxmsg=f"n={n} a<{a_lt} b<={hi} {pred}")
    ctx.close()


def test_capacity_is_kept():
    """More matches than the capacity: the first rows of the result and the overflow status."""
    ctx = pv.Context(0)
    n = 100_001
    tables = {"t": datagen.table_filter_agg(n, seed=9)}
    register(ctx, tables)
    plan = workloads.filter_project_plan(50, 0, 99)
    w = want(plan, tables)
    assert len(w[0]) > 20_000
    with pytest.raises(pv.PVError) as e:
        ctx.query(dict(plan, capacity_hint=20_000), pv.variant(exec="multi"))
    assert e.value.status == -7
    exact = ctx.query(dict(plan, capacity_hint=len(w[0])), pv.variant(exec="multi"))
    assert_same(exact, w)
    ctx.close()
