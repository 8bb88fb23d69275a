"""Ordered projections where the emit kernel's units, tiles and supers end: row counts
around a unit (1024 rows), a tile (8192), a super (131,072) and the count past which
the marks take four items a lane; few, half and all rows matching.  Rows must equal
numpy's, in order."""
import numpy as np
import pytest

from paper_1709_00700_gb300 import pv, workloads
from tests.gpu_util import register

pytestmark = pytest.mark.gpu


def _same(got, want):
    assert len(got) == len(want)
    for g, w in zip(got, want):
        assert np.array_equal(g, w.astype(np.int64))


@pytest.mark.parametrize("n", [1, 31, 1023, 1024, 1025, 8191, 8193, 131_071, 131_073, 311_295, 311_297, 2_000_003,
                               20_000_003])
def test_units(n):
    r = np.random.default_rng(n)
    a, b = (r.integers(0, 100, n).astype(np.int32) for _ in range(2))
    price = r.integers(100, 10**7, n).astype(np.int64)
    p = r.integers(-9, 9, 100).astype(np.int32)
    key = r.permutation(100).astype(np.int32)
    ctx = pv.Context(0)
    register(ctx, {"t": {"a": a, "b": b, "price": price}, "d": {"key": key, "p": p}})
    pay = np.empty(100, dtype=np.int64)
    pay[key] = p
    for a_lt, b_hi, pred in ((2, 40, "branch"), (50, 99, "predicated"), (100, 99, "branch")):
        hit = (a < a_lt) & (b <= b_hi)
        var = pv.variant(exec="multi", pred=pred, items_per_thread=1, block=128)
        _same(ctx.query(workloads.filter_project_plan(a_lt, 0, b_hi), var), [a[hit], price[hit]])
        plan = {"fact": "t", "filters": [["a", "lt", a_lt]],
                "builds": [{"table": "d", "key": "key", "filters": [["p", "lt", 5]], "payload": ["p"]}],
                "probes": [{"build": 0, "fk": "b"}], "project": [["payload", 0, 0], "price"]}
        hit = (a < a_lt) & (pay[b] < 5)
        for kind in ("perfect", "linear"):
            _same(ctx.query(plan, var, pv.ht_variant(kind)), [pay[b][hit], price[hit]])
    cap = int((a < 50).sum()) // 2
    if cap > 0:
        plan = {"fact": "t", "filters": [["a", "lt", 50]], "project": ["b", "price"], "capacity_hint": cap}
        res = None
        with pytest.raises(pv.PVError) as e:
            res = ctx.query(plan, pv.variant(exec="multi"))
        assert e.value.status == -7 and res is None
    ctx.close()
