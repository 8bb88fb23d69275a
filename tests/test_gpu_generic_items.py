"""The generic aggregation kernels by items of 4 rows: tables that end inside an
item, columns of every type, few groups (copied local tables), MIN/MAX, both
evaluation modes, and result columns that start off a 16-byte boundary.
Results are integers and must equal the oracle's."""
import numpy as np
import pytest

from oracle import oracle
from paper_1709_00700_gb300 import pv
from tests.gpu_util import assert_same, register, want

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = pv.Context(0)
    yield c
    c.close()


def _tables(n, seed=3):
    r = np.random.default_rng(seed + n)
    fact = {"i": r.integers(-50, 50, n).astype(np.int32), "u": r.integers(0, 256, n).astype(np.uint8),
            "l": r.integers(-2**40, 2**40, n).astype(np.int64), "fk": r.integers(-5, 205, n).astype(np.int32),
            "fl": r.integers(-5, 205, n).astype(np.int64), "g": r.integers(3, 8, n).astype(np.int32)}
    dim = {"key": r.permutation(200).astype(np.int32), "p": r.integers(-9, 9, 200).astype(np.int32)}
    return {"f": fact, "d": dim}


AGGS = [["sum", [["x", "l"], ["c_minus_x", "u", 100]]], ["min", [["x", "l"]]], ["max", [["x_plus_c", "i", -7]]],
        ["count"]]
PLANS = [
    {"fact": "f", "filters": [["i", "between", -40, 30], ["u", "ge", 16], ["l", "lt", 2**39]], "aggs": AGGS},
    {"fact": "f", "filters": [["i", "eq", 7]], "aggs": AGGS[:3]},
    {"fact": "f", "filters": [["i", "ge", -45]], "group_by": ["g"], "aggs": AGGS[:3]},
    {"fact": "f", "builds": [{"table": "d", "key": "key", "filters": [["p", "lt", 5]], "payload": ["p"]}],
     "probes": [{"build": 0, "fk": "fk"}, {"build": 0, "fk": "fl"}], "group_by": [["payload", 0, 0], "g"],
     "aggs": [["sum", [["x", ["payload", 1, 0]], ["x", "u"]]], ["count"]]},
]


@pytest.mark.parametrize("n", [1, 3, 6, 257, 2055, 60_003])
@pytest.mark.parametrize("pred", ["branch", "predicated"])
def test_items(ctx, n, pred):
    tables = _tables(n)
    register(ctx, tables)
    for plan in PLANS:
        w = want(plan, tables)
        kws = [dict()] if "group_by" not in plan else [
            dict(agg="local", ht="perfect"), dict(agg="global", ht="perfect"), dict(agg="local", ht="linear"),
            dict(agg="global", ht="linear")]
        for kw in kws:
            got = ctx.query(plan, pv.variant(pred=pred, block=128 if n < 300 else 1024, interp=1, **kw),
                            pv.ht_variant("perfect" if n % 2 else "linear"))
            assert_same(got, w, ordered=False, ctxmsg=f"n={n} {pred} {kw} {plan}")


@pytest.mark.parametrize("groups", [5, 6, 7, 8])
def test_result_columns_of_any_alignment(ctx, groups):
    """An aggregation over a grouped result's second column, `groups` + 1 words after the first."""
    n = 3001
    r = np.random.default_rng(groups)
    tables = {"f": {"k": (np.arange(n) % groups).astype(np.int32), "v": r.integers(-99, 99, n).astype(np.int64)}}
    register(ctx, tables)
    chain = [{"name": "s", "columns": ["k", "s", "c"],
              "plan": {"fact": "f", "group_by": ["k"], "aggs": [["sum", [["x", "v"]]], ["count"]]}},
             {"name": "t", "columns": ["m", "x"],
              "plan": {"fact": "s", "filters": [["c", "ge", 1]],
                       "aggs": [["max", [["x", "s"]]], ["sum", [["x", "s"], ["x", "k"]]]]}}]
    w = oracle.run_chain(chain, tables, nthreads=2)
    ch = ctx.run_chain(chain, {"s": pv.variant(agg="global", ht="perfect"), "t": pv.variant()}, pv.ht_variant("linear"))
    assert_same(ch.fetch(1), w[1]["cols"])
    ch.free()
