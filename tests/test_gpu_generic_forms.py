"""The generic grouped kernels on both sides of the rule that picks their form: by items
of four rows for CTA-local perfect arrays, by rows for tables of fewer rows than three
a thread, global arrays and hash tables.  Results must equal the oracle's."""
import numpy as np
import pytest

from paper_1709_00700_gb300 import pv
from tests.gpu_util import assert_same, register, want

pytestmark = pytest.mark.gpu

AGGS = [["sum", [["x", "v"]]], ["min", [["x", "v"]]], ["max", [["x_plus_c", "v", 3]]], ["count"]]


@pytest.mark.parametrize("n", [1, 767, 768, 1535, 1536, 100_003])
@pytest.mark.parametrize("groups", [3, 4_000])
def test_forms(n, groups):
    r = np.random.default_rng(n + groups)
    tables = {"f": {"a": r.integers(0, 100, n).astype(np.int32), "k": r.integers(-2, groups - 2, n).astype(np.int32),
                    "v": r.integers(-2**40, 2**40, n).astype(np.int64)}}
    ctx = pv.Context(0)
    register(ctx, tables)
    for aggs in (AGGS, AGGS[:3]):
        plan = {"fact": "f", "filters": [["a", "ge", 30]], "group_by": ["k"], "aggs": aggs, "capacity_hint": groups}
        w = want(plan, tables)
        for kw in (dict(agg="local", ht="perfect"), dict(agg="global", ht="perfect"), dict(agg="local", ht="linear"),
                   dict(agg="global", ht="linear"), dict(agg="global", ht="cuckoo", exec="multi")):
            for block, pred in ((256, "branch"), (512, "predicated")):
                got = ctx.query(plan, pv.variant(pred=pred, block=block, interp=1, **kw))
                assert_same(got, w, ordered=False, ctxmsg=f"{n} {groups} {kw} {block}")
    ctx.close()
