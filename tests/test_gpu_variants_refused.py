"""A grouped variant that the general kernels refuse is refused at every size: above the
row count from which tables may be partitioned, and below.  Accepted ones give the
oracle's groups at both."""
import numpy as np
import pytest

from paper_1709_00700_gb300 import datagen, pv, workloads
from tests.gpu_util import assert_same, register, want

pytestmark = pytest.mark.gpu

SMALL, LARGE = 20_011, (1 << 20) + 11


def _status(ctx, plan, var, exact):
    try:
        got = ctx.query(plan, var)
    except pv.PVError as e:
        return e.status
    assert_same(got, exact, ordered=False)
    return 0


@pytest.mark.parametrize("ht", ["perfect", "linear"])
@pytest.mark.parametrize("shape", ["keyval", "filtered", "three parts"])
def test_same_variants_at_every_size(ht, shape):
    statuses = []
    for n in (SMALL, LARGE):
        r = np.random.default_rng(n)
        key = datagen.zipf_keys(7, 0, n, 1_100_000)
        key[0], key[-1] = 0, 1_099_999
        if shape == "three parts":
            part = np.where(r.random(n) < 0.6, 5, r.integers(0, 104, n)).astype(np.int32)  # one value is hot
            part[:2] = (0, 103)
            tables = {"k3": {c: part for c in "abc"}}
            tables["k3"]["val"] = r.integers(0, 1 << 20, n)
            plan = workloads.keys3_plan()
        else:
            tables = {"kv": {"key": key, "val": r.integers(0, 1 << 20, n)}}
            plan = workloads.keyval_plan(900_000 if shape == "filtered" else None)
        exact = want(plan, tables)
        ctx = pv.Context(0)
        register(ctx, tables)
        row = {}
        for items in (1, 2, 4):
            for block in (64, 1024):
                for pred, access, prefetch in (("branch", "grid", 0), ("predicated", "chunked", 0), ("branch", "grid", 2)):
                    var = pv.variant(agg="global", ht=ht, items_per_thread=items, block=block, pred=pred, access=access,
                                     prefetch=prefetch, warp_agg=1)
                    row[items, block, pred, access, prefetch] = _status(ctx, plan, var, exact)
        statuses.append(row)
        ctx.close()
    assert statuses[0] == statuses[1]
    assert 0 in statuses[0].values() and -2 in statuses[0].values()
