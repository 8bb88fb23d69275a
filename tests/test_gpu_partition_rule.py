"""Which calls the partitioned aggregation takes: by the share of rows that pass, the
table's size and the keys' skew (from a sample), not by warp_agg.  The route is read
off the number of kernels (partitioned 3, and 5 for hash tables with their fallback;
general 2); the groups must equal numpy's on every route."""
import numpy as np
import pytest

from paper_1709_00700_gb300 import datagen, pv, workloads
from tests.gpu_util import register, rows_sorted

pytestmark = pytest.mark.gpu


def _want(code, names, val, keep):
    """Groups of the kept rows: code[i] is row i's group, names[g] its key."""
    count = np.bincount(code[keep], minlength=len(names))
    total = np.bincount(code[keep], weights=val[keep], minlength=len(names)).astype(np.int64)  # exact below 2^53
    live = np.nonzero(count)[0]
    return rows_sorted([names[live], total[live], count[live]])


def _run(ctx, plan, var, want):
    res = ctx.run(plan, var)
    kernels = ctx.last_launch_count()
    for _ in range(2):
        for g, w in zip(rows_sorted(ctx.fetch(res)), want):
            assert np.array_equal(g, w)
        ctx.rerun(res)
    ctx.sync()
    ctx.free(res)
    return kernels


M = 1 << 20


# rows, groups, skewed, share kept (None: no filter) -> partitioned
@pytest.mark.parametrize("n,groups,skew,keep,part", [
    (M - 1, 9_000_000, True, None, False), (M, 9_000_000, False, None, True), (M, 4_095, True, None, False),
    (M, 4_096, True, None, True), (M, 4_096, False, None, False), (M, 50_000, True, 0.35, True),
    (M, 50_000, True, 0.1, False), (M, 50_000, False, 0.9, False), (4 * M + 5, 50_000, True, 0.15, True),
    (4 * M + 5, 50_000, True, 0.05, False), (M + 3, 1_000_000, False, None, True),
    (M + 3, 1_000_000, False, 0.9, False), (M + 3, 9_000_000, False, 0.1, True), (M + 3, 9_000_000, False, 0.02, False),
    (2 * M, 3_000_000, False, 0.2, True), (4 * M - 1, 5_000, False, None, False), (4 * M, 5_000, False, None, True),
    (16 * M, 9_999, False, None, True), (16 * M, 60_000, False, None, False), (16 * M + 9, 5_000, False, 0.9, True),
    (16 * M + 9, 5_000, False, 0.5, False)])
def test_perfect(n, groups, skew, keep, part):
    r = np.random.default_rng(n + groups)
    key = datagen.zipf_keys(5, 0, n, groups) if skew else r.integers(0, groups, n, dtype=np.int32)
    key[0], key[-1] = 0, groups - 1
    val = r.integers(0, 1 << 20, n)
    val[0], val[-1] = 0, (1 << 20) - 1
    ctx = pv.Context(0)
    register(ctx, {"kv": {"key": key, "val": val}})
    lt = int(keep * (1 << 20)) if keep else 1 << 40
    want = _want(key, np.arange(groups), val, val < lt)
    for warp_agg in (0, 1) if n < 16 * M else (1,):
        var = pv.variant(agg="global", ht="perfect", items_per_thread=1, warp_agg=warp_agg)
        assert _run(ctx, workloads.keyval_plan(lt if keep else None), var, want) == (3 if part else 2)
    ctx.close()


@pytest.mark.parametrize("n,groups,skew,keep,part", [
    (M, 600_000, False, 0.5, True), (M, 600_000, False, 0.2, False), (M, 60_000, True, 0.9, False),
    (4 * M, 60_000, True, 0.5, True), (4 * M, 60_000, True, 0.1, False), (4 * M, 60_000, False, 0.9, False),
    (4 * M, 300_000, False, 0.5, True), (4 * M, 300_000, False, None, False), (4 * M, 900_000, False, None, True),
    (4 * M, 2_000, False, None, True), (9 * M, 60_000, False, 0.5, True), (9 * M, 60_000, False, 0.9, False),
    (16 * M, 2_000, False, None, True), (16 * M, 60_000, False, None, False), (16 * M, 60_000, False, 0.02, True),
    (16 * M, 60_000, False, 0.005, False)])
def test_linear(n, groups, skew, keep, part):
    r = np.random.default_rng(n + groups)
    code = datagen.zipf_keys(5, 0, n, groups) if skew else r.integers(0, groups, n, dtype=np.int32)
    code[::1009] = groups
    names = (np.arange(groups + 1) * 4_093).astype(np.int32)  # wraps: negative keys too
    names[groups] = -1
    val = r.integers(0, 1 << 20, n)
    val[0], val[-1] = 0, (1 << 20) - 1
    ctx = pv.Context(0)
    register(ctx, {"kv": {"key": names[code], "val": val}})
    lt = int(keep * (1 << 20)) if keep else 1 << 40
    plan = dict(workloads.keyval_plan(lt if keep else None), capacity_hint=groups + 1)
    kernels = _run(ctx, plan, pv.variant(agg="global", ht="linear", items_per_thread=1),
                   _want(code, names, val, val < lt))
    assert kernels == (5 if part else 2)
    ctx.close()


def test_range_that_overflows():
    """65,536 slots for 60,001 keys, one of them hot: some range of slots gets more keys than it has, and the
    general kernels run the pipeline again."""
    n = 4 * M + 4099
    r = np.random.default_rng(8)
    key = (r.permutation(n) % 60_000).astype(np.int32)
    key[r.random(n) < 0.1] = 60_000
    val = r.integers(0, 1 << 20, n)
    ctx = pv.Context(0)
    register(ctx, {"kv": {"key": key, "val": val}})
    plan = dict(workloads.keyval_plan(2**40), capacity_hint=32_000)
    want = _want(key, np.arange(60_001), val, val < 2**40)
    assert _run(ctx, plan, pv.variant(agg="global", ht="linear", items_per_thread=1), want) == 5
    with pytest.raises(pv.PVError) as e:
        ctx.query(dict(plan, capacity_hint=16_000), pv.variant(agg="global", ht="linear", items_per_thread=1))
    assert e.value.status == -3
    ctx.close()


@pytest.mark.parametrize("n", [M, M + 4_099])
def test_three_part_keys(n):
    """Past L2: partitioned, with the scatter that filters and loads its keys item by item."""
    r = np.random.default_rng(n)
    parts = [r.integers(-3, 207, n).astype(np.int32) for _ in range(3)]
    for p in parts:
        p[0], p[-1] = -3, 206
    val = r.integers(0, 1 << 20, n)
    ctx = pv.Context(0)
    register(ctx, {"k3": dict(zip("abc", parts), val=val)})
    res = ctx.run(workloads.keys3_plan(), pv.variant(agg="global", ht="perfect", items_per_thread=1))
    assert ctx.last_launch_count() == 3
    want = _want(((parts[0] + 3) * 210 + parts[1] + 3) * 210 + parts[2] + 3, np.arange(210**3), val, slice(None))
    for _ in range(2):
        a, b, c, s, k = ctx.fetch(res)
        got = rows_sorted([((a + 3) * 210 + b + 3) * 210 + c + 3, s, k])
        for g, w in zip(got, want):
            assert np.array_equal(g, w)
        ctx.rerun(res)
    ctx.close()
