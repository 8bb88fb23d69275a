"""Grouped aggregation through range-partitioned records: domains and tables at
the edges of their ranges, skew that shares a range between units, keys at the
ends of their type, hints too small for the keys, replays.  Integer results
must equal numpy's, group by group."""
import numpy as np
import pytest

from paper_1709_00700_gb300 import datagen, pv, workloads
from tests.gpu_util import register, rows_sorted

pytestmark = pytest.mark.gpu

N = (1 << 20) + 4099      # past the smallest row count that is partitioned, ending inside an item
N_HASH = (4 << 20) + 4099  # of a small hash table


@pytest.fixture(scope="module")
def ctx():
    c = pv.Context(0)
    yield c
    c.close()


def _want(key, val, keep=None):
    if keep is not None:
        key, val = key[keep], val[keep]
    k, inv = np.unique(key, return_inverse=True)
    s = np.zeros(len(k), dtype=np.int64)
    np.add.at(s, inv, val)
    return [k.astype(np.int64), s, np.bincount(inv, minlength=len(k)).astype(np.int64)]


def _check(got, want):
    for g, w in zip(rows_sorted(got), want):
        assert np.array_equal(g, w)


def _keys(dist, groups, r, n=N):
    if dist == "zipf":
        return datagen.zipf_keys(groups, 0, n, groups).astype(np.int32)
    if dist == "one":
        return np.full(n, groups // 2, dtype=np.int32)
    return r.integers(0, groups, n).astype(np.int32)


@pytest.mark.parametrize("groups", [4096, 4097, 262_144, 262_145, 5_000_000, 16_777_216, 16_777_217])
@pytest.mark.parametrize("dist", ["uniform", "zipf", "one"])
def test_perfect(ctx, groups, dist):
    r = np.random.default_rng(groups)
    key = _keys(dist, groups, r) - 7
    key[0], key[-1] = -7, groups - 8  # the whole domain
    val = r.integers(-2**62, 2**62, N)
    register(ctx, {"kv": {"key": key, "val": val}})
    var = pv.variant(agg="global", ht="perfect", items_per_thread=1, warp_agg=1)
    res = ctx.run(workloads.keyval_plan(), var)
    _check(ctx.fetch(res), _want(key, val))
    ctx.rerun(res)  # the table and the scratch are clean again
    _check(ctx.fetch(res), _want(key, val))
    ctx.free(res)


@pytest.mark.parametrize("groups", [3, 300, 5_000, 200_000, 1_000_000])
@pytest.mark.parametrize("dist", ["uniform", "zipf"])
@pytest.mark.parametrize("limit", [2**40, 1 << 19, -1])
def test_linear(ctx, groups, dist, limit):
    r = np.random.default_rng(groups)
    key = (_keys(dist, groups, r, N_HASH).astype(np.int64) * 4_093).astype(np.int32)  # wraps: negative keys too
    key[::1009] = -1
    key[1::1013] = np.iinfo(np.int32).min
    val = r.integers(0, 1 << 20, N_HASH)
    register(ctx, {"kv": {"key": key, "val": val}})
    w = _want(key, val, val < limit)
    for kw in (dict(warp_agg=1), dict(hash="multshift")):
        plan = dict(workloads.keyval_plan(limit), capacity_hint=max(groups + 2, 4))
        res = ctx.run(plan, pv.variant(agg="global", ht="linear", items_per_thread=1, **kw))
        for _ in range(2):
            _check(ctx.fetch(res), w)
            ctx.rerun(res)
        ctx.sync()
        ctx.free(res)


def test_linear_hint_too_small(ctx):
    """A table loaded past a range's share still gives the result; one with fewer slots than keys still fails."""
    r = np.random.default_rng(8)
    key = (r.permutation(N_HASH) % 60_000).astype(np.int32)
    val = r.integers(0, 1 << 20, N_HASH)
    register(ctx, {"kv": {"key": key, "val": val}})
    var = pv.variant(agg="global", ht="linear", items_per_thread=1)
    plan = dict(workloads.keyval_plan(2**40), capacity_hint=32_000)  # 65,536 slots for 60,000 keys
    res = ctx.run(plan, var)
    for _ in range(2):
        _check(ctx.fetch(res), _want(key, val))
        ctx.rerun(res)
    ctx.sync()
    ctx.free(res)
    with pytest.raises(pv.PVError) as e:
        ctx.query(dict(plan, capacity_hint=16_000), var)  # 32,768 slots
    assert e.value.status == -3
