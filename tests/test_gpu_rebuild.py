"""Rebuilds of perfect arrays, whose probes read presence bits or payload codes:
domains at the edges of a word, inputs changed in place, and the errors of the
first build (duplicate key, key or payload outside its domain).  Also the
single-pass projection below, at and above the rows a warp stages."""
import numpy as np
import pytest

from oracle import oracle
from paper_1709_00700_gb300 import datagen, pv, workloads
from tests.gpu_util import assert_same, register, want

pytestmark = pytest.mark.gpu


def _plan(payload):
    p = {"fact": "f", "builds": [{"table": "d", "key": "key", "filters": [["w", "lt", 60]], "payload": payload}],
         "probes": [{"build": 0, "fk": "fk"}], "aggs": [["count"]]}
    if payload:
        p["aggs"] = [["count"], ["sum", [["x", ["payload", 0, 0]]]]]
    return p


@pytest.mark.parametrize("n", [1, 31, 32, 33, 1025, 300_001])
@pytest.mark.parametrize("payload", [[], ["p"]])
def test_rebuild_follows_its_columns(n, payload):
    import torch
    r = np.random.default_rng(n)
    ctx = pv.Context(0)
    dim = {"key": (r.permutation(n) - 5).astype(np.int32), "w": r.integers(0, 100, n).astype(np.uint8),
           "p": r.integers(-120, 130, n).astype(np.int32)}
    dim["p"][0], dim["p"][-1], dim["w"][0], dim["w"][-1] = -120, 129, 0, 0
    fact = {"fk": r.integers(-8, n, 20_011).astype(np.int32)}
    dev = {c: torch.from_numpy(v).cuda() for c, v in dim.items()}
    ctx.register_table("d", dev)
    ctx.register_table("f", {"fk": torch.from_numpy(fact["fk"]).cuda()})
    plan = _plan(payload)
    hts = ctx.build_all(plan, pv.ht_variant("perfect"))
    res = ctx.run(plan, pv.variant(interp=1), hts)
    assert_same(ctx.fetch(res), oracle.run(plan, {"f": fact, "d": dim})["cols"])
    dim["w"] = r.integers(0, 100, n).astype(np.uint8)
    dim["p"] = r.permutation(dim["p"])
    for c in ("w", "p"):
        dev[c].copy_(torch.from_numpy(dim[c]))
    torch.cuda.synchronize()
    for _ in range(2):
        for h in hts:
            ctx.rebuild(h)
        ctx.rerun(res)
    assert_same(ctx.fetch(res), oracle.run(plan, {"f": fact, "d": dim})["cols"])
    # errors
    def broken(col, i, v, status):
        keep = dev[col][i].item()
        dev["w"][i] = 0
        dev[col][i] = v
        torch.cuda.synchronize()
        ctx.rebuild(hts[0])
        with pytest.raises(pv.PVError) as e:
            ctx.sync()
        assert e.value.status == status
        dev[col][i] = keep
    if n > 1:
        dev["w"][:2] = 0
        broken("key", 0, dev["key"][1].item(), -6)
    broken("key", n - 1, n + 5, -5)
    if payload:
        broken("p", 0, 1000, -5)
    ctx.close()


@pytest.mark.parametrize("n", [1, 127, 4099, 300_007])
@pytest.mark.parametrize("items", [1, 2, 4])
def test_single_pass_projection(n, items):
    """Selectivities from a few rows a warp to whole trips, with and without a probe's payload."""
    ctx = pv.Context(0)
    tables = {"t": datagen.table_filter_agg(n, seed=n)}
    register(ctx, tables)
    for a_lt, hi in ((1, 30), (15, 99), (25, 99), (60, 99), (100, 99)):
        plan = workloads.filter_project_plan(a_lt, 0, hi)
        got = ctx.query(plan, pv.variant(exec="single", items_per_thread=items, block=64 * items))
        assert_same(got, want(plan, tables), ordered=False, ctxmsg=f"{n} {a_lt} {hi}")
    plan = dict(workloads.filter_project_plan(50, 0, 99), capacity_hint=n // 4 + 1)
    if n > 1000:
        with pytest.raises(pv.PVError) as e:
            ctx.query(plan, pv.variant(exec="single", items_per_thread=items))
        assert e.value.status == -7
    ctx.close()
