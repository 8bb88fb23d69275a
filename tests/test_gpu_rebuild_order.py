"""Rebuilds of presence bits whose rows meet in the words: keys in table order, starting
inside a word, with duplicates inside one warp and in two.  Counts must equal numpy's."""
import numpy as np
import pytest

from paper_1709_00700_gb300 import pv
from tests.gpu_util import register

pytestmark = pytest.mark.gpu

PLAN = {"fact": "f", "builds": [{"table": "d", "key": "key", "filters": [["w", "lt", 60]], "payload": []}],
        "probes": [{"build": 0, "fk": "fk"}], "aggs": [["count"]]}


@pytest.mark.parametrize("n", [1, 31, 33, 1024, 100_003, 700_001])
@pytest.mark.parametrize("first", [0, -5, 17])
@pytest.mark.parametrize("order", ["ascending", "descending", "by sevens"])
def test_keys_in_order(n, first, order):
    import torch
    r = np.random.default_rng(n)
    key = np.arange(first, first + n).astype(np.int32)
    if order == "descending":
        key = key[::-1].copy()
    elif order == "by sevens":
        key = first + ((np.arange(n, dtype=np.int64) * 7) % n).astype(np.int32) if n % 7 else key
    w = r.integers(0, 100, n).astype(np.uint8)
    w[0] = 0
    fk = r.integers(first - 8, first + n + 8, 20_011).astype(np.int32)
    dev = {"key": torch.from_numpy(key).cuda(), "w": torch.from_numpy(w).cuda()}
    ctx = pv.Context(0)
    ctx.register_table("d", dev)
    register(ctx, {"f": {"fk": fk}})
    hts = ctx.build_all(PLAN, pv.ht_variant("perfect"))
    res = ctx.run(PLAN, pv.variant(interp=1), hts)
    for keep in (100, 60, 3):
        w = r.integers(0, 100, n) % keep
        w[0] = 0
        dev["w"].copy_(torch.from_numpy(w.astype(np.uint8)))
        torch.cuda.synchronize()
        ctx.rebuild(hts[0])
        ctx.rerun(res)
        assert int(ctx.fetch(res)[0][0]) == int(np.isin(fk, key[w < 60]).sum())
    for i, j in ((0, 1), (0, n - 1), (n // 2, n - 1)):  # duplicates: of a neighbour, far apart
        if i == j or n < 2:
            continue
        keep = dev["key"][i].item()
        dev["w"].zero_()
        dev["key"][i] = dev["key"][j].item()
        torch.cuda.synchronize()
        ctx.rebuild(hts[0])
        with pytest.raises(pv.PVError) as e:
            ctx.sync()
        assert e.value.status == -6
        dev["key"][i] = keep
    ctx.close()
