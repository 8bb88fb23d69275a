"""Single-pass projections at every block size the ABI takes: the rows a warp stages and
the registers a thread holds must leave room for 1024 threads wherever the
kernels without stages ran.  Rows must equal the oracle's."""
import numpy as np
import pytest

from paper_1709_00700_gb300 import pv, workloads
from tests.gpu_util import assert_same, register, want

pytestmark = pytest.mark.gpu

N = 40_003


def _plans():
    d = [{"table": "d", "key": "key", "filters": [["f", "lt", 60]], "payload": ["p"]}]
    pr = [{"build": 0, "fk": "b"}]
    return [workloads.filter_project_plan(30, 0, 70),
            {"fact": "t", "filters": [["a", "lt", 30]], "project": ["b", "price"]},
            {"fact": "t", "builds": d, "probes": pr, "project": [["payload", 0, 0], "price"]},
            {"fact": "t", "filters": [["a", "lt", 30]], "builds": d, "probes": pr,
             "project": [["payload", 0, 0], "price"]},
            {"fact": "t", "builds": d, "probes": pr, "project": ["a", "b"]},
            {"fact": "t", "filters": [["a", "lt", 30]], "builds": d, "probes": pr,
             "project": ["c", ["payload", 0, 0]]}]


@pytest.mark.parametrize("block", [64, 512, 1024])
@pytest.mark.parametrize("items", [1, 2])
@pytest.mark.parametrize("pred", ["branch", "predicated"])
@pytest.mark.parametrize("access", ["grid", "chunked"])
def test_blocks(block, items, pred, access):
    r = np.random.default_rng(block)
    tables = {"t": {"a": r.integers(0, 100, N).astype(np.int32), "b": r.integers(0, 100, N).astype(np.int32),
                    "c": r.integers(0, 9, N).astype(np.int32), "price": r.integers(100, 10**7, N).astype(np.int64)},
              "d": {"key": r.permutation(100).astype(np.int32), "f": r.integers(0, 100, 100).astype(np.int32),
                    "p": r.integers(-9, 9, 100).astype(np.int32)}}
    ctx = pv.Context(0)
    register(ctx, tables)
    for i, plan in enumerate(_plans()):
        got = ctx.query(plan, pv.variant(exec="single", pred=pred, access=access, items_per_thread=items, block=block),
                        pv.ht_variant("perfect"))
        assert_same(got, want(plan, tables), ordered=False, ctxmsg=f"{i} {block} {items} {pred} {access}")
    ctx.close()
