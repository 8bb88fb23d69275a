"""Device memory that cannot be had: the call that needs it reports PV_ERR_OOM and
the next call runs; optional scratch that is refused leaves the query to the
general kernels."""
import numpy as np
import pytest

from paper_1709_00700_gb300 import datagen, pv, workloads
from tests.gpu_util import assert_same, register, want

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("use_torch_allocator", [False, True])
def test_query_runs_after_a_refused_allocation(use_torch_allocator):
    ctx = pv.Context(0, use_torch_allocator=use_torch_allocator)
    tables = {"t": datagen.table_filter_agg(5_003, seed=5)}
    register(ctx, tables)
    plan = workloads.filter_project_plan(10, 0, 99)
    for _ in range(2):
        with pytest.raises(pv.PVError) as e:
            ctx.run(dict(plan, capacity_hint=1 << 50), pv.variant())
        assert e.value.status == -10
        assert_same(ctx.query(plan, pv.variant()), want(plan, tables), ordered=False)
    ctx.close()


N = (1 << 20) + 77
PLAN = workloads.keyval_plan()
VAR = pv.variant(agg="global", ht="perfect", items_per_thread=1)


class Budget:
    """torch's allocator with a limit on the bytes of one allocation and on the bytes held."""

    def __init__(self, monkeypatch):
        import torch
        self.alloc, self.free = torch.cuda.caching_allocator_alloc, torch.cuda.caching_allocator_delete
        self.held, self.one, self.total = {}, 1 << 62, 1 << 62
        monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", self._alloc)
        monkeypatch.setattr(torch.cuda, "caching_allocator_delete", self._free)

    def _alloc(self, nbytes, *args):
        if nbytes > self.one or sum(self.held.values()) + nbytes > self.total:
            raise RuntimeError("no memory")
        p = self.alloc(nbytes, *args)
        self.held[p] = nbytes
        return p

    def _free(self, p):
        del self.held[p]
        self.free(p)


@pytest.fixture
def setup(monkeypatch):
    budget = Budget(monkeypatch)
    ctx = pv.Context(0)
    r = np.random.default_rng(3)
    tables = {"kv": {"key": np.where(r.random(N) < 0.1, 17, r.integers(0, 5_000, N)).astype(np.int32),
                     "val": r.integers(0, 1 << 20, N)}, "t": datagen.table_filter_agg(3_000_003, seed=5)}
    register(ctx, tables)
    yield ctx, budget, tables, want(PLAN, tables)
    ctx.close()


def _same(ctx, res, exact):
    assert_same(ctx.fetch(res), exact, ordered=False)


def test_refused_scratch(setup):
    ctx, budget, _, exact = setup
    budget.one = 12 * N - 1  # the records do not fit, everything else does
    res = ctx.run(PLAN, VAR)
    assert ctx.last_launch_count() == 2
    for _ in range(2):
        _same(ctx, res, exact)
        ctx.rerun(res)
    ctx.sync()


def test_scratch_gives_way(setup):
    ctx, budget, tables, exact = setup
    res = [ctx.run(PLAN, VAR) for _ in range(2)]
    assert ctx.last_launch_count() == 3
    held = sum(budget.held.values())
    plan = workloads.filter_project_plan(100, 0, 99)  # its result takes 36 MB, which only the scratch leaves
    budget.total = held + (16 << 20)
    got = ctx.query(plan, pv.variant())
    assert_same(got, want(plan, tables), ordered=False)
    assert sum(budget.held.values()) <= held - 2 * 12 * N
    for q in res:  # on the general kernels from now on, over clean tables
        _same(ctx, q, exact)
        for _ in range(2):
            ctx.rerun(q)
            assert ctx.last_launch_count() == 2
            _same(ctx, q, exact)
    budget.total = 1 << 62
    again = ctx.run(PLAN, VAR)
    assert ctx.last_launch_count() == 3
    _same(ctx, again, exact)


def test_graph_keeps_its_scratch(setup):
    ctx, budget, _, exact = setup
    res = ctx.run(PLAN, VAR)
    ch = pv.Chain(ctx, [("q", [], res)])
    ch.capture()
    budget.total = sum(budget.held.values()) + (1 << 20)
    with pytest.raises(pv.PVError) as e:
        ctx.run(workloads.filter_project_plan(100, 0, 99), pv.variant())
    assert e.value.status == -10
    for _ in range(2):
        ch.launch()
        _same(ctx, res, exact)
    ctx.rerun(res)
    assert ctx.last_launch_count() == 3
    _same(ctx, res, exact)
    ch.free()
