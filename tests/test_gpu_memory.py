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
