"""The measured work: what a user of this library has it do, through its public entry points.

Each listed case is one query (or one training step of the cost model) on one GPU; `draw` gives more of the same
families over the ranges of the variant-selection suite (rows 1M to 100M, groups 10 to 1e7, selectivity 0.1% to 90%).
Tables are seeded synthetic tables with the columns, types and value distributions of datagen.py, drawn on the GPU.

A state holds registered columns, built tables and a result handle of one process-wide context, as a program that
keeps a Context open does; `run` is one query of it with its result delivered.  Grouped results come in no stated
order, so `run` delivers them on the GPU as a table indexed by group (dense keys) or ordered by key (sparse keys).
"""
import ctypes
import math

import torch

from paper_1709_00700_gb300 import costmodel, datagen, pv, workloads

DAY0, NDAYS = datagen.DAY0, datagen.NDAYS
_CTX = None


def context():
    """The process's context, set up as the README shows."""
    global _CTX
    if _CTX is None:
        _CTX = pv.Context(0)
        _CTX.set_l2_fetch_bytes(32)
    return _CTX


# ---- cases ------------------------------------------------------------------

def listed():
    return [
        # An interactive query on a small table: plan, run, synchronise, fetch and free, all through query().
        {"name": "query_small", "family": "query", "rows": 100_003, "a_lt": 10, "b_n": 21},
        # Filter, then SUM and COUNT, on a large fact table (the filter/aggregate configuration at 100M rows).
        {"name": "filter_agg_100m", "family": "filter_agg", "rows": 100_000_000, "a_lt": 10, "b_n": 21},
        # Rows of a filter in table order (the multi-pass projection), an odd row count.
        {"name": "project_ordered_50m", "family": "project", "rows": 50_000_003, "a_lt": 10, "b_n": 21},
        # Low-cardinality grouped aggregation with 8 aggregates (TPC-H Q1 shape), the benchmark's workload.
        {"name": "lowcard_6m", "family": "lowcard", "rows": 6_000_000, "day_hi": DAY0 + 2475},
        # GROUP BY a key of 1,000 values: the groups fit a thread block's shared memory.
        {"name": "group_1k_60m", "family": "group", "rows": 60_000_000, "groups": 1_000, "dist": "uniform"},
        # GROUP BY a key of 1e7 values: the group table outgrows every cache.
        {"name": "group_10m_60m", "family": "group", "rows": 60_000_000, "groups": 10_000_000, "dist": "uniform"},
        # Filtered GROUP BY over sparse, skewed keys in a linear-probing table.
        {"name": "group_hash_zipf_20m", "family": "group_hash", "rows": 20_000_001, "groups": 200_000, "dist": "zipf",
         "val_lt": 500_000},
        # Star join: four dimension builds and the probe pipeline, replayed as one graph.
        {"name": "star_60m", "family": "star", "rows": 60_000_000, "build": "perfect", "t_a": 20, "t_b": 20, "t_c": 5,
         "t_d": 10},
        # TPC-H Q5 shape: four dependent pipelines with their builds, replayed as one graph.
        {"name": "q5_60m", "family": "q5", "rows": 60_000_000, "regions": 3},
        # Ad-hoc query without a compiled shape (TPC-H Q6 shape): three filters, one product sum.
        {"name": "adhoc_agg_30m", "family": "adhoc_agg", "rows": 30_000_001, "days": 365, "qty_lt": 24},
        # Ad-hoc join without a compiled shape: two probes, grouped on one payload.
        {"name": "adhoc_join_20m", "family": "adhoc_join", "rows": 20_000_003, "years": 6},
        # One training step of the cost model (forward, backward, Adam) at the suite's number of samples.
        {"name": "mlp_step_24k", "family": "mlp", "batch": 24_001, "features": 45},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["query", "filter_agg", "project", "lowcard", "group", "group", "group_hash", "star", "q5",
                         "adhoc_agg", "adhoc_group", "adhoc_join", "mlp"])
    c = {"family": family}
    if family in ("query", "filter_agg", "project"):
        c["rows"] = _log(rng, 1_000, 1_000_000) if family == "query" else _log(rng, 1_000_000, 100_000_000) \
            if family == "filter_agg" else _log(rng, 1_000_000, 50_000_000)
        c.update(a_lt=_log(rng, 1, 100), b_n=_log(rng, 1, 90))
    elif family == "lowcard":
        c.update(rows=_log(rng, 1_000_000, 60_000_000), day_hi=DAY0 + rng.randrange(NDAYS // 2, NDAYS))
    elif family == "group":
        c.update(rows=_log(rng, 1_000_000, 60_000_000), groups=_log(rng, 10, 10_000_000),
                 dist=rng.choice(["uniform", "uniform", "zipf"]))
        if c["dist"] == "zipf":
            c["rows"] = min(c["rows"], 20_000_000)
    elif family == "group_hash":
        c.update(rows=_log(rng, 1_000_000, 20_000_000), groups=_log(rng, 1_000, 1_000_000),
                 dist=rng.choice(["uniform", "zipf"]), val_lt=_log(rng, 10_000, 900_000))
    elif family == "star":
        c.update(rows=_log(rng, 1_000_000, 60_000_000), build=rng.choice(["perfect", "perfect", "linear"]),
                 t_a=rng.randrange(1, 41), t_b=rng.randrange(1, 41), t_c=rng.randrange(1, 21),
                 t_d=rng.randrange(1, 21))
    elif family == "q5":
        c.update(rows=_log(rng, 1_000_000, 60_000_000), regions=rng.randrange(1, 5))
    elif family == "adhoc_agg":
        c.update(rows=_log(rng, 1_000_000, 30_000_000), days=_log(rng, 30, 2400), qty_lt=rng.randrange(2, 51))
    elif family == "adhoc_group":
        c.update(rows=_log(rng, 1_000_000, 20_000_000), qty_ge=rng.randrange(1, 45))
    elif family == "adhoc_join":
        c.update(rows=_log(rng, 1_000_000, 20_000_000), years=rng.randrange(1, 8))
    else:
        c.update(batch=_log(rng, 500, 24_001), features=rng.randrange(20, 61))
    return c


# ---- tables (the recipes of datagen.py, drawn on the GPU) ---------------------

class Draws:
    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(seed)

    def ints(self, n, lo, hi, dtype=torch.int32):
        return torch.randint(lo, hi, (n,), generator=self.g, device="cuda", dtype=dtype)

    def zipf(self, n, g):
        """Zipf(1) keys over [0, g), the hot ranks scattered over the domain as datagen.zipf_keys does."""
        cdf = torch.cumsum(1.0 / torch.arange(1, g + 1, device="cuda", dtype=torch.float64), 0)
        p = torch.rand(n, generator=self.g, device="cuda", dtype=torch.float64) * cdf[-1]
        r = torch.searchsorted(cdf, p, right=True).clamp_(max=g - 1)
        return ((r * datagen.coprime_multiplier(g) + g // 3) % g).to(torch.int32)

    def shuffled_keys(self, n):
        return torch.randperm(n, generator=self.g, device="cuda", dtype=torch.int32)


def filter_table(d, n):
    return {"a": d.ints(n, 0, 100), "b": d.ints(n, 0, 100), "price": d.ints(n, 100, 10_000_000, torch.int64)}


def lineitem_table(d, n):
    return {"date": d.ints(n, DAY0, DAY0 + NDAYS), "k1": d.ints(n, 65, 67, torch.uint8),
            "k2": d.ints(n, 88, 90, torch.uint8), "qty": d.ints(n, 1, 51, torch.int64),
            "price": d.ints(n, 100, 10_000_000, torch.int64), "disc": d.ints(n, 0, 11, torch.int64),
            "tax": d.ints(n, 0, 9, torch.int64)}


def star_tables(d, n):
    t = {"fact": {"fk_" + name[2:]: d.ints(n, 0, rows) for name, rows, _ in datagen.STAR_DIMS}}
    t["fact"]["revenue"] = d.ints(n, 100, 10_000_000, torch.int64)
    for name, rows, groups in datagen.STAR_DIMS:
        t[name] = {"key": d.shuffled_keys(rows), "f": d.ints(rows, 0, 100)}
        if groups:
            t[name]["g"] = d.ints(rows, 0, groups)
    return t


def q5_tables(d, n):
    orders, cust = max(1, n // 4), max(1, n // 40)
    nation = torch.arange(25, device="cuda", dtype=torch.int32)
    return {"nation": {"n_nationkey": nation, "n_regionkey": (nation // 5).to(torch.int32)},
            "customer": {"c_custkey": d.shuffled_keys(cust), "c_nationkey": d.ints(cust, 0, 25)},
            "orders": {"o_orderkey": d.shuffled_keys(orders), "o_custkey": d.ints(orders, 0, cust),
                       "o_orderdate": d.ints(orders, DAY0, DAY0 + datagen.TPCH_DAYS)},
            "lineitem": {"l_orderkey": d.ints(n, 0, orders),
                         "l_extendedprice": d.ints(n, 100, 10_000_000, torch.int64),
                         "l_discount": d.ints(n, 0, 11, torch.int64)}}


def join_tables(d, n):
    (_, custs), _, (_, days) = datagen.STAR3_DIMS
    nation = d.ints(custs, 0, 25)
    day = torch.arange(days, device="cuda")
    return {"fact": {"fk_cust": d.ints(n, 0, custs), "fk_date": d.ints(n, 0, days),
                     "revenue": d.ints(n, 100, 10_000_000, torch.int64)},
            "d_cust": {"key": d.shuffled_keys(custs), "region": (nation // 5).to(torch.int32)},
            "d_date": {"key": day.to(torch.int32),
                       "year": (datagen.STAR3_YEAR0 + (day // 365).clamp(max=6)).to(torch.int32)}}


# ---- states -------------------------------------------------------------------

class State:
    """Registered columns, tables and a result of the shared context, released with the state."""

    def __init__(self, family):
        self.family, self.ctx = family, context()
        self.handles, self.names, self.chain = [], [], None
        self.device_groups, self.spans = False, ()

    def register(self, tables):
        for name, cols in tables.items():
            self.ctx.register_table(name, cols)
            self.names += [(name, c) for c in cols]
        self.columns = [self.ctx.cols[k] for k in self.names]
        self.tensors = [self.ctx.keep.pop(k) for k in self.names]

    def deliver_to(self, res, device, groups=0):
        """Where the result's live rows go: page-locked host memory, or device memory by group."""
        self.res = res
        ctx, cap, live, n_cols, kind = self.ctx, ctypes.c_int64(), ctypes.c_int64(), ctypes.c_int32(), ctypes.c_int32()
        ctx._check(ctx.lib.pv_result_capacity(ctx.h, res, ctypes.byref(cap)))
        ctx._check(ctx.lib.pv_result_shape(ctx.h, res, ctypes.byref(live), ctypes.byref(n_cols)))
        self.live, kinds = live.value, []
        for c in range(n_cols.value):
            ctx._check(ctx.lib.pv_result_col_type(ctx.h, res, c, ctypes.byref(kind)))
            kinds.append({pv.PV_I32: torch.int32, pv.PV_I64: torch.int64, pv.PV_U8: torch.uint8}[kind.value])
        if device and len(set(kinds)) == 1:  # one block, its rows the result's columns
            self.block = torch.zeros((len(kinds), cap.value), dtype=kinds[0], device="cuda")
            self.rows = self.block[:, :self.live]
            cols, count = list(self.block), torch.zeros(1, dtype=torch.int64, device="cuda")
        else:
            place = (lambda t: t.cuda()) if device else (lambda t: t.pin_memory())
            cols = [place(torch.zeros(max(cap.value, 1), dtype=k)) for k in kinds]
            count = place(torch.zeros(1, dtype=torch.int64))
        self.outputs = cols + [count]
        self.fetch_args = (n_cols.value, (ctypes.c_void_p * len(cols))(*[t.data_ptr() for t in cols]),
                           (ctypes.c_int64 * len(cols))(*[t.numel() for t in cols]),
                           ctypes.c_void_p(count.data_ptr()))
        if groups:
            self.device_groups = True
            self.table = torch.zeros((groups, len(kinds)), dtype=torch.int64, device="cuda").t()
            self.outputs = [self.table, count]
        torch.cuda.synchronize()

    def __del__(self):
        try:
            if self.chain is not None:
                self.chain.free()
            for h in self.handles:
                self.ctx.free(h)
            for h in getattr(self, "columns", ()):
                self.ctx.free(h)
        except Exception:  # noqa: BLE001 - the process is ending
            pass


def prepare(case, seed):
    f, d = case["family"], Draws(seed)
    if f == "mlp":
        return prepare_mlp(case, d)
    n, s = case["rows"], State(f)
    ctx = s.ctx
    if f in ("query", "filter_agg", "project"):
        s.register({"t": filter_table(d, n)})
        b0 = (100 - case["b_n"]) // 4
        make = workloads.filter_project_plan if f == "project" else workloads.filter_agg_plan
        plan = make(case["a_lt"], b0, b0 + case["b_n"] - 1)
        if f == "query":
            s.plan, s.var = plan, pv.variant(pred="branch", items_per_thread=4, block=512)
            s.names_now = dict(zip(s.names, s.columns))
            return s
        if f == "filter_agg":
            var = pv.variant(pred="compacted", items_per_thread=2, block=256, first_items=2)
        else:
            # room for the matches the optimiser expects, with a margin
            plan["capacity_hint"] = min(n, int(1.2 * n * case["a_lt"] / 100 * case["b_n"] / 100) + 10_000)
            var = pv.variant(exec="multi", pred="branch", items_per_thread=4, block=256)
        res = ctx.run(plan, var)
        s.handles.append(res)
        s.deliver_to(res, device=f == "project")
        return s
    if f == "lowcard":
        s.register({"li": lineitem_table(d, n)})
        var = pv.variant(agg="local", ht="perfect", threads_per_table=1, pred="predicated", items_per_thread=1)
        res, s.spans = ctx.run(workloads.lowcard_plan(case["day_hi"]), var), (2,)  # entry 2 k1 + k2
        groups = 2 * 66 + 89 + 1
    elif f in ("group", "group_hash"):
        g = case["groups"]
        key = d.zipf(n, g) if case["dist"] == "zipf" else d.ints(n, 0, g)
        val = d.ints(n, 0, 1_000_000, torch.int64)
        if f == "group":
            s.register({"kv": {"key": key, "val": val}})
            small = g * 24 <= 190_000  # the group table fits a block's shared memory
            var = pv.variant(agg="local", ht="perfect", items_per_thread=1, block=1024 if g * 24 > 110_000 else 512) \
                if small else pv.variant(agg="global", ht="perfect", items_per_thread=1, block=256,
                                         warp_agg=int(case["dist"] == "zipf"))
            res, groups = ctx.run(workloads.keyval_plan(), var), g
        else:
            s.register({"kv": {"key": (key * 2_039 + 11).to(torch.int32), "val": val}})
            var = pv.variant(agg="global", ht="linear", items_per_thread=1, block=256, warp_agg=1)
            res, groups = ctx.run(dict(workloads.keyval_plan(case["val_lt"]), capacity_hint=g), var), g
    elif f == "star":
        s.register(star_tables(d, n))
        plan = workloads.star_plan({"d_a": case["t_a"], "d_b": case["t_b"], "d_c": case["t_c"], "d_d": case["t_d"]})
        var = pv.variant(agg="local", ht="perfect" if case["build"] == "perfect" else "linear", pred="compacted",
                         items_per_thread=2, block=512)
        step = {"name": "by_group", "columns": ["ga", "gb", "revenue", "rows"], "plan": plan}
        s.chain = ctx.run_chain([step], {"by_group": var}, pv.ht_variant(case["build"]))
        res, s.spans, groups = s.chain.steps[-1][2], (25,), 300
    elif f == "q5":
        s.register(q5_tables(d, n))
        vs = {"cust": pv.variant(items_per_thread=1), "ord": pv.variant(items_per_thread=1),
              "nat": pv.variant(agg="local", ht="perfect", items_per_thread=1, block=512),
              "region": pv.variant(agg="global", ht="perfect")}
        s.chain = ctx.run_chain(workloads.q5_chain(case["regions"]), vs, pv.ht_variant("perfect"))
        res, groups = s.chain.steps[-1][2], 5
    elif f == "adhoc_agg":
        s.register({"li": lineitem_table(d, n)})
        plan = {"fact": "li", "filters": [["date", "between", DAY0 + 60, DAY0 + 59 + case["days"]],
                                          ["disc", "between", 5, 7], ["qty", "lt", case["qty_lt"]]],
                "aggs": [["sum", [["x", "price"], ["x", "disc"]]], ["count"]]}
        res = ctx.run(plan, pv.variant())
        s.handles.append(res)
        s.deliver_to(res, device=False)
        return s
    elif f == "adhoc_group":
        s.register({"li": lineitem_table(d, n)})
        plan = {"fact": "li", "filters": [["qty", "ge", case["qty_ge"]]], "group_by": ["k1", "k2"],
                "aggs": [["sum", [["x", "qty"]]], ["sum", [["x", "price"]]], ["min", [["x", "price"]]],
                         ["max", [["x", "price"]]], ["count"]]}
        res, s.spans, groups = ctx.run(plan, pv.variant(agg="local", ht="perfect")), (2,), 2 * 66 + 89 + 1
    else:
        s.register(join_tables(d, n))
        y0 = datagen.STAR3_YEAR0
        plan = {"fact": "fact",
                "builds": [{"table": "d_cust", "key": "key", "filters": [["region", "eq", 2]], "payload": []},
                           {"table": "d_date", "key": "key", "filters": [["year", "lt", y0 + case["years"]]],
                            "payload": ["year"]}],
                "probes": [{"build": 0, "fk": "fk_cust"}, {"build": 1, "fk": "fk_date"}],
                "group_by": [["payload", 1, 0]], "aggs": [["sum", [["x", "revenue"]]], ["count"]]}
        hts = ctx.build_all(plan, pv.ht_variant("perfect"))
        res, groups = ctx.run(plan, pv.variant(agg="local", ht="perfect"), hts), y0 + 7
        s.handles += hts
    if s.chain is None:
        s.handles.insert(0, res)
    s.deliver_to(res, device=True, groups=groups)
    if s.chain is not None:
        s.chain.capture()
        s.chain.launch()
        ctx.sync()
    return s


def run(state):
    f = state.family
    if f == "mlp":
        return run_mlp(state)
    ctx = state.ctx
    if f == "query":
        ctx.cols.update(state.names_now)
        return ctx.query(state.plan, state.var)
    if state.chain is not None:
        state.chain.launch()
    else:
        ctx.rerun(state.res)
    ctx._check(ctx.lib.pv_enqueue_fetch_rows(ctx.h, state.res, *state.fetch_args))
    if state.device_groups:
        with torch.cuda.stream(ctx.stream):
            rows = state.rows
            if f == "group_hash":  # ORDER BY key
                state.table[:, :state.live] = rows.index_select(1, torch.argsort(rows[0]))
            else:
                at = rows[0]
                for i, span in enumerate(state.spans):
                    at = torch.add(rows[i + 1], at, alpha=span)
                state.table.index_copy_(1, at, rows)
    return state.outputs


# ---- the cost model's training step ---------------------------------------------

ADAM = dict(lr=5e-4, b1=0.9, b2=0.999, eps=1e-8)
STEP0 = 200  # steps taken before


def mlp_inputs(case, d):
    """Standardised features, log times, and a network some hundred steps into its training."""
    B, F, H = case["batch"], case["features"], costmodel.H

    def normal(*shape):
        return torch.randn(shape, generator=d.g, device="cuda", dtype=torch.float32)

    n = costmodel.n_params(F)
    p = torch.cat([normal(F * H) * math.sqrt(2.0 / F), 0.1 * normal(H), normal(H * H) * math.sqrt(2.0 / H),
                   0.1 * normal(H), normal(H) * math.sqrt(2.0 / H), 0.1 * normal(1)])
    x = 3.0 + 2.0 * normal(B, F)
    t = torch.sin(x[:, 0]) + 0.5 * x[:, 1] + 0.1 * normal(B)
    return {"p": p, "x": x, "t": t, "mu": torch.full((F,), 3.0, device="cuda"),
            "sigma": torch.full((F,), 2.0, device="cuda"), "m": 0.01 * normal(n), "v": 1e-3 * (0.1 + normal(n).abs())}


class MlpState(dict):
    family = "mlp"


def prepare_mlp(case, d):
    B, F, H = case["batch"], case["features"], costmodel.H
    s = MlpState(mlp_inputs(case, d), B=B, F=F, step=STEP0)
    s["ctx"] = context()

    def empty(n):
        return torch.empty(n, dtype=torch.float32, device="cuda")

    s.update(y=empty(B), act=empty(B * 2 * H), dz=empty(B * (2 * H + 1)), grad=empty(s["p"].numel()), loss=empty(1))
    s["ptr"] = {k: ctypes.c_void_p(v.data_ptr()) for k, v in s.items() if isinstance(v, torch.Tensor)}
    torch.cuda.synchronize()
    return s


def run_mlp(s):
    ctx, q, B, F = s["ctx"], s["ptr"], s["B"], s["F"]
    lib, h = ctx.lib, ctx.h
    s["step"] += 1
    ctx._check(lib.pv_mlp_forward(h, q["p"], q["x"], q["mu"], q["sigma"], B, F, q["y"], q["act"]))
    ctx._check(lib.pv_mlp_backward(h, q["p"], q["x"], q["mu"], q["sigma"], q["act"], q["y"], q["t"], B, F, q["dz"],
                                   q["grad"], q["loss"]))
    ctx._check(lib.pv_mlp_adam(h, q["p"], q["grad"], q["m"], q["v"], s["p"].numel(), ADAM["lr"], ADAM["b1"],
                               ADAM["b2"], ADAM["eps"], s["step"]))
    return [s[k] for k in ("y", "act", "loss", "grad", "p", "m", "v")]


def exact(case, seed):
    """The training step in 64 bits.  Every other case returns whole numbers, which have to be equal anyway."""
    if case["family"] != "mlp":
        return None
    F, H = case["features"], costmodel.H
    s = {k: v.double() for k, v in mlp_inputs(case, Draws(seed)).items()}
    p = s["p"].clone().requires_grad_(True)
    w1, b1, w2, b2, w3, b3 = torch.split(p, [F * H, H, H * H, H, H, 1])
    z1 = ((s["x"] - s["mu"]) / s["sigma"]) @ w1.view(F, H) + b1
    z2 = torch.relu(z1) @ w2.view(H, H) + b2
    y = torch.relu(z2) @ w3 + b3
    loss = ((y - s["t"]) ** 2).mean()
    grad, = torch.autograd.grad(loss, p)
    step = STEP0 + 1
    m = ADAM["b1"] * s["m"] + (1 - ADAM["b1"]) * grad
    v = ADAM["b2"] * s["v"] + (1 - ADAM["b2"]) * grad * grad
    new = p.detach() - ADAM["lr"] * (m / (1 - ADAM["b1"] ** step)) / (torch.sqrt(v / (1 - ADAM["b2"] ** step)) +
                                                                     ADAM["eps"])
    return [y.detach(), torch.cat([z1, z2], 1).detach().reshape(-1), loss.detach().reshape(1), grad, new, m, v]


# ---- bytes and operations -------------------------------------------------------

def touched(keep, size):
    """Share of a column's 32-byte sectors that hold a row kept with probability `keep`."""
    return 1.0 - (1.0 - keep) ** (32 // size)


def work(case):
    """Bytes: the first column in full; of each later one the sectors that hold a row still alive; the result once."""
    f = case["family"]
    if f == "mlp":
        B, F, H = case["batch"], case["features"], costmodel.H
        n = costmodel.n_params(F)
        return {"bytes": 4.0 * (B * (F + 2) + B * 2 * H + 7 * n),
                "flops": 2.0 * B * (2 * (F * H + H * H + H) + H * H)}
    n = case["rows"]
    if f in ("query", "filter_agg", "project"):
        a, b = case["a_lt"] / 100, case["b_n"] / 100
        out = n * a * b * 12 if f == "project" else 16
        return {"bytes": n * (4 + 4 * touched(a, 4) + 8 * touched(a * b, 8)) + out, "flops": 0}
    if f == "lowcard":
        return {"bytes": 38.0 * n + 4 * 80, "flops": 0}
    if f == "group":
        return {"bytes": 12.0 * n + 24 * min(n, case["groups"]), "flops": 0}
    if f == "group_hash":
        return {"bytes": n * (8 + 4 * touched(case["val_lt"] / 1e6, 4)) + 24 * min(n, case["groups"]), "flops": 0}
    if f == "star":
        keep, total = 1.0, 0.0
        for t in ("t_c", "t_d", "t_a", "t_b"):  # the probes' order
            total += 4 * touched(keep, 4)
            keep *= case[t] / 100
        dims = sum(rows * (12 if groups else 8) for _, rows, groups in datagen.STAR_DIMS)
        return {"bytes": n * (total + 8 * touched(keep, 8)) + dims + 300 * 32, "flops": 0}
    if f == "q5":
        nations = case["regions"] / 5
        year = 365 / datagen.TPCH_DAYS
        keep = nations * year
        orders, cust = n // 4, n // 40
        return {"bytes": n * (4 + 16 * touched(keep, 8)) + orders * (4 + 4 * touched(year, 4) + 4 * touched(keep, 4)) +
                cust * (4 + 4 * touched(nations, 4)), "flops": 0}
    if f == "adhoc_agg":
        k1 = min(1.0, case["days"] / NDAYS)
        k2 = k1 * 3 / 11
        k3 = k2 * min(1.0, (case["qty_lt"] - 1) / 50)
        return {"bytes": n * (4 + 8 * touched(k1, 8) + 8 * touched(k2, 8) + 8 * touched(k3, 8)), "flops": 0}
    if f == "adhoc_group":
        k = (51 - case["qty_ge"]) / 50
        return {"bytes": n * (8 + 2 * touched(k, 1) + 8 * touched(k, 8)) + 4 * 56, "flops": 0}
    k = min(1.0, 365 * case["years"] / 2_556)
    return {"bytes": n * (4 + 4 * touched(0.2, 4) + 8 * touched(0.2 * k, 8)) + 30_000 * 8 + 2_556 * 8, "flops": 0}
