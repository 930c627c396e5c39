"""Performance cases of the plan simulator and the plan searches.

Every case is a call (or the two calls, new availability and search) that a planner built on this package makes:
searching a space for one job, re-planning when availability changed, simulating a batch of candidate plans it has
made itself, and the per-stage searches.  Workloads are the package's own (`workloads.CONFIGS`): a case takes a
configuration's model, cluster, space and objective, with a profile and an availability snapshot of its own per seed.

A case names what is called ("call") and, per call:
  plan       sailor_set_availability + sailor_plan on a context that exists ("mode": pruned, every, screen, degree)
  cold       sailor_create, sailor_set_availability, sailor_plan, sailor_destroy: a planner run once per job
  records    sailor_simulate on "n" explicit plans ("where": device, pinned or numpy; "plans": random or space)
  mixed      sailor_simulate_mixed on "n" plans of up to 32 stages whose stages mix GPU types (device)
  plan_mixed sailor_plan_mixed: search over such plans
  dp         sailor_plan_dp: a GPU type per stage by dynamic programming ("budget": with the budget loop)
"depth" is the deepest pipeline kept of the configuration's list; "zoned" gives every zone its own prices, as clouds
do by region; "poly" gives every link a fitted bandwidth polynomial.
"""
from __future__ import annotations

import weakref

import numpy as np
import torch

from paper_2504_17096_b200 import binding as B
from paper_2504_17096_b200 import workloads as W

MODES = {"pruned": 0, "every": B.FLAG_EVAL_ALL, "screen": B.FLAG_EVAL_ALL | B.FLAG_F32_SCREEN, "degree": B.FLAG_DEGREE_ORDER}
BASE_PLANS = 1 << 13          # distinct plans of a large batch; the batch draws from them


def listed():
    return [
        # the smallest call: one job on one zone, 6 768 candidates; launch and hand-over latencies count
        dict(name="plan_one_zone", call="plan", config=1, depth=24, mode="pruned", k=8, zoned=False, poly=False),
        # an elastic job re-plans after an availability change: two passes, budget relative to the cheapest plan
        dict(name="replan_budget", call="plan", config=2, depth=32, mode="pruned", k=4, zoned=False, poly=False),
        # a large space the way a planner searches it, five zones with regional prices, throughput per USD
        dict(name="plan_five_zones", call="plan", config=3, depth=48, mode="pruned", k=32, zoned=True, poly=False),
        # the exhaustive stress sweep: every candidate's time and cost
        dict(name="plan_every", call="plan", config=5, depth=16, mode="every", k=32, zoned=False, poly=False),
        # the same kind of sweep with the binary32 screen, recomputation on and off
        dict(name="plan_screened", call="plan", config=3, depth=48, mode="screen", k=32, zoned=False, poly=False),
        # a planner invoked once per job: fresh tables, first search of the space
        dict(name="plan_cold", call="cold", config=2, depth=32, mode="pruned", k=8, zoned=False, poly=False),
        # a handful of plans from host arrays (a scheduler comparing its own proposals)
        dict(name="records_few_numpy", call="records", config=2, n=1000, where="numpy", plans="random", zoned=False, poly=False),
        # a large batch resident on the device, up to 96 stages and 16 runs a plan
        dict(name="records_many", call="records", config=5, n=4194301, where="device", plans="random", zoned=False, poly=False),
        # plans whose stages mix GPU types among their replicas
        dict(name="mixed_many", call="mixed", config=5, n=262147, zoned=False, poly=False),
        # search over such plans: two pipeline depths, replicas split in quarters
        dict(name="plan_mixed", call="plan_mixed", config=2, depth=4, parts=4, k=32, zoned=False, poly=False),
        # a GPU type per stage, 48-block model on five zones
        dict(name="dp_five_zones", call="dp", config=3, depth=48, orders=1, budget=False, k=32, zoned=False, poly=False),
        # the same recursion steered by a budget, pipelines of up to 8 stages, every zone order
        dict(name="dp_budget", call="dp", config=2, depth=8, orders=4, budget=True, k=32, zoned=False, poly=False),
    ]


def _log_size(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    call = rng.choice(["plan", "plan", "plan", "cold", "records", "records", "mixed", "plan_mixed", "dp"])
    c = dict(call=call, zoned=rng.random() < 0.3, poly=rng.random() < 0.2)
    if call in ("plan", "cold"):
        c["config"] = rng.choice([1, 2, 3, 5, 6])
        c["depth"] = rng.choice([p for p in W.CONFIGS[c["config"]]().p_values if p >= 8])      # shallower: few plans fit
        c["mode"] = "pruned" if call == "cold" else rng.choice(["pruned", "pruned", "every", "screen", "degree"])
        if c["mode"] == "screen" and c["config"] in (2, 6):       # the screen covers unconstrained searches
            c["mode"] = "every"
        if c["mode"] == "degree" and c["config"] == 3:            # the order is defined for throughput and for cost
            c["mode"] = "pruned"
        c["k"] = rng.randint(1, 32)
    elif call == "records":
        c.update(config=rng.choice([1, 2, 3, 5]), where=rng.choice(["device", "device", "pinned", "numpy"]),
                 plans=rng.choice(["random", "space"]))
        c["n"] = _log_size(rng, 1, 4194301 if c["where"] == "device" else 1 << 20) | rng.randint(0, 1)
    elif call == "mixed":
        c.update(config=rng.choice([1, 2, 3, 5]), n=_log_size(rng, 1, 262147))
    elif call == "plan_mixed":
        c.update(config=2, depth=rng.choice([2, 4]), parts=rng.choice([1, 2, 4]), k=rng.randint(1, 32))
    else:
        c.update(config=rng.choice([1, 2, 3, 5]), budget=rng.random() < 0.3, k=rng.randint(1, 32))
        if c["budget"]:
            c["config"] = 2
        w = W.CONFIGS[c["config"]]()
        c["depth"] = 8 if c["budget"] else rng.choice([p for p in w.p_values if p >= 8])
        c["orders"] = rng.randint(1, 4) if w.n_zones == 2 else 1
    return c


# ---- inputs ---------------------------------------------------------------------------------------------------------

def _workload(case, rng):
    """The configuration with a profile and an availability snapshot of its own."""
    w = W.CONFIGS[case["config"]]()
    for name in ("fwd", "bwd", "upd"):
        t = getattr(w, name)
        setattr(w, name, t * rng.lognormal(0.0, 0.02, t.shape))
    shape = w.avail.shape
    if case["config"] == 2:
        w.avail = rng.integers(0, 33, shape).astype(np.uint16)
    elif case["config"] in (3, 5):
        mean, total = (24.0, 512) if case["config"] == 3 else (21.0, 1024)
        a = rng.poisson(mean, shape)
        w.avail = (a * min(1.0, total / a.sum())).astype(np.uint16)
    elif case["config"] == 1:                                      # other jobs have taken a part
        w.avail = (w.avail - rng.integers(0, 5, shape)).astype(np.uint16)
    else:                                                          # the scenario's counts, or some more: fewer miss its throughput
        w.avail = (w.avail + rng.integers(0, 33, shape)).astype(np.uint16)
    if case["zoned"]:
        w.price_per_hour = w.price_per_hour * rng.uniform(0.85, 1.25, (w.n_zones, 1))
    if case["poly"]:
        w = W.with_bandwidth_polynomials(w, int(rng.integers(1 << 30)))
    if "depth" in case:
        w.p_values = [p for p in w.p_values if p <= case["depth"]]
    return w


class Context:
    """A context on the current device and stream, destroyed with the object."""

    def __init__(self, w):
        self.ctx = B.sailor_create(w, torch.cuda.current_device(), torch.cuda.current_stream().cuda_stream)
        weakref.finalize(self, B.sailor_destroy, self.ctx)
        B.sailor_set_availability(self.ctx, w.avail)


def _depths(w, n, rng, p_max):
    deepest = min(w.n_blocks, p_max)
    some = rng.choice(np.array(w.p_values), n)
    return np.minimum(np.where(rng.random(n) < 0.7, some, rng.integers(1, deepest + 1, n)), deepest)


def _lengths(total, parts, columns, rng):
    """Per row: `total` cut at parts - 1 random places into at most `columns` positive lengths (zeros at the end)."""
    n = total.size
    cuts = 1 + (rng.random((n, columns - 1)) * np.maximum(total - 1, 1)[:, None]).astype(np.int64)
    cuts = np.where(np.arange(columns - 1)[None, :] < (parts - 1)[:, None], cuts, total[:, None])
    cuts = np.sort(np.minimum(cuts, total[:, None]), axis=1)
    edges = np.concatenate([np.zeros((n, 1), np.int64), cuts, total[:, None]], axis=1)
    lens = np.diff(edges, axis=1)
    return np.take_along_axis(lens, np.argsort(lens == 0, axis=1, kind="stable"), axis=1)


def _records(case, w, ctx, n, rng):
    """n plan records: with random runs, or the candidates at random flat indices of the configuration's space."""
    if case["plans"] == "space":
        space = B.make_space(w)
        flats = rng.integers(0, B.sailor_space_size(ctx, space), n)
        return np.frombuffer(b"".join(bytes(B.sailor_decode(ctx, space, int(f))) for f in flats), dtype=B.REC_DTYPE).copy()
    P = _depths(w, n, rng, 96)
    lens = _lengths(P, 1 + (rng.random(n) * np.minimum(P, 16)).astype(np.int64), 16, rng)
    used = lens > 0
    return B.pack_records({
        "P": P, "mbs_idx": rng.integers(0, len(w.mbs_values), n), "rc": rng.choice(np.array(w.rc_values), n),
        "n_runs": used.sum(axis=1), "D": rng.choice(np.array(w.d_values), n), "n_stages": lens,
        "type": np.where(used, rng.integers(0, w.n_types, lens.shape), 0),
        "zone": np.where(used, rng.integers(0, w.n_zones, lens.shape), 0),
        "tp_idx": np.where(used, rng.integers(0, len(w.tp_values), lens.shape), 0)})


MIXED_STAGES = 32


def _mixed_records(w, n, rng):
    """n plans of up to 32 stages; three quarters of them split a stage's replicas into up to four groups."""
    S, out = MIXED_STAGES, np.zeros(n, dtype=B.mixed_dtype(MIXED_STAGES))
    P, D = _depths(w, n, rng, S), rng.choice(np.array(w.d_values), n)
    out["P"], out["D"], out["mbs_idx"] = P, D, rng.integers(0, len(w.mbs_values), n)
    out["rc"] = rng.choice(np.array(w.rc_values), n)
    stage = np.arange(S)[None, :] < P[:, None]
    moves = np.where(rng.random((n, S)) < 0.3, np.arange(S)[None, :], 0)
    zone = np.take_along_axis(rng.integers(0, w.n_zones, (n, S)), np.maximum.accumulate(moves, axis=1), axis=1)
    parts = 1 + (rng.random((n, S)) * np.minimum(D, 4)[:, None]).astype(np.int64)
    parts[rng.random(n) < 0.25] = 1
    count = _lengths(np.repeat(D, S), parts.reshape(-1), 4, rng).reshape(n, S, 4) * stage[:, :, None]
    out["stage"]["zone"] = zone * stage
    out["stage"]["n_groups"] = (count > 0).sum(axis=2)
    out["stage"]["group"]["count"] = count
    out["stage"]["group"]["type"] = np.where(count > 0, rng.integers(0, w.n_types, count.shape), 0)
    out["stage"]["group"]["tp_idx"] = np.where(count > 0, rng.integers(0, len(w.tp_values), count.shape), 0)
    return out


def _many(base, n, seed, pinned=False):
    """A batch of n records drawn from `base`, as bytes on the device (or in pinned host memory)."""
    rows = torch.from_numpy(base.view(np.uint8).reshape(base.size, -1)).cuda()
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    pick = rows[torch.randint(0, base.size, (n,), generator=g, device="cuda")] if n > base.size else rows[:n].contiguous()
    return pick.cpu().pin_memory() if pinned else pick


def _result_buffers(n, **where):
    make = dict(dtype=torch.float64, **where), dict(dtype=torch.int64, **where), dict(dtype=torch.int32, **where)
    return [torch.zeros(n, **make[j]) for j in (0, 1, 0, 2)]       # t_iter, peak_mem, cost, status


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    w = _workload(case, rng)
    s = {"case": case, "w": w}
    if case["call"] == "cold":
        s["space"], s["objective"] = B.make_space(w), B.make_objective(w, flags=MODES[case["mode"]])
        return s
    s["handle"] = Context(w)
    ctx = s["ctx"] = s["handle"].ctx
    if case["call"] == "plan":
        s["space"], s["objective"] = B.make_space(w), B.make_objective(w, flags=MODES[case["mode"]])
    elif case["call"] == "records":
        base = _records(case, w, ctx, min(case["n"], BASE_PLANS), rng)
        if case["where"] == "numpy":
            s["plans"] = base[rng.integers(0, base.size, case["n"])]
        else:
            pinned = case["where"] == "pinned"
            s["plans"] = _many(base, case["n"], seed, pinned)
            s["out"] = _result_buffers(case["n"], **({"pin_memory": True} if pinned else {"device": "cuda"}))
    elif case["call"] == "mixed":
        s["plans"] = _many(_mixed_records(w, min(case["n"], BASE_PLANS), rng), case["n"], seed)
        s["out"] = _result_buffers(case["n"], device="cuda")
    elif case["call"] == "plan_mixed":
        s["space"] = B.make_mixed_space(w, case["parts"], [min(g, len(w.tp_values) - 1) for g in range(w.n_types)],
                                        mbs_idx=[1], d_values=[4, 8])
        s["objective"] = B.Objective(W.OBJ_MAX_THROUGHPUT, 0, 0.0, 0.0, 0.0)
    else:
        s["space"] = B.make_space(w)
        s["orders"] = ([list(range(w.n_zones))] if case["orders"] == 1 else B.all_zone_orders(w.n_zones))[: case["orders"]]
        s["limit"] = 0.0
        if case["budget"]:                                         # 1.2 x the cheapest plan of the segment space
            cheapest, _ = B.sailor_plan(ctx, s["space"], B.Objective(W.OBJ_MIN_COST, 0, 0.0, 0.0, 0.0), 1)
            s["limit"] = 1.2 * cheapest[0].cost if cheapest else 1.0
    return s


# ---- one pass -------------------------------------------------------------------------------------------------------

def _column(values, k, dtype=np.float64):
    """The values as an array of k entries; slots without a result hold -1."""
    return np.array(values + [-1] * (k - len(values)), dtype)


def _found(best, k, counts):
    return {"flat": _column([r.flat for r in best], k, np.int64), "score": _column([r.score for r in best], k),
            "t_iter": _column([r.t_iter for r in best], k), "cost": _column([r.cost for r in best], k),
            "peak_mem": _column([r.peak_mem for r in best], k, np.int64), "counts": counts}


def _counts(st):
    return np.array([st.n_total, st.n_invalid, st.n_oom, st.n_over_avail, st.n_over_constraint, st.n_feasible], np.int64)


def run(s):
    case, w = s["case"], s["w"]
    call, k = case["call"], case.get("k", 0)
    if call == "cold":
        ctx = B.sailor_create(w, torch.cuda.current_device(), torch.cuda.current_stream().cuda_stream)
        try:
            B.sailor_set_availability(ctx, w.avail)
            best, st = B.sailor_plan(ctx, s["space"], s["objective"], k)
        finally:
            B.sailor_destroy(ctx)
        return _found(best, k, _counts(st))
    ctx = s["ctx"]
    if call == "plan":
        B.sailor_set_availability(ctx, w.avail)
        best, st = B.sailor_plan(ctx, s["space"], s["objective"], k)
        return dict(_found(best, k, _counts(st)), cheapest=st.min_feasible_cost, budget=st.budget_used)
    if call == "records":
        if case["where"] == "numpy":
            return B.sailor_simulate(ctx, s["plans"])
        ask = B.sailor_simulate_device if case["where"] == "device" else B.sailor_simulate_host
        ask(ctx, s["plans"].data_ptr(), case["n"], *(o.data_ptr() for o in s["out"]))
        return s["out"]
    if call == "mixed":
        B.sailor_simulate_mixed_device(ctx, s["plans"].data_ptr(), case["n"], *(o.data_ptr() for o in s["out"]),
                                       record_bytes=s["plans"].shape[1])
        return s["out"]
    if call == "plan_mixed":
        best, st = B.sailor_plan_mixed(ctx, s["space"], s["objective"], k)
        return dict(_found(best, k, _counts(st)), cheapest=st.min_feasible_cost)
    best, st = B.sailor_plan_dp(ctx, s["space"], s["orders"], k, budget=s["limit"], budget_loop=case["budget"])
    return {"value": _column([r.value for r in best], k), "t_iter": _column([r.t_iter for r in best], k),
            "cost": _column([r.cost for r in best], k), "peak_mem": _column([r.peak_mem for r in best], k, np.int64),
            "config": _column([r.config for r in best], k, np.int64), "order": _column([r.order for r in best], k, np.int64),
            "types": np.frombuffer(b"".join([bytes(r.type) for r in best] + [b"\xff" * B.P_MAX] * (k - len(best))), np.uint8),
            "counts": np.array([st.n_problems, st.n_solved, st.n_over_constraint, st.n_unfinished], np.int64)}


# ---- what a pass cannot do without -----------------------------------------------------------------------------------

def _configs(w):
    return len(w.mbs_idx) * len(w.tp_idx) * len(w.rc_values) * len(w.d_values)


def _table_bytes(w):
    return sum(getattr(w, t).nbytes for t in ("fwd", "bwd", "upd", "act_saved", "act_ckpt", "act_work", "price_per_hour",
                                              "inter_inv_bw", "intra_inv_bw", "zone_inv_bw", "egress", "avail"))


def _dp_states(w):
    """Reachable (stage, type, zone, stages per type so far) states of all configurations, one zone order."""
    total = 0
    for P in w.p_values:
        for tp in (w.tp_values[i] for i in w.tp_idx):
            for D in w.d_values:
                for z in range(w.n_zones):
                    ways = np.zeros(P + 1)
                    ways[0] = 1
                    for g in range(w.n_types):
                        cap = int(w.avail[z, g]) // (D * tp)
                        if 1 <= cap < P:
                            ways = np.convolve(ways, np.ones(cap + 1))[: P + 1]
                    total += w.n_types * float(np.cumsum(ways)[1:].sum())
    return total * len(w.mbs_idx) * len(w.rc_values)


def work(case):
    """Bytes: the tables or records read once and the results written once.  Operations: binary64 additions,
    multiplications and comparisons that the definition of a plan's time and cost leaves when sums over equal
    beginnings are formed once."""
    w = W.CONFIGS[case["config"]]()
    call, n = case["call"], case.get("n", 0)
    if "depth" in case:
        w.p_values = [p for p in w.p_values if p <= case["depth"]]
    if call in ("plan", "cold"):
        base = _configs(w)
        if case["mode"] in ("every", "screen"):      # a candidate: its last segment's stages (time and price), then the closing terms
            flops = sum(base * w.radix ** min(p, w.seg_max) * (2.0 * -(-p // w.seg_max) + 12.0) for p in w.p_values)
        else:                                        # a configuration: time, memory and update of every stage on every type
            flops = sum(base * p * w.n_types * 12.0 for p in w.p_values)
        return {"bytes": float(_table_bytes(w) + case["k"] * 120), "flops": flops}
    if call == "records":                            # two additions per stage (19 on average in random plans, 9 in spaces)
        return {"bytes": 100.0 * n, "flops": n * (60.0 if case["plans"] == "random" else 40.0)}
    if call == "mixed":                              # about 9 stages of 20 B, five different pipelines a plan
        return {"bytes": n * (8 + 9 * 20 + 28.0), "flops": n * 9 * 5 * 4.0}
    if call == "plan_mixed":
        combs = {1: 3, 2: 6, 4: 15}[case["parts"]]
        return {"bytes": float(_table_bytes(w) + case["k"] * 1976), "flops": sum(2.0 * (w.n_zones * combs) ** min(p, 4) * p * 12 for p in w.p_values)}
    if case["budget"]:                               # the cheapest conceivable rest of every pipeline, per order
        flops = sum(_configs(w) * p * w.n_types * w.n_zones * 5.0 for p in w.p_values) * case["orders"]
    else:                                            # every state tries every type for the next stage
        flops = _dp_states(w) * w.n_types * 8.0 * case["orders"]
    return {"bytes": float(_table_bytes(w) + case["k"] * 248), "flops": flops}


def tolerance(case):
    # the order of the binary64 operations is part of the interface (include/sailor.h): results are the same bits
    return "exact"
