"""GPU parity of sailor_simulate_mixed (plans whose stages mix GPU types among their replicas; Sailor
Sec. 4.2, Sec. 4.3) against the oracle on the same seeded plans: status and bytes bit-exact, times and
costs within 1e-5 relative and identical in their bits."""
import glob
import json
import math
import os

import numpy as np
import pytest

from helpers import GOLDEN, REL_TOL_F64, rel_close, workload_from_tables
from oracle.binding import Oracle
from paper_2504_17096_b200 import binding as B
from paper_2504_17096_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _needs_cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("the gpu tests need a CUDA device")


class Ctx:
    def __init__(self, w):
        self.ctx = B.sailor_create(w, 0, 0)
        B.sailor_set_availability(self.ctx, w.avail)

    def __enter__(self):
        return self

    def __exit__(self, *exc):
        B.sailor_destroy(self.ctx)


def assert_equal(gpu, orc, what):
    t, m, c, s = gpu
    so, to, co, mo = orc
    assert np.array_equal(s, so), f"{what}: status differs at {np.flatnonzero(s != so)[:5]}"
    assert np.array_equal(m, mo), f"{what}: peak memory differs at {np.flatnonzero(m != mo)[:5]}"
    assert rel_close(t, to, REL_TOL_F64) and rel_close(c, co, REL_TOL_F64), what
    ok = ~np.isnan(to)
    assert np.array_equal(np.isnan(t), np.isnan(to)) and np.array_equal(np.isnan(c), np.isnan(co)), what
    assert np.array_equal(t[ok].view(np.uint64), to[ok].view(np.uint64)), f"{what}: t_iter bits"
    assert np.array_equal(c[ok].view(np.uint64), co[ok].view(np.uint64)), f"{what}: cost bits"


def test_hand_worked_mixed_plans():
    for path in sorted(glob.glob(os.path.join(GOLDEN, "mixed", "*.json"))):
        with open(path) as f:
            case = json.load(f)
        w = workload_from_tables(case["tables"], case["name"])
        plan = {**case["plan"], "stages": [{"zone": s["zone"], "groups": [tuple(g) for g in s["groups"]]}
                                           for s in case["plan"]["stages"]]}
        with Ctx(w) as cx:
            t, m, c, s = B.sailor_simulate_mixed(cx.ctx, B.pack_mixed_plans([plan]))
        e = case["expect"]
        assert s[0] == e["status"] and m[0] == e["peak_mem"]
        assert t[0] == pytest.approx(e["t_iter"], rel=1e-12) and c[0] == pytest.approx(e["cost"], rel=1e-12)


@pytest.mark.parametrize("cfg", [1, 2, 3, 5, 6])
def test_random_mixed_plans_match_oracle(cfg):
    w = W.CONFIGS[cfg]()
    n = 6007                              # several blocks and a ragged tail
    plans = W.random_mixed_plans(w, n, seed=300 + cfg)
    with Ctx(w) as cx:
        gpu = B.sailor_simulate_mixed(cx.ctx, B.pack_mixed_plans(plans))
    assert_equal(gpu, Oracle(w).simulate_mixed_batch(plans), f"cfg{cfg}")
    assert len(np.unique(gpu[3])) >= 3


def test_mixed_tiny_with_latency_polynomials_and_recomputation():
    for w in (W.tiny(seed=5, n_types=3, n_zones=2, L=7, p_values=[1, 2, 3, 7]),
              W.with_bandwidth_polynomials(W.tiny(seed=41, n_types=3, n_zones=2), seed=1),
              W.tiny(seed=21, n_types=8, n_zones=8, L=32, p_values=[32, 16, 5], d_values=(1, 2, 5, 64), gbs=640)):
        plans = W.random_mixed_plans(w, 3000, seed=17)
        with Ctx(w) as cx:
            gpu = B.sailor_simulate_mixed(cx.ctx, B.pack_mixed_plans(plans))
        assert_equal(gpu, Oracle(w).simulate_mixed_batch(plans), w.name)


@pytest.mark.parametrize("cfg", [0, 5])
def test_deep_mixed_plans_match_oracle(cfg):
    """Plans of up to 96 stages (a lane owns up to three stages): the full records and records cut to the deepest plan."""
    w = W.CONFIGS[cfg]() if cfg else W.tiny(seed=23, n_types=8, n_zones=8, L=96, p_values=[96, 65, 64, 33, 32, 5],
                                            d_values=(1, 2, 5, 64), gbs=640)
    plans = W.random_mixed_plans(w, 4001, seed=500 + cfg, p_max=96)
    depths = [p["P"] for p in plans]
    assert max(depths) > 64 and sum(1 for d in depths if 32 < d <= 64) > 0 and min(depths) <= 32
    orc = Oracle(w).simulate_mixed_batch(plans)
    with Ctx(w) as cx:
        assert_equal(B.sailor_simulate_mixed(cx.ctx, B.pack_mixed_plans(plans, stages=B.MIX_P_MAX)), orc, f"cfg{cfg} full records")
        assert_equal(B.sailor_simulate_mixed(cx.ctx, B.pack_mixed_plans(plans)), orc, f"cfg{cfg} cut records")
        # the boundaries of the lane tiles, one plan each
        edge = [p for p in plans if p["P"] in (31, 32, 33, 63, 64, 65, 95, 96)]
        if edge:
            assert_equal(B.sailor_simulate_mixed(cx.ctx, B.pack_mixed_plans(edge)), Oracle(w).simulate_mixed_batch(edge), "tile edges")


def test_mixed_record_sizes():
    """sailor_simulate_mixed_strided: record sizes it takes, and a plan deeper than its record."""
    import torch
    w = W.config1()
    plans = [p for p in W.random_mixed_plans(w, 800, seed=9) if p["P"] <= 8]
    orc = Oracle(w).simulate_mixed_batch(plans)
    with Ctx(w) as cx:
        for stages in (8, 10, 32, 96):
            assert_equal(B.sailor_simulate_mixed(cx.ctx, B.pack_mixed_plans(plans, stages=stages)), orc, f"{stages} stages per record")
        L = B.load()
        packed = B.pack_mixed_plans(plans, stages=8)
        out = np.empty(len(plans)); st = np.empty(len(plans), np.uint32)
        for bad_bytes in (0, 24, 28, 36, 1936):
            assert L.sailor_simulate_mixed_strided(cx.ctx, packed.ctypes.data, len(plans), bad_bytes, 0, out.ctypes.data, None, None,
                                                   st.ctypes.data) == B.E_ARG
        deep = packed[:3].copy()
        deep["P"][1] = 9                                 # more stages than the record holds
        with pytest.raises(B.SailorError) as e:
            B.sailor_simulate_mixed(cx.ctx, deep)
        assert e.value.code == B.E_RANGE
        d = torch.from_numpy(deep.view(np.uint8).reshape(3, deep.itemsize).copy()).cuda()
        ds = torch.zeros(3, dtype=torch.int32, device="cuda"); dt = torch.zeros(3, dtype=torch.float64, device="cuda")
        B.sailor_simulate_mixed_device(cx.ctx, d.data_ptr(), 3, dt.data_ptr(), 0, 0, ds.data_ptr(), record_bytes=deep.itemsize)
        torch.cuda.synchronize()
        assert ds.cpu().tolist()[1] == B.ST_BAD_RECORD and ds.cpu().tolist()[0] == int(orc[0][0]) and math.isnan(dt.cpu().tolist()[1])


def test_mixed_host_batch_in_chunks():
    """A host batch of more chunks than staging slots (64 MB of records a chunk, three slots), deep plans among them."""
    w = W.config5()
    plans = W.random_mixed_plans(w, 3001, seed=31, p_max=96)
    base = B.pack_mixed_plans(plans, stages=B.MIX_P_MAX)            # 1 928 B a record: 34 807 records a chunk
    n = 5 * 34_807 + 1_234
    big = np.tile(base, n // 3001 + 1)[:n]
    so, to, co, mo = Oracle(w).simulate_mixed_batch(plans)
    idx = np.arange(n) % 3001
    with Ctx(w) as cx:
        assert_equal(B.sailor_simulate_mixed(cx.ctx, big), (so[idx], to[idx], co[idx], mo[idx]), "mixed host batch in chunks")


def test_mixed_with_one_group_equals_sailor_simulate():
    """No mixing: the same numbers as the run-length records of sailor_simulate."""
    w = W.config2()
    recs = W.random_plans(w, 2000, seed=4, max_runs=8, hetero_tp=True)
    keep = [j for j in range(2000) if recs["P"][j] <= B.MIX_P_MAX]
    plans = []
    for j in keep:
        stages = []
        for r in range(recs["n_runs"][j]):
            for _ in range(recs["n_stages"][j, r]):
                stages.append({"zone": int(recs["zone"][j, r]),
                               "groups": [(int(recs["type"][j, r]), int(recs["tp_idx"][j, r]), int(recs["D"][j]))]})
        plans.append({"P": int(recs["P"][j]), "mbs_idx": int(recs["mbs_idx"][j]), "rc": int(recs["rc"][j]),
                      "D": int(recs["D"][j]), "stages": stages})
    with Ctx(w) as cx:
        t, m, c, s = B.sailor_simulate(cx.ctx, B.pack_records(recs))
        tm, mm, cm, sm = B.sailor_simulate_mixed(cx.ctx, B.pack_mixed_plans(plans))
    keep = np.array(keep)
    assert np.array_equal(s[keep], sm) and np.array_equal(m[keep], mm)
    ok = ~np.isnan(tm)
    assert np.array_equal(t[keep][ok].view(np.uint64), tm[ok].view(np.uint64))
    assert np.array_equal(c[keep][ok].view(np.uint64), cm[ok].view(np.uint64))


def test_mixed_device_pointers_empty_and_bad_records():
    import torch
    w = W.config1()
    plans = W.random_mixed_plans(w, 1500, seed=8)
    packed = B.pack_mixed_plans(plans)
    with Ctx(w) as cx:
        t, m, c, s = B.sailor_simulate_mixed(cx.ctx, np.zeros(0, dtype=B.MIX_DTYPE))
        assert t.size == 0
        n = packed.size
        d = torch.from_numpy(packed.view(np.uint8).reshape(n, packed.itemsize).copy()).cuda()
        dt = torch.empty(n, dtype=torch.float64, device="cuda"); dc = torch.empty(n, dtype=torch.float64, device="cuda")
        dm = torch.empty(n, dtype=torch.int64, device="cuda"); ds = torch.empty(n, dtype=torch.int32, device="cuda")
        B.sailor_simulate_mixed_device(cx.ctx, d.data_ptr(), n, dt.data_ptr(), dm.data_ptr(), dc.data_ptr(), ds.data_ptr(),
                                       record_bytes=packed.itemsize)
        torch.cuda.synchronize()
        gpu = (dt.cpu().numpy(), dm.cpu().numpy().view(np.uint64), dc.cpu().numpy(), ds.cpu().numpy().view(np.uint32))
        assert_equal(gpu, Oracle(w).simulate_mixed_batch(plans), "device pointers")
        # host records with an index outside its table are refused; on the device the kernel flags them
        bad = packed[:2].copy()
        bad["stage"]["group"]["type"][1, 0, 0] = 7
        with pytest.raises(B.SailorError) as e:
            B.sailor_simulate_mixed(cx.ctx, bad)
        assert e.value.code == B.E_RANGE
        d2 = torch.from_numpy(bad.view(np.uint8).reshape(2, bad.itemsize).copy()).cuda()
        st = torch.zeros(2, dtype=torch.int32, device="cuda"); tt = torch.zeros(2, dtype=torch.float64, device="cuda")
        B.sailor_simulate_mixed_device(cx.ctx, d2.data_ptr(), 2, tt.data_ptr(), 0, 0, st.data_ptr(), record_bytes=bad.itemsize)
        torch.cuda.synchronize()
        assert st.cpu().tolist()[1] == B.ST_BAD_RECORD and not (st.cpu().tolist()[0] & B.ST_BAD_RECORD)
        assert math.isnan(tt.cpu().tolist()[1])


@pytest.mark.parametrize("D,stages", [(2, 1), (32, 5), (33, 32), (64, 31), (65, 33), (300, 96), (7, 64)])
def test_mixed_interval_edges(D, stages):
    """Up to four groups a stage, cut differently.  A warp per plan (calls with 16 plans, plans of more than 32 stages) finds
    intervals between boundaries by one bit per replica up to D = 64 and boundary by boundary beyond, and takes items and
    pipelines in several rounds of 32 lanes when there are many; blocks (40 plans that can be deep) have other ways."""
    w = W.tiny(seed=37, n_types=4, n_zones=3, L=max(stages, 4), gbs=D * 4, d_values=(D,), p_values=[stages])
    w.gpus_per_node[...] = [4, 64, 700, 2]
    rng = W.SplitMix64(D * 131 + stages)
    plans = []
    for j in range(40):
        st = []
        for i in range(stages):
            cuts = sorted({rng.randint(1, D - 1) for _ in range(rng.randint(0, 3))})
            b = [0] + cuts + [D]
            if j % 7 == 3 and i == stages // 2:
                b[-1] += 1                                       # one replica too many: an invalid plan
            st.append({"zone": rng.randint(0, 2) if j % 3 else 1,
                       "groups": [(rng.randint(0, 3), rng.randint(0, 2), b[q + 1] - b[q]) for q in range(len(b) - 1)]})
        plans.append({"P": stages, "mbs_idx": rng.randint(0, 2), "rc": j & 1, "D": D, "stages": st})
    o = Oracle(w)
    ctx = B.sailor_create(w, 0, 0)
    try:
        B.sailor_set_availability(ctx, w.avail)
        packed = B.pack_mixed_plans(plans)
        whole = B.sailor_simulate_mixed(ctx, packed)
        parts = [B.sailor_simulate_mixed(ctx, packed[j : j + 16]) for j in range(0, len(plans), 16)]
    finally:
        B.sailor_destroy(ctx)
    so, to, co, mo = o.simulate_mixed_batch(plans)
    for t, m, c, s in (whole, tuple(np.concatenate(x) for x in zip(*parts))):
        assert np.array_equal(s, so) and np.array_equal(m, mo)
        assert np.array_equal(t, to, equal_nan=True) and np.array_equal(c, co, equal_nan=True)


@pytest.mark.parametrize("D,stages,n,node", [(6, 3, 16, 8), (6, 3, 17, 8),           # either side of the smallest batch that blocks take
                                             (127, 32, 700, 8), (128, 32, 700, 8),   # the largest replica numbers that are kept,
                                             (129, 32, 40, 8),                       # and boundaries numbered in order
                                             (4, 8, 3000, 8190), (4, 8, 300, 8191),  # the largest node its items can tell apart, and a larger one
                                             (3, 1, 5000, 8), (2, 33, 50, 8)])       # one stage; deep plans, and shallow ones among them
def test_mixed_batches_at_their_edges(D, stages, n, node):
    """Plans of one depth (and some shallower) in records of 32 stages and more, most stages with four groups, refused records
    in between: the same bits as the oracle, and the refused ones flagged."""
    import torch
    w = W.tiny(seed=51, n_types=4, n_zones=3, L=max(stages, 32), gbs=D * 4, d_values=(D,), p_values=[stages])
    w.gpus_per_node[...] = [4, node, 700, 2]
    rng = W.SplitMix64(D * 977 + stages)
    plans = []
    for j in range(n):
        P = stages if j % 5 else rng.randint(1, stages)
        st = []
        for i in range(P):
            cuts = sorted({rng.randint(1, D - 1) for _ in range(3 if j % 3 else rng.randint(0, 3))})
            b = [0] + cuts + [D]
            st.append({"zone": rng.randint(0, 2) if j % 3 else 1,
                       "groups": [(rng.randint(0, 3), rng.randint(0, 2), b[q + 1] - b[q]) for q in range(len(b) - 1)]})
        plans.append({"P": P, "mbs_idx": rng.randint(0, 2), "rc": j & 1, "D": D, "stages": st})
    so, to, co, mo = Oracle(w).simulate_mixed_batch(plans)
    packed = B.pack_mixed_plans(plans, stages=max(32, stages + stages % 2))
    refused = np.arange(n) % 11 == 5
    for j in np.flatnonzero(refused):
        if j % 2:
            packed["stage"]["group"]["type"][j, int(packed["P"][j]) - 1, 0] = 4
        else:
            packed["stage"]["n_groups"][j, 0] = 0
    so[refused], mo[refused], to[refused], co[refused] = B.ST_BAD_RECORD, 0, math.nan, math.nan
    with Ctx(w) as cx:
        d = torch.from_numpy(packed.view(np.uint8).reshape(n, packed.itemsize).copy()).cuda()
        dt = torch.empty(n, dtype=torch.float64, device="cuda"); dc = torch.empty(n, dtype=torch.float64, device="cuda")
        dm = torch.empty(n, dtype=torch.int64, device="cuda"); ds = torch.empty(n, dtype=torch.int32, device="cuda")
        B.sailor_simulate_mixed_device(cx.ctx, d.data_ptr(), n, dt.data_ptr(), dm.data_ptr(), dc.data_ptr(), ds.data_ptr(),
                                       record_bytes=packed.itemsize)
        torch.cuda.synchronize()
    gpu = (dt.cpu().numpy(), dm.cpu().numpy().view(np.uint64), dc.cpu().numpy(), ds.cpu().numpy().view(np.uint32))
    assert_equal(gpu, (so, to, co, mo), f"D {D}, {stages} stages, {n} plans")


def _run_on_device(w, packed):
    """t_iter, peak_mem, cost and status of the records, which are copied to the device."""
    import torch
    n = packed.size
    with Ctx(w) as cx:
        d = torch.from_numpy(packed.view(np.uint8).reshape(n, packed.itemsize).copy()).cuda()
        dt = torch.empty(n, dtype=torch.float64, device="cuda"); dc = torch.empty(n, dtype=torch.float64, device="cuda")
        dm = torch.empty(n, dtype=torch.int64, device="cuda"); ds = torch.empty(n, dtype=torch.int32, device="cuda")
        B.sailor_simulate_mixed_device(cx.ctx, d.data_ptr(), n, dt.data_ptr(), dm.data_ptr(), dc.data_ptr(), ds.data_ptr(),
                                       record_bytes=packed.itemsize)
        torch.cuda.synchronize()
    return dt.cpu().numpy(), dm.cpu().numpy().view(np.uint64), dc.cpu().numpy(), ds.cpu().numpy().view(np.uint32)


def _plans_of_degrees(rng, n, degrees, depths):
    """Plans with a degree and a depth of the lists in turn, up to four groups a stage; some boundaries are equal to the
    stage's before, some plans have a replica too many (or too few) or a group without any."""
    plans = []
    for j in range(n):
        D, P, st = degrees[j % len(degrees)], depths[j // 3 % len(depths)], []
        cuts = []
        for i in range(P):
            if not (cuts and rng.randint(0, 3) == 0):
                near = rng.randint(0, 1)                             # boundaries among the first, or anywhere
                cuts = sorted({rng.randint(1, min(D - 1, 9) if near else D - 1) for _ in range(rng.randint(0, 3))}) if D > 1 else []
            b = [0] + cuts + [D]
            if j % 13 == 7 and i == P // 2:
                b[-1] += 1 if D < 65_535 else -1
            groups = [(rng.randint(0, 3), rng.randint(0, 1), b[q + 1] - b[q]) for q in range(len(b) - 1)]
            if j % 17 == 9 and i == P - 1 and len(groups) < 4:
                groups.insert(0, (0, 0, 0))
            st.append({"zone": rng.randint(0, 2) if j % 3 else 1, "groups": groups})
        plans.append({"P": P, "mbs_idx": rng.randint(0, 2), "rc": j & 1, "D": D, "stages": st})
    return plans


@pytest.mark.parametrize("degrees,gbs,n,poly", [((4, 128, 129, 300), 4 * 412_800, 900, False),
                                                ((129, 300), 4 * 412_800, 400, True),
                                                ((65_535, 17, 257, 1), 4 * 65_535, 400, False),
                                                ((256,), 1024, 30_000, False)])        # windows of a hundred plans
def test_mixed_batches_of_unlike_degrees(degrees, gbs, n, poly):
    """Degrees either side of 128 in one batch: of the larger ones a boundary is known by its place among the plan's."""
    w = W.tiny(seed=52, n_types=4, n_zones=3, L=32, gbs=gbs, d_values=(4,), p_values=[32], tp_values=(1, 2))
    w.gpus_per_node[...] = [4, 64, 700, 2]
    w.avail[...] = 60_000
    w.capacity[:] = np.uint64(1 << 44)
    if poly:
        w = W.with_bandwidth_polynomials(w, seed=3)
    few = min(n, 900)
    plans = _plans_of_degrees(W.SplitMix64(len(degrees) * 31 + n), few, degrees, [32, 1, 7, 31, 2, 16, 5])
    so, to, co, mo = Oracle(w).simulate_mixed_batch(plans)
    for D in degrees:
        assert sum(1 for j, p in enumerate(plans) if p["D"] == D and not np.isnan(to[j])) > few // len(degrees) // 2
    idx = np.arange(n) % few
    gpu = _run_on_device(w, B.pack_mixed_plans(plans)[idx])
    assert_equal(gpu, (so[idx], to[idx], co[idx], mo[idx]), f"degrees {degrees}")


def test_mixed_batches_of_large_degrees_keep_pace():
    """6e4 plans of 256 replicas take no longer than twice those of 128 (left to a few warps of a block they took four
    times as long)."""
    import torch
    w = W.config3()
    n, took = 60_000, {}
    with Ctx(w) as cx:
        outs = [torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(3)] + [torch.empty(n, dtype=torch.int32, device="cuda")]
        batches = {}
        for D in (128, 256):
            w.d_values = [D]
            packed = B.pack_mixed_plans(W.random_mixed_plans(w, 2000, seed=77), stages=32)[np.arange(n) % 2000]
            batches[D] = torch.from_numpy(packed.view(np.uint8).reshape(n, -1).copy()).cuda()
        for _ in range(6):                                           # in turn, the fastest of each
            for D, d in batches.items():
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                torch.cuda.synchronize()
                a.record()
                for _ in range(5):
                    B.sailor_simulate_mixed_device(cx.ctx, d.data_ptr(), n, *(o.data_ptr() for o in outs), record_bytes=d.shape[1])
                b.record()
                torch.cuda.synchronize()
                took[D] = min(took.get(D, math.inf), a.elapsed_time(b))
    assert took[256] <= 2.0 * took[128], took


@pytest.mark.parametrize("what", ["items", "plans", "windows"])
def test_mixed_batches_of_full_blocks(what):
    """What a block meets only in large batches, two blocks an SM: twelve plans of 32 stages with four groups each have
    1 536 items, more than the 960 that are evaluated together, so some are put back; plans of one stage, more than the 60
    that are; and more plans than the 256 that are ordered together, degrees either side of 128 among them."""
    import torch
    blocks = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    rng = W.SplitMix64(len(what))
    w = W.tiny(seed=54, n_types=4, n_zones=3, L=32, gbs=4 * 300 * 127, d_values=(4,), p_values=[32], tp_values=(1, 2))
    w.gpus_per_node[...] = [4, 64, 700, 2]
    w.avail[...] = 60_000
    w.capacity[:] = np.uint64(1 << 44)
    if what == "items":
        n, plans = 25 * blocks + 7, []
        for j in range(60):
            st = []
            for i in range(32):
                b = [0] + sorted(rng.randint(0, 40) * 3 + q for q in (1, 2, 3)) + [127]
                st.append({"zone": rng.randint(0, 2), "groups": [(rng.randint(0, 3), rng.randint(0, 1), b[q + 1] - b[q]) for q in range(4)]})
            plans.append({"P": 32, "mbs_idx": rng.randint(0, 2), "rc": j & 1, "D": 127, "stages": st})
    elif what == "plans":
        n, plans = 150 * blocks + 11, _plans_of_degrees(rng, 901, [4, 127, 1], [1, 2, 1])
    else:
        n, plans = 600 * blocks + 13, _plans_of_degrees(rng, 2003, [4, 127, 300, 1], [3, 1, 6, 2])
    so, to, co, mo = Oracle(w).simulate_mixed_batch(plans)
    idx = np.arange(n) % len(plans)
    packed = B.pack_mixed_plans(plans)[idx]
    refused = np.arange(n) % 997 == 500
    packed["stage"]["n_groups"][refused, 0] = 5
    so, to, co, mo = so[idx], to[idx], co[idx], mo[idx]
    so[refused], mo[refused], to[refused], co[refused] = B.ST_BAD_RECORD, 0, math.nan, math.nan
    assert np.count_nonzero(~np.isnan(to)) > n // 2
    assert_equal(_run_on_device(w, packed), (so, to, co, mo), what)


@pytest.mark.parametrize("stages,blocks,types,n", [(8, 8, 3, 4095), (8, 8, 3, 4096), (8, 40, 3, 4096), (32, 8, 3, 4095),   # room, or the model, for few stages
                                                   (16, 16, 3, 1535), (10, 40, 3, 1536), (32, 16, 3, 1536),
                                                   (24, 40, 2, 2047), (24, 24, 2, 2048), (32, 40, 2, 17), (24, 24, 3, 17)])
def test_mixed_batches_either_side_of_their_kernels(stages, blocks, types, n):
    """How many plans blocks take depends on how deep they can be, the records' room and the model's blocks: same bits on
    both sides."""
    w = W.tiny(seed=57, n_types=types, n_zones=1 if types == 2 else 2, L=blocks, gbs=768, d_values=(1, 3, 16, 128),
               p_values=[p for p in (1, 2, 5, 8, 13, 24, 32) if p <= min(stages, blocks)], tp_values=(1, 2))
    w.avail[...] = 60_000
    w.capacity[:] = np.uint64(1 << 44)
    plans = W.random_mixed_plans(w, n, seed=n, p_max=min(stages, blocks))
    assert_equal(_run_on_device(w, B.pack_mixed_plans(plans, stages=stages)), Oracle(w).simulate_mixed_batch(plans), f"{stages} of {blocks}")
