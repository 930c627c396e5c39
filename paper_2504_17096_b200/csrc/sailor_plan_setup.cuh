// Kernels around a plan search: the end of a long pass, the tables of a space (built once), the waves of a search in
// degree order.
#pragma once

#include "sailor_plan_kernels.cuh"

namespace sailor {

extern template PlanKernel plan_kernel_of<SAILOR_OBJ_MAX_THROUGHPUT>(bool, bool, bool, bool);
extern template PlanKernel plan_kernel_of<SAILOR_OBJ_MIN_COST>(bool, bool, bool, bool);
extern template PlanKernel plan_kernel_of<SAILOR_OBJ_MAX_THROUGHPUT_PER_USD>(bool, bool, bool, bool);

// The end of a pass as a launch of its own (one block), after a search kernel that is not FUSED.
__global__ void __launch_bounds__(PLAN_THREADS) finish_kernel(const __grid_constant__ PlanParams pp, uint32_t n_partial) {
    extern __shared__ __align__(16) unsigned char dyn[];      // the static tables, then SAILOR_K_MAX words
    __shared__ Hit s_hits[PLAN_WARPS][SAILOR_K_MAX];
    __shared__ uint64_t mbar;
    __shared__ uint32_t s_n;
    const uint32_t tid = threadIdx.x;
    const uint32_t static_bytes = reinterpret_cast<const TabHdr*>(pp.blob)->static_bytes;
    if (!bulk_load(dyn, pp.blob, static_bytes, &mbar)) {
        if (tid == 0) atomicExch(&pp.ctrl->error, 1u);
        for (uint32_t x = tid; x < static_bytes / 16; x += PLAN_THREADS)
            reinterpret_cast<uint4*>(dyn)[x] = reinterpret_cast<const uint4*>(pp.blob)[x];
        __syncthreads();
    }
    TabView v;
    v.bind(dyn, pp.blob);
    finish_pass(pp, v, s_hits, reinterpret_cast<uint32_t*>(dyn + static_bytes), &s_n, n_partial);
}

// The tables of every configuration, built once per (context, space) and kept in global memory: all of them but
// the availability mask of the last segment depend on the context and the configuration only, so a search after
// a new snapshot copies them instead of rebuilding them.  One block per configuration at a time.
__global__ void __launch_bounds__(PLAN_THREADS, PLAN_MIN_BLOCKS) cfg_cache_kernel(const __grid_constant__ PlanParams pp, uint4* cache) {
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ CfgShared cs;
    const uint32_t tid = threadIdx.x;
    const TabHdr* gh = reinterpret_cast<const TabHdr*>(pp.blob);
    const uint32_t static_bytes = gh->static_bytes;
    if (!bulk_load(dyn, pp.blob, static_bytes, &cs.mbar)) {
        if (tid == 0) atomicExch(&pp.ctrl->error, 1u);
        for (uint32_t x = tid; x < static_bytes / 16; x += PLAN_THREADS)
            reinterpret_cast<uint4*>(dyn)[x] = reinterpret_cast<const uint4*>(pp.blob)[x];
        __syncthreads();
    }
    TabView v;
    v.bind(dyn, pp.blob);
    const uint32_t T = v.h->T, Z = v.h->Z;
    CfgArrays a;
    carve(dyn, static_bytes, pp.p_max, T, Z, a);
    // the whole cached region starts from zero, so that records do not depend on what the block did before
    for (uint32_t x = tid; x < pp.cache_arr16; x += PLAN_THREADS) reinterpret_cast<uint4*>(a.rec)[x] = make_uint4(0, 0, 0, 0);
    for (uint32_t x = tid; x < pp.cache_head16; x += PLAN_THREADS) reinterpret_cast<uint4*>(&cs)[x] = make_uint4(0, 0, 0, 0);
    __syncthreads();
    for (uint32_t c = blockIdx.x; c < pp.n_config; c += gridDim.x) {
        __syncthreads();
        build_config<true>(pp, v, cs, a, c);
        __syncthreads();
        uint4* dst = cache + (size_t)c * (pp.cache_head16 + pp.cache_arr16);
        for (uint32_t x = tid; x < pp.cache_head16; x += PLAN_THREADS) dst[x] = reinterpret_cast<const uint4*>(&cs)[x];
        for (uint32_t x = tid; x < pp.cache_arr16; x += PLAN_THREADS) dst[pp.cache_head16 + x] = reinterpret_cast<const uint4*>(a.rec)[x];
    }
}

// Which prefixes can matter at all?  Per configuration: the digits of every segment whose type can
// host tp and whose stages fit in memory (H2: independent of availability), hence the number of
// chunks of prefixes made of such digits only, and -- in closed form -- how many candidates are
// invalid or out of memory.  Runs once per (context, space); the plan search then enumerates only
// the live prefixes.  One block per configuration at a time.  The same pass lays down where every
// configuration's candidates and chunks start when nothing is pruned.
constexpr int SURVEY_THREADS = 128;

__global__ void __launch_bounds__(SURVEY_THREADS)
survey_kernel(const unsigned char* __restrict__ blob, SpaceDesc sp, uint32_t n_config, uint32_t* __restrict__ live_chunks,
              uint32_t* __restrict__ chunk_start /* [n_config + 1] */, uint64_t* __restrict__ flat_base /* [n_config] */,
              unsigned long long* __restrict__ closed /* total, invalid, oom */,
              unsigned long long* __restrict__ cfg_closed /* [n_config][3], the same per configuration; may be null */) {
    __shared__ uint32_t oom_stage[SAILOR_P_MAX];
    __shared__ Config k;
    __shared__ uint32_t valid;
    __shared__ uint64_t n_b;
    TabView v;
    v.bind(blob, blob);
    const TabHdr* h = v.h;
    const uint32_t T = h->T, R = h->R, tid = threadIdx.x;
    for (uint32_t c = blockIdx.x; c < n_config; c += gridDim.x) {
        __syncthreads();
        if (tid == 0) {
            k = config_of(sp, c);
            const uint32_t tp = h->tp_values[k.tpi];
            const uint64_t dm = (uint64_t)k.D * h->mbs_values[k.mi];
            valid = (k.D >= 1 && h->gbs % dm == 0 && h->heads % tp == 0) ? 1u : 0u;
            n_b = k.D >= 1 ? h->gbs / dm : 0;
        }
        for (uint32_t i = tid; i < SAILOR_P_MAX; i += SURVEY_THREADS) oom_stage[i] = 0;
        __syncthreads();
        const uint32_t P = k.P;
        if (valid) {
            const uint32_t base = h->n_blocks / P, extra = h->n_blocks % P;
            for (uint32_t x = tid; x < P * T; x += SURVEY_THREADS) {
                const uint32_t i = x / T, g = x % T;
                const uint32_t nb = base + (i < extra ? 1u : 0u);
                const bool e = (i == 0) && h->has_embed, hd = (i == P - 1) && h->has_head;
                const uint64_t inflight = (uint64_t)(P - i) < n_b ? (uint64_t)(P - i) : n_b;
                const StageMem sm = stage_memory(v, k.tpi, k.mi, k.rc, nb, e, hd, inflight);
                if (sm.mem + h->reserved[g] > h->capacity[g]) atomicOr(&oom_stage[i], 1u << g);
            }
        }
        __syncthreads();
        if (tid == 0) {
            const uint64_t n_all = ipow64(R, k.nseg);
            uint32_t chunks = 0;
            unsigned long long mine[3] = {n_all, n_all, 0};     // total, invalid, oom of this configuration
            if (valid) {
                const uint32_t tp = h->tp_values[k.tpi];
                uint32_t type_ok = 0;                      // types whose nodes can host tp
                for (uint32_t g = 0; g < T; ++g)
                    if (tp <= h->gpn[g]) type_ok |= 1u << g;
                const uint64_t n_valid = ipow64((uint64_t)__popc(type_ok) * h->Z, k.nseg);
                uint64_t live = 1, fit = 1;
                for (uint32_t s = 0; s < k.nseg; ++s) {
                    const uint32_t sa = (s * P + k.nseg - 1) / k.nseg, se = ((s + 1) * P + k.nseg - 1) / k.nseg;
                    uint32_t oom = 0;
                    for (uint32_t i = sa; i < se; ++i) oom |= oom_stage[i];
                    const uint64_t g_cnt = (uint64_t)__popc(type_ok & ~oom) * h->Z;     // usable digits of the segment
                    fit *= g_cnt;
                    if (s + 1 < k.nseg) live *= g_cnt;
                }
                if (fit) chunks = (uint32_t)((live + PLAN_THREADS - 1) / PLAN_THREADS);
                mine[1] = n_all - n_valid;
                mine[2] = n_valid - fit;
            }
            for (int j = 0; j < 3; ++j) {
                if (mine[j]) atomicAdd(&closed[j], mine[j]);
                if (cfg_closed) cfg_closed[3 * (size_t)c + j] = mine[j];
            }
            live_chunks[c] = chunks;
            // candidates and chunks of the configurations before this one: whole sub-spaces, then equal ones
            const uint32_t per_p = sp.n_mbs * sp.n_tp * sp.n_rc * sp.n_d;
            uint64_t flat = 0;
            uint32_t chunk = 0;
            for (uint32_t j = 0; j <= c / per_p; ++j) {
                const uint32_t before = j < c / per_p ? per_p : c - j * per_p;
                const uint64_t items = ipow64(R, nseg_of(sp.p_values[j], sp.seg_max) - 1);
                const uint32_t per_cfg = (uint32_t)((items + PLAN_THREADS - 1) / PLAN_THREADS);
                flat += before * items * R;
                chunk += before * per_cfg;
                if (c + 1 == n_config && j == c / per_p) chunk_start[n_config] = chunk + per_cfg;
            }
            flat_base[c] = flat;
            chunk_start[c] = chunk;
        }
    }
}

// Live chunks per configuration -> where each configuration's live chunks start, in place (exclusive scan, one
// block); the total and the closed-form counts go to the host.
struct SurveyOut {
    uint32_t live_chunks, _pad;
    unsigned long long closed[3];
};
constexpr int SCAN_THREADS = 1024;

__global__ void __launch_bounds__(SCAN_THREADS)
live_scan_kernel(uint32_t* __restrict__ live, uint32_t n_config, const unsigned long long* __restrict__ closed, SurveyOut* out) {
    __shared__ uint32_t warp_sum[SCAN_THREADS / 32];
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t per = (n_config + SCAN_THREADS - 1) / SCAN_THREADS;
    const uint32_t c0 = min(tid * per, n_config), c1 = min(c0 + per, n_config);
    uint32_t mine = 0;
    for (uint32_t c = c0; c < c1; ++c) mine += live[c];
    uint32_t incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t up = __shfl_up_sync(FULL, incl, o);
        if (lane >= (uint32_t)o) incl += up;
    }
    if (lane == 31) warp_sum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const uint32_t w = warp_sum[lane];
        uint32_t wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t up = __shfl_up_sync(FULL, wi, o);
            if (lane >= (uint32_t)o) wi += up;
        }
        warp_sum[lane] = wi - w;
        if (lane == 31) { live[n_config] = wi; out->live_chunks = wi; }
        if (lane < 3) out->closed[lane] = closed[lane];
    }
    __syncthreads();
    uint32_t at = warp_sum[warp] + incl - mine;
    for (uint32_t c = c0; c < c1; ++c) {
        const uint32_t here = live[c];
        live[c] = at;
        at += here;
    }
}

// ---- searches in degree order (H3 / H4) -----------------------------------------------------------
//
// A group is a configuration without its data-parallel degree; its degrees sit next to each other in
// the configuration index (c = group * n_d + position in d_values).  The rule of a group is
// sequential (try the next degree only while the last one improved), but the groups are independent,
// so they advance together: wave w evaluates, for every group still going, the w-th degree of the
// order.  Between two waves one small block applies the rule to what the last wave found and lays
// out the chunk table of the next one; nothing returns to the host in between.
struct GroupState {
    unsigned long long prev_bits;      // best score at the last degree that had a feasible plan
    uint32_t state;                    // 0: no feasible degree yet, 1: going, 2: stopped
    uint32_t _pad;
};

struct WaveParams {
    const uint32_t* live_start;        // [n_config + 1] chunk offsets when every configuration is searched
    const unsigned long long* cfg_closed;   // [n_config][3] total, invalid, oom per configuration
    uint32_t* wave_start;              // [n_config + 1] out: chunk offsets of this wave
    unsigned long long* cfg_best;      // [n_config]
    GroupState* groups;                // [n_config / n_d]
    Ctrl* ctrl;
    PlanOut* out;
    uint32_t n_config, n_d, wave;
    uint32_t first;                    // this launch is the call's first: it stamps the start
    uint8_t order[SAILOR_ND_MAX];      // positions in d_values, in the order they are tried
};

constexpr int WAVE_THREADS = 1024;

__global__ void __launch_bounds__(WAVE_THREADS) wave_step_kernel(const __grid_constant__ WaveParams wp) {
    __shared__ uint32_t warp_sum[WAVE_THREADS / 32];
    __shared__ unsigned long long s_closed[3];
    __shared__ uint32_t s_eval;
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t n_groups = wp.n_config / wp.n_d;
    const unsigned long long inf_bits = (unsigned long long)__double_as_longlong(make_inf());
    if (tid < 3) s_closed[tid] = 0;
    if (tid == 0) s_eval = 0;
    if (wp.first && tid == 0) wp.out->span.start = device_ns();
    // the rule, applied to what the previous wave found
    for (uint32_t g = tid; g < n_groups; g += WAVE_THREADS) {
        GroupState gs = wp.groups[g];
        if (wp.wave == 0) { gs.prev_bits = inf_bits; gs.state = 0; gs._pad = 0; }
        else if (gs.state != 2) {
            const unsigned long long best = wp.cfg_best[(size_t)g * wp.n_d + wp.order[wp.wave - 1]];
            if (best == inf_bits) { if (gs.state == 1) gs.state = 2; }         // nothing feasible at that degree
            else if (gs.state == 1 && !(best < gs.prev_bits)) gs.state = 2;     // no strict improvement
            else { gs.prev_bits = best; gs.state = 1; }
        }
        wp.groups[g] = gs;
    }
    __syncthreads();
    // chunk table of this wave: the configuration (group, order[wave]) of every group still going
    const uint32_t per = (wp.n_config + WAVE_THREADS - 1) / WAVE_THREADS;
    const uint32_t c0 = min(tid * per, wp.n_config), c1 = min(c0 + per, wp.n_config);
    const uint32_t pick = wp.order[wp.wave];
    uint32_t mine = 0, n_eval = 0;
    unsigned long long closed[3] = {0, 0, 0};
    for (uint32_t c = c0; c < c1; ++c) {
        if (c % wp.n_d != pick || wp.groups[c / wp.n_d].state == 2) continue;
        mine += wp.live_start[c + 1] - wp.live_start[c];
        wp.cfg_best[c] = inf_bits;
        ++n_eval;
        for (int j = 0; j < 3; ++j) closed[j] += wp.cfg_closed[3 * (size_t)c + j];
    }
    uint32_t incl = mine;                                   // exclusive scan of `mine` over the block
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t up = __shfl_up_sync(FULL, incl, o);
        if (lane >= (uint32_t)o) incl += up;
    }
    if (lane == 31) warp_sum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = warp_sum[lane], wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t up = __shfl_up_sync(FULL, wi, o);
            if (lane >= (uint32_t)o) wi += up;
        }
        warp_sum[lane] = wi - w;
        if (lane == 31) {
            wp.wave_start[wp.n_config] = wi;
            wp.ctrl->wave_chunks = wi;
            wp.ctrl->work_counter = 0;
        }
    }
    __syncthreads();
    uint32_t at = warp_sum[warp] + incl - mine;
    for (uint32_t c = c0; c < c1; ++c) {
        wp.wave_start[c] = at;
        if (c % wp.n_d == pick && wp.groups[c / wp.n_d].state != 2) at += wp.live_start[c + 1] - wp.live_start[c];
    }
    for (int j = 0; j < 3; ++j)
        if (closed[j]) atomicAdd(&s_closed[j], closed[j]);
    if (n_eval) atomicAdd(&s_eval, n_eval);
    __syncthreads();
    if (tid < 3 && s_closed[tid]) atomicAdd(&wp.ctrl->stats[tid], s_closed[tid]);
    if (tid == 0) wp.ctrl->n_cfg_evaluated += s_eval;
}

}  // namespace sailor
