// Per-stage GPU types by dynamic programming (Sailor Sec. 4.2.2: Eq. 1 and T_total).
//
// A problem is one configuration (P, mbs, tp, rc, D) with one zone order.  Its states are
// (stage i, type g of stage i, zone position zp of stage i, u = stages per type already placed in
// that zone, stage i included).  Zones before zp are never revisited and zones after it are
// untouched (first fit), so nothing else of the past matters.  A type that a zone could give to all
// P stages is not counted in u, and a type that fits no stage's memory is never placed.  The value of
// a state is the best plan of stages i.. from it: (sum of stage times, straggler, slowest
// synchronisation, slowest update).
//
// Only states that stage i can be in are visited.  First fit leaves a zone only when one of its types
// is used up, so position zp is reached after at least lo(zp) = sum of the smallest caps of the earlier
// positions and after at most mx(zp) = sum of all their caps stages: a stage i in position zp has
//     max(0 or 1, i + 1 - mx(zp))  <=  stages counted in u  <=  i + 1 - lo(zp)
// behind it (in the first zone of counted types only: exactly i + 1).  The count vectors of a position are
// numbered sum by sum (within a sum in lexicographic order), so the vectors of a stage are one contiguous range
// per position, and a move of one stage is a look-up: `nxt` holds, per vector and type, the vector with one more
// stage of that type.  Vectors, ranges and moves depend on (P, D * tp, zone order, types that fit) only -- a
// *layout*, shared by all problems alike in these and laid down once per call by dp_layout_kernel.
// A problem without a type for some stage's memory has no plan and no tables.
//
// Tables are filled from the last stage to the first: a thread owns one count vector for all types of stage i,
// tries every type for the next stage, and each value of the next stage is read by exactly one vector of the same
// position.  Small problems take one block through all their stages; the others advance together, a launch per
// distance from the last stage.  Per-configuration quantities (stage times per type, synchronisation per digit,
// message times per digit pair) are formed once per configuration by dp_tables_kernel.
#pragma once

#include "sailor_plan_kernels.cuh"

namespace sailor {

constexpr int DP_THREADS = 256;
constexpr uint8_t DP_NONE = 255;
constexpr uint32_t DP_SELF = 0x80000000u;        // in a row of `nxt`: the vector holds a stage of this type (or need not count it)
constexpr uint32_t DP_NO_VEC = 0x7fffffffu;      // no room for one more stage of this type in the position
constexpr uint32_t DP_NO_STATE = 0xffffffffu;
constexpr uint32_t DP_SMALL = 2048;              // most vectors a stage of a small problem has: eight rounds of one block

struct alignas(32) DpVal {           // best plan of stages i.. from a state; sum = +inf: there is none.  Aligned to its
                                     // size: a value then moves in one load or store
    double sum, mx, sy, up;
};

struct DpLayout {
    uint32_t P, nz;                  // positions that a pipeline of P stages can reach
    uint32_t nxt_off;                // first row of `nxt`
    uint32_t live_off;               // first word of its live rows
    uint32_t vec_base[SAILOR_Z_MAX + 1];           // first vector of each position
    uint32_t sum_max[SAILOR_Z_MAX];  // largest sum a position's vectors have
    uint32_t w_off[SAILOR_Z_MAX];    // its rank table: W[j][s], j = 0 .. n_counted, s = 0 .. P (vectors of the counted
                                     // types from the j-th on that add up to at most s)
    uint32_t first_vec[SAILOR_Z_MAX][SAILOR_T_MAX];     // the vector of "one stage, of this type"
    uint8_t zone[SAILOR_Z_MAX];      // zone of each position of the order
    uint8_t n_counted[SAILOR_Z_MAX];
    uint8_t counted[SAILOR_Z_MAX];   // bit g: type g is counted
    uint8_t cap[SAILOR_Z_MAX][SAILOR_T_MAX];            // stages a (position, type) can host, saturated at 255
    uint8_t first_later[SAILOR_Z_MAX][SAILOR_T_MAX];    // first position after zp that can host a stage of the type
};
static_assert(sizeof(DpLayout) % 4 == 0, "copied word by word");
// A live row (one per stage): count of live vectors, count before this stage (two words), then per position (first vector,
// slot of that vector); a vector's slot is its place among the live vectors of the stage.
__host__ __device__ inline uint32_t dp_live_words(uint32_t nz) { return 3 + 2 * nz; }
constexpr uint32_t DP_LIVE_WORDS_MAX = 3 + 2 * SAILOR_Z_MAX;
__host__ __device__ inline uint64_t live_before(const uint32_t* row) { return (uint64_t)row[2] << 32 | row[1]; }
__host__ __device__ inline uint32_t live_vec(const uint32_t* row, uint32_t zp) { return row[3 + 2 * zp]; }
__host__ __device__ inline uint32_t live_slot(const uint32_t* row, uint32_t zp) { return row[4 + 2 * zp]; }

struct DpJob {                       // a problem that has tables
    uint64_t val_off;                // first entry of its two level buffers
    uint64_t succ_off;               // first byte of its successors: [stage][slot][type]
    uint32_t config, index, layout, P;   // index = config * n_orders + order
    uint32_t slots, _pad;            // most live vectors of a stage: a type's values are this many entries, slot after slot (a
                                     // warp's gathers then fall into a few lines instead of one each: workload 3 1 853 -> 1 764
                                     // us a call, workload 5 432 -> 412)
};
static_assert(sizeof(DpJob) % 8 == 0, "copied by eight bytes");

struct DpResult {                    // per problem that has a plan, written by dp_finish_kernel
    double t_iter, cost;             // the simulator's figures for the plan (stage order)
    uint64_t peak_mem;
    uint32_t status, _pad;
    uint8_t type[SAILOR_P_MAX];
    uint8_t zone[SAILOR_P_MAX];
};

// Per-configuration tables in global memory, one block of `stride` doubles per configuration:
//   fb[p_max][T], upd[p_max][T], sync[p_max][R], c2x[R][R] (2 * message time, [next digit][this digit]),
//   then ok[p_max] (u32 bit g: stage fits type g and tp fits its node), n_b (u64), valid (u32).
struct DpTabLayout {
    uint32_t p_max, T, R;
    __host__ __device__ size_t off_fb() const { return 0; }
    __host__ __device__ size_t off_upd() const { return (size_t)p_max * T; }
    __host__ __device__ size_t off_sync() const { return 2 * (size_t)p_max * T; }
    __host__ __device__ size_t off_c2x() const { return 2 * (size_t)p_max * T + (size_t)p_max * R; }
    __host__ __device__ size_t off_ok() const { return off_c2x() + (size_t)R * R; }               // in doubles
    __host__ __device__ size_t off_nb() const { return off_ok() + (p_max + 1) / 2; }
    __host__ __device__ size_t stride() const { return off_nb() + 2; }
};

__global__ void __launch_bounds__(DP_THREADS)
dp_tables_kernel(const unsigned char* __restrict__ blob, SpaceDesc sp, uint32_t n_config, uint32_t n_orders, DpTabLayout lay,
                 const uint8_t* __restrict__ wanted /* [n_config], null: all */, double* __restrict__ tabs,
                 double* __restrict__ value /* [n_config * n_orders]: +inf, no plan so far */, DeviceSpan* span) {
    __shared__ uint64_t s_params[SAILOR_P_MAX];
    __shared__ uint32_t s_ok[SAILOR_P_MAX];
    TabView v;
    v.bind(blob, blob);
    const TabHdr* h = v.h;
    const uint32_t T = h->T, R = h->R, tid = threadIdx.x;
    if (blockIdx.x == 0 && tid == 0) span->start = device_ns();          // the call's first kernel
    for (uint32_t c = blockIdx.x; c < n_config; c += gridDim.x) {
        __syncthreads();
        for (uint32_t q = tid; q < n_orders; q += DP_THREADS) value[(size_t)c * n_orders + q] = make_inf();
        if (wanted && !wanted[c]) continue;
        const Config k = config_of(sp, c);
        double* tab = tabs + (size_t)c * lay.stride();
        const uint32_t tp = h->tp_values[k.tpi];
        const uint64_t dm = (uint64_t)k.D * h->mbs_values[k.mi];
        const bool valid = k.D >= 1 && h->gbs % dm == 0 && h->heads % tp == 0;
        const uint64_t n_b = valid ? h->gbs / dm : 0;
        if (tid == 0) {
            *reinterpret_cast<uint64_t*>(tab + lay.off_nb()) = n_b;
            *reinterpret_cast<uint32_t*>(tab + lay.off_nb() + 1) = valid ? 1u : 0u;
        }
        for (uint32_t i = tid; i < SAILOR_P_MAX; i += DP_THREADS) s_ok[i] = 0;
        __syncthreads();
        if (!valid) continue;
        const uint32_t P = k.P, base = h->n_blocks / P, extra = h->n_blocks % P;
        for (uint32_t x = tid; x < P * T; x += DP_THREADS) {
            const uint32_t i = x / T, g = x % T;
            const uint32_t nb = base + (i < extra ? 1u : 0u);
            const bool e = (i == 0) && h->has_embed, hd = (i == P - 1) && h->has_head;
            const StageTimes st = stage_times(v, g, k.tpi, k.mi, nb, e, hd);
            const double b = k.rc ? add_rn(st.b, st.f) : st.b;
            tab[lay.off_fb() + x] = add_rn(st.f, b);
            tab[lay.off_upd() + x] = st.u;
            const uint64_t inflight = (uint64_t)(P - i) < n_b ? (uint64_t)(P - i) : n_b;
            const StageMem sm = stage_memory(v, k.tpi, k.mi, k.rc, nb, e, hd, inflight);
            if (sm.mem + h->reserved[g] <= h->capacity[g] && tp <= h->gpn[g]) atomicOr(&s_ok[i], 1u << g);
            if (g == 0) s_params[i] = sm.params;
        }
        __syncthreads();
        const double steps = (double)(2 * (uint64_t)(k.D - 1)), coef = steps / (double)k.D;
        for (uint32_t x = tid; x < P * R; x += DP_THREADS) {
            const uint32_t i = x / R, d = x % R;
            tab[lay.off_sync() + x] = k.D > 1 ? allreduce_time(v, d % T, d, tp, k.D, s_params[i], steps, coef) : 0.0;
        }
        const double msg = (double)v.p2p[k.mi];
        for (uint32_t x = tid; x < R * R; x += DP_THREADS) {
            const uint32_t dn = x / R, d = x % R;          // [next][this]
            tab[lay.off_c2x() + x] = mul_rn(2.0, boundary_time(v, d % T, d / T, tp, dn % T, dn / T, tp, k.D, msg));
        }
        for (uint32_t i = tid; i < P; i += DP_THREADS) reinterpret_cast<uint32_t*>(tab + lay.off_ok())[i] = s_ok[i];
    }
}

// ---- layouts -------------------------------------------------------------------------------------------
//
// With W[j][s] as above, the vectors with exactly `s` stages of the types from j on whose first count is below x are
// W[j + 1][s] - W[j + 1][s - x] many, and the vectors of sum s start behind the W[0][s - 1] with a smaller sum.

struct DpLayoutParams {
    const DpLayout* layouts;
    const uint32_t* blk_prefix;      // [n_layouts + 1] blocks before each layout
    const uint32_t* wtab;
    uint32_t* nxt;                   // [vector][TM]
    uint32_t n_layouts, T;
};

template <uint32_t TM>
__global__ void __launch_bounds__(DP_THREADS) dp_layout_kernel(const __grid_constant__ DpLayoutParams lp) {
    __shared__ DpLayout L;
    const uint32_t tid = threadIdx.x, T = lp.T;
    uint32_t which = 0;
    {
        uint32_t hi = lp.n_layouts;
        while (hi - which > 1) {
            const uint32_t mid = (which + hi) >> 1;
            if (lp.blk_prefix[mid] <= blockIdx.x) which = mid; else hi = mid;
        }
    }
    for (uint32_t x = tid; x < sizeof(DpLayout) / 4; x += DP_THREADS)
        reinterpret_cast<uint32_t*>(&L)[x] = reinterpret_cast<const uint32_t*>(lp.layouts + which)[x];
    __syncthreads();
    const uint32_t v = (blockIdx.x - lp.blk_prefix[which]) * DP_THREADS + tid;
    if (v >= L.vec_base[L.nz]) return;
    uint32_t zp = 0;
    while (v >= L.vec_base[zp + 1]) ++zp;
    const uint32_t w = L.P + 1, base = L.vec_base[zp], e = v - base, most = L.sum_max[zp], counted = L.counted[zp];
    const uint32_t* W = lp.wtab + L.w_off[zp];
    uint32_t s = 0;                                          // the sum: the smallest with W[0][s] > e
    for (uint32_t hi = most; s < hi;) {
        const uint32_t mid = (s + hi) >> 1;
        if (W[mid] > e) hi = mid; else s = mid + 1;
    }
    uint32_t u[SAILOR_T_MAX], r = e - (s ? W[s - 1] : 0u), rem = s, j = 0;
#pragma unroll
    for (uint32_t t = 0; t < SAILOR_T_MAX; ++t) {
        u[t] = 0;
        if ((counted >> t) & 1u) {
            const uint32_t* row = W + (j + 1) * w;
            const uint32_t top = row[rem];
            uint32_t lo = 0, hi = min((uint32_t)L.cap[zp][t], rem);
            while (lo < hi) {                                // the largest count that leaves at most r vectors before it
                const uint32_t mid = (lo + hi + 1) >> 1;
                if (top - row[rem - mid] <= r) lo = mid; else hi = mid - 1;
            }
            r -= top - row[rem - lo];
            u[t] = lo;
            rem -= lo;
            ++j;
        }
    }
    uint32_t out[TM];
#pragma unroll
    for (uint32_t g = 0; g < TM; ++g) {
        out[g] = DP_NO_VEC;
        if (g >= T) continue;
        if ((counted >> g) & 1u) {
            if (u[g] < L.cap[zp][g] && s < most) {
                uint32_t at = W[s], left = s + 1, q = 0;
#pragma unroll
                for (uint32_t t = 0; t < SAILOR_T_MAX; ++t)
                    if ((counted >> t) & 1u) {
                        const uint32_t x = u[t] + (t == g ? 1u : 0u);
                        const uint32_t* row = W + (q + 1) * w;
                        at += row[left] - row[left - x];
                        left -= x;
                        ++q;
                    }
                out[g] = base + at;
            }
            if (u[g]) out[g] |= DP_SELF;
        } else if (L.cap[zp][g]) {
            out[g] = v | DP_SELF;                            // room for every stage: not counted
        }
    }
    uint4* dst = reinterpret_cast<uint4*>(lp.nxt + (size_t)(L.nxt_off + v) * TM);
#pragma unroll
    for (uint32_t q = 0; q < TM / 4; ++q) dst[q] = make_uint4(out[4 * q], out[4 * q + 1], out[4 * q + 2], out[4 * q + 3]);
}

// ---- the stages ----------------------------------------------------------------------------------------

struct DpLevelParams {
    const DpLayout* layouts;
    const DpJob* jobs;
    const uint32_t* live;
    const uint32_t* nxt;
    const double* tabs;
    DpVal* val[2];                   // level buffers [type][slot]; stage i lives in val[(P - 1 - i) & 1]
    uint8_t* succ;                   // [stage][slot][type]: type of the next stage in the best plan (DP_NONE: there is none)
    const uint32_t* blk_prefix;      // per-stage launches: [n_active + 1] blocks before each job of this launch
    DpTabLayout lay;
    uint32_t T, n_active;
    uint32_t dist;                   // stage i = P - 1 - dist
};

// A value in one 32-byte load or store.  Both are memory accesses to the compiler: a block reads values it wrote before its last
// barrier, and kernels launched early read after griddepcontrol.wait.
__device__ __forceinline__ DpVal load_val(const DpVal* p) {
    DpVal v;
    asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];" : "=d"(v.sum), "=d"(v.mx), "=d"(v.sy), "=d"(v.up) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void store_val(DpVal* p, const DpVal& v) {
    asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p), "d"(v.sum), "d"(v.mx), "d"(v.sy), "d"(v.up) : "memory");
}

// What a stage of a job reads of the job's tables, kept in shared memory (every vector of the stage reads it).
struct DpStageTab {
    double nb;
    uint32_t ok, ok_next;            // types that fit the stage, and the next
    double fb[SAILOR_T_MAX], upd[SAILOR_T_MAX], sync[R_MAX];
};
// Thread `x` of the block brings in its part of stage i's.
__device__ __forceinline__ void dp_stage_tab(const DpLevelParams& lp, const double* tab, uint32_t P, uint32_t i, uint32_t x, DpStageTab& st) {
    const uint32_t* okv = reinterpret_cast<const uint32_t*>(tab + lp.lay.off_ok());
    if (x < lp.lay.R) st.sync[x] = tab[lp.lay.off_sync() + (size_t)i * lp.lay.R + x];
    else if (x >= 64 && x < 64 + lp.T) st.fb[x - 64] = tab[lp.lay.off_fb() + i * lp.T + (x - 64)];
    else if (x >= 96 && x < 96 + lp.T) st.upd[x - 96] = tab[lp.lay.off_upd() + i * lp.T + (x - 96)];
    else if (x == 128) st.ok = okv[i];
    else if (x == 129) st.ok_next = i + 1 < P ? okv[i + 1] : 0u;
    else if (x == 130) st.nb = (double)*reinterpret_cast<const uint64_t*>(tab + lp.lay.off_nb());
}
static_assert(R_MAX <= 64 && SAILOR_T_MAX <= 32 && DP_THREADS > 130, "a thread per entry");

// Stage i of a job for the vector in `slot` of the stage, all its types at once (TM >= T types).  `here` and `then` are
// the live rows of stages i and i + 1, `st` the stage's tables (shared memory).
// AFTER_LEVEL: launched while the level it reads may still be running.
template <uint32_t TM, bool AFTER_LEVEL>
__device__ __forceinline__ void dp_vector(const DpLevelParams& lp, const DpLayout& L, const DpJob& job, const uint32_t* here,
                                          const uint32_t* then, const DpStageTab& st, uint32_t i, uint32_t slot) {
    const uint32_t T = lp.T, dist = job.P - 1 - i;
    const double* c2x = lp.tabs + (size_t)job.config * lp.lay.stride() + lp.lay.off_c2x();
    const double nb = st.nb;
    uint32_t zp = 0;
    while (zp + 1 < L.nz && live_slot(here, zp + 1) <= slot) ++zp;
    const uint32_t v = live_vec(here, zp) + (slot - live_slot(here, zp));
    uint32_t nx[TM];                                         // (nothing so far depends on another stage)
    {
        const uint4* row = reinterpret_cast<const uint4*>(lp.nxt + (size_t)(L.nxt_off + v) * TM);
#pragma unroll
        for (uint32_t q = 0; q < TM / 4; ++q) {
            const uint4 x = __ldg(row + q);
            nx[4 * q] = x.x; nx[4 * q + 1] = x.y; nx[4 * q + 2] = x.z; nx[4 * q + 3] = x.w;
        }
    }
    if (AFTER_LEVEL) asm volatile("griddepcontrol.wait;" ::: "memory");       // the level after this stage is complete
    // what follows a stage of each type g2: the state it leads to (the same for every type of stage i) and its value
    const DpVal* nxt = lp.val[(dist & 1) ^ 1] + job.val_off;
    DpVal n[TM];
    uint32_t d2[TM];
#pragma unroll
    for (uint32_t g2 = 0; g2 < TM; ++g2) {
        d2[g2] = 0;
        n[g2].sum = make_inf(); n[g2].mx = n[g2].sy = n[g2].up = 0.0;
    }
    if (dist != 0) {
        const uint32_t ok_next = st.ok_next;
#pragma unroll
        for (uint32_t g2 = 0; g2 < TM; ++g2) {
            if (g2 >= T || !((ok_next >> g2) & 1u)) continue;
            // first fit: this position while it has room for one more stage of the type, else the next that has
            uint32_t zp2 = zp, id = nx[g2] & DP_NO_VEC;
            if (id == DP_NO_VEC) {
                zp2 = L.first_later[zp][g2];
                if (zp2 == DP_NONE) continue;
                id = L.first_vec[zp2][g2];
            }
            const uint32_t slot2 = live_slot(then, zp2) + (id - live_vec(then, zp2));
            if (slot2 >= then[0]) continue;                  // (a move of a live state leads to a live state)
            d2[g2] = L.zone[zp2] * T + g2;
            n[g2] = load_val(nxt + (size_t)g2 * job.slots + slot2);
        }
    }
    const uint32_t ok_here = st.ok;
    DpVal* cur = lp.val[dist & 1] + job.val_off + slot;
    uint8_t* succ = lp.succ + job.succ_off + (live_before(here) + slot) * T;
    uint32_t picks[TM / 4];                                  // a byte per type, written together where T allows it
#pragma unroll
    for (uint32_t q = 0; q < TM / 4; ++q) picks[q] = 0xffffffffu;
#pragma unroll
    for (uint32_t g = 0; g < TM; ++g) {
        if (g >= T) break;
        // a state holds stage i itself: its type must fit the stage and, when counted, be counted at least once
        if (!((ok_here >> g) & 1u) || !(nx[g] & DP_SELF)) continue;
        const uint32_t d = L.zone[zp] * T + g;
        const double fb = st.fb[g], upd = st.upd[g], sync = st.sync[d];
        DpVal best;
        uint32_t pick = DP_NONE;
        if (dist == 0) {                                     // the last stage sends nothing
            best.sum = fb; best.mx = fb; best.sy = sync; best.up = upd;
        } else {
            best.sum = make_inf(); best.mx = best.sy = best.up = 0.0;
            double best_v = make_inf();
#pragma unroll
            for (uint32_t g2 = 0; g2 < TM; ++g2) {
                if (!(n[g2].sum < make_inf())) continue;     // (also where there is no such state)
                const double t = add_rn(fb, c2x[d2[g2] * lp.lay.R + d]);
                DpVal c;
                c.sum = add_rn(t, n[g2].sum);
                c.mx = dmax(t, n[g2].mx);
                c.sy = dmax(sync, n[g2].sy);
                c.up = dmax(upd, n[g2].up);
                const double val = add_rn(add_rn(add_rn(c.sum, mul_rn(nb, c.mx)), c.sy), c.up);
                if (pick == DP_NONE || val < best_v) { best = c; best_v = val; pick = g2; }
            }
        }
        store_val(cur + (size_t)g * job.slots, best);
        picks[g / 4] = (picks[g / 4] & ~(0xffu << (8 * (g % 4)))) | pick << (8 * (g % 4));
    }
    if (T == TM) {                                           // (every problem's successors start on a 64-byte line)
        if (TM == 4) *reinterpret_cast<uint32_t*>(succ) = picks[0];
        else *reinterpret_cast<uint2*>(succ) = make_uint2(picks[0], picks[TM / 4 - 1]);
    } else {
#pragma unroll
        for (uint32_t g = 0; g < TM; ++g)
            if (g < T) succ[g] = (uint8_t)(picks[g / 4] >> (8 * (g % 4)));
    }
}

// One stage (a distance from the last) of every job of the launch; a thread per live vector.
template <uint32_t TM>
__global__ void __launch_bounds__(DP_THREADS, TM <= 4 ? 3 : 2) dp_level_kernel(const __grid_constant__ DpLevelParams lp) {
    __shared__ DpLayout L;
    __shared__ DpJob job;
    __shared__ uint32_t rows[2][DP_LIVE_WORDS_MAX];
    __shared__ DpStageTab st;
    __shared__ uint32_t s_lo;
    const uint32_t tid = threadIdx.x;
    uint32_t which = 0;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");      // the next stage's blocks may find their way meanwhile
    // the job whose blocks include this one: a search with DP_THREADS probes per round, so that a block waits for one or
    // two loads, not for a chain of them
    {
        uint32_t lo = 0, n = lp.n_active;                    // invariant: prefix[lo] <= block < prefix[lo + n]
        while (n > 1) {
            const uint32_t step = (n + DP_THREADS - 1) / DP_THREADS;
            const uint32_t a = lo + tid * step, b = a + step < lo + n ? a + step : lo + n;
            if (a < lo + n && lp.blk_prefix[a] <= blockIdx.x && blockIdx.x < lp.blk_prefix[b]) s_lo = a;
            __syncthreads();
            const uint32_t got = s_lo;
            __syncthreads();
            n = got + step < lo + n ? step : lo + n - got;
            lo = got;
        }
        which = lo;
    }
    const uint32_t slot = (blockIdx.x - lp.blk_prefix[which]) * DP_THREADS + tid;
    const DpJob& gj = lp.jobs[which];
    const DpLayout* gl = lp.layouts + gj.layout;
    const uint32_t i = gj.P - 1 - lp.dist;
    if (tid < sizeof(DpJob) / 8) reinterpret_cast<uint64_t*>(&job)[tid] = reinterpret_cast<const uint64_t*>(&gj)[tid];
    for (uint32_t x = tid; x < sizeof(DpLayout) / 4; x += DP_THREADS)
        reinterpret_cast<uint32_t*>(&L)[x] = reinterpret_cast<const uint32_t*>(gl)[x];
    const uint32_t words = dp_live_words(gl->nz);
    if (tid < words) {
        const uint32_t* row = lp.live + gl->live_off + (size_t)i * words + tid;
        rows[0][tid] = row[0];
        rows[1][tid] = lp.dist ? row[words] : 0u;
    }
    dp_stage_tab(lp, lp.tabs + (size_t)gj.config * lp.lay.stride(), gj.P, i, tid, st);
    __syncthreads();
    if (slot < rows[0][0]) dp_vector<TM, true>(lp, L, job, rows[0], rows[1], st, i, slot);
}

// Small problems: a block takes one job through all its stages, from the last to the first, with a barrier between
// stages (a stage reads only what the same block wrote for the stage after it).
template <uint32_t TM>
__global__ void __launch_bounds__(DP_THREADS, TM <= 4 ? 3 : 2) dp_problem_kernel(const __grid_constant__ DpLevelParams lp) {
    __shared__ DpLayout L;
    __shared__ DpJob job;
    __shared__ uint32_t rows[3][DP_LIVE_WORDS_MAX];          // of this stage, the one after it and the one before it: one
    __shared__ DpStageTab st[2];                             // barrier a stage
    const uint32_t tid = threadIdx.x;
    const DpJob& gj = lp.jobs[blockIdx.x];
    const DpLayout* gl = lp.layouts + gj.layout;
    if (tid < sizeof(DpJob) / 8) reinterpret_cast<uint64_t*>(&job)[tid] = reinterpret_cast<const uint64_t*>(&gj)[tid];
    for (uint32_t x = tid; x < sizeof(DpLayout) / 4; x += DP_THREADS)
        reinterpret_cast<uint32_t*>(&L)[x] = reinterpret_cast<const uint32_t*>(gl)[x];
    __syncthreads();
    const uint32_t words = dp_live_words(L.nz);
    const double* tab = lp.tabs + (size_t)job.config * lp.lay.stride();
    for (uint32_t dist = 0; dist < job.P; ++dist) {
        const uint32_t i = job.P - 1 - dist;
        uint32_t* here = rows[dist % 3];
        if (tid < words) here[tid] = lp.live[L.live_off + (size_t)i * words + tid];
        dp_stage_tab(lp, tab, job.P, i, tid, st[dist & 1]);
        __syncthreads();                                     // the row, and the values of the stage after this one
        for (uint32_t slot = tid; slot < here[0]; slot += DP_THREADS)
            dp_vector<TM, false>(lp, L, job, here, rows[(dist + 2) % 3], st[dist & 1], i, slot);
    }
}

// A plan of one degree simulated by a warp, lane i taking stage i (then i + 32, ...): `gz` holds type | zone << 8 of every
// stage, `cnt` a counter per (zone, type) (both shared memory, the warp's own).  Per-stage terms are formed side by side; the
// sums whose order is part of the result run over the lanes' terms in stage order, so the bits are those of simulate_runs.
// Every lane returns the same.
__device__ __forceinline__ SimOut simulate_stages(const TabView& v, const uint16_t* __restrict__ avail, const Config& k,
                                                  const uint16_t* gz, uint32_t* cnt, uint32_t lane) {
    const TabHdr* h = v.h;
    const uint32_t T = h->T, Z = h->Z, P = k.P, D = k.D, mi = k.mi, tp = h->tp_values[k.tpi];
    SimOut o;
    o.t_iter = o.cost = make_nan();
    for (uint32_t d = lane; d < h->R; d += 32) cnt[d] = 0;
    __syncwarp();
    for (uint32_t i = lane; i < P; i += 32) atomicAdd(&cnt[(gz[i] >> 8) * T + (gz[i] & 0xffu)], 1u);       // stages
    __syncwarp();
    const uint64_t dm = (uint64_t)D * h->mbs_values[mi], n_b = h->gbs / dm;
    uint32_t status = (n_b * dm != h->gbs || h->heads % tp != 0) ? SAILOR_ST_INVALID : 0u;
    const uint32_t base = h->n_blocks / P, extra = h->n_blocks - base * P;
    const double msg = (double)v.p2p[mi], steps = (double)(2 * (uint64_t)(D - 1)), coef = steps / (double)D;
    const double xbytes = (double)(2 * n_b * (uint64_t)D * v.p2p[mi]);
    double sum_t = 0.0, max_t = 0.0, max_sync = 0.0, max_u = 0.0, rate = 0.0, c_comm = 0.0;
    uint64_t peak = 0;
    for (uint32_t at = 0; at < P; at += 32) {
        const uint32_t i = at + lane;
        double t = 0.0, gpu_rate = 0.0, comm = 0.0;
        bool crosses = false;
        if (i < P) {
            const uint32_t g = gz[i] & 0xffu, z = gz[i] >> 8, d = z * T + g;
            const bool e = (i == 0) && h->has_embed, hd = (i == P - 1) && h->has_head;
            const size_t comp = (size_t)((e ? 2u : 0u) + (hd ? 1u : 0u)) * h->chain_len + base + (i < extra ? 1u : 0u);
            const size_t ct = comp * h->n_tp + k.tpi;
            t = v.cmp_fb[(((comp * T + g) * h->n_tp + k.tpi) * h->n_mbs + mi) * 2 + k.rc];
            max_u = dmax(max_u, v.cmp_upd[(comp * T + g) * h->n_tp + k.tpi]);
            const uint64_t* mm = v.cmp_mem + ((ct * h->n_mbs + mi) * 2 + k.rc) * 2;
            const uint64_t inflight = (uint64_t)(P - i) < n_b ? (uint64_t)(P - i) : n_b;
            const uint64_t m = mm[0] + h->reserved[g] + inflight * mm[1];
            if (m > h->capacity[g]) status |= SAILOR_ST_OOM;
            if (tp > h->gpn[g]) status |= SAILOR_ST_INVALID;
            if ((uint64_t)cnt[d] * D * tp > avail[d]) status |= SAILOR_ST_OVER_AVAIL;
            peak = m > peak ? m : peak;
            if (D > 1) max_sync = dmax(max_sync, allreduce_bytes_time(v, d, (uint64_t)D * tp <= h->gpn[g], v.cmp_grad[ct], D, steps, coef));
            gpu_rate = mul_rn((double)(D * tp), v.price_s[d]);
            if (i + 1 < P) {
                const uint32_t gn = gz[i + 1] & 0xffu, zn = gz[i + 1] >> 8;
                t = add_rn(t, mul_rn(2.0, boundary_time(v, g, z, tp, gn, zn, tp, D, msg)));
                crosses = zn != z;
                if (crosses) comm = mul_rn(xbytes, v.egress[z * Z + zn]);
            }
            max_t = dmax(max_t, t);
        }
        const uint32_t n = P - at < 32 ? P - at : 32;
        for (uint32_t l = 0; l < n; ++l) {                   // in stage order
            sum_t = add_rn(sum_t, __shfl_sync(FULL, t, l));
            rate = add_rn(rate, __shfl_sync(FULL, gpu_rate, l));
        }
        for (uint32_t m = __ballot_sync(FULL, crosses); m; m &= m - 1) c_comm = add_rn(c_comm, __shfl_sync(FULL, comm, __ffs(m) - 1));
    }
#pragma unroll 1
    for (int x = 16; x; x >>= 1) {
        max_t = dmax(max_t, __shfl_xor_sync(FULL, max_t, x));
        max_sync = dmax(max_sync, __shfl_xor_sync(FULL, max_sync, x));
        max_u = dmax(max_u, __shfl_xor_sync(FULL, max_u, x));
        const uint64_t other = __shfl_xor_sync(FULL, peak, x);
        peak = other > peak ? other : peak;
    }
    o.peak_mem = peak;
    o.status = __reduce_or_sync(FULL, status);
    if (o.status & SAILOR_ST_INVALID) return o;
    o.t_iter = add_rn(add_rn(add_rn(sum_t, mul_rn((double)n_b, max_t)), max_sync), max_u);
    o.cost = add_rn(mul_rn(rate, o.t_iter), c_comm);
    return o;
}

// What a warp of the kernels that end a search keeps in shared memory.
struct DpFinishWarp {
    uint16_t gz[SAILOR_P_MAX];       // type | zone << 8 of every stage
    uint32_t cnt[R_MAX];
    uint8_t used[SAILOR_T_MAX];
};
constexpr int DP_FINISH_WARPS = 4, DP_FINISH_THREADS = 32 * DP_FINISH_WARPS;

// Stage 0 and the walk through the kept successors, a warp per job.  The walk is a chain of one round of loads per stage (the
// successor's type, and next to it the moves of the state's vector for every type it can be) and what the kernel's time is;
// the simulation is the lanes'.  520 jobs of up to 48 stages: 107 us by a thread each, 43 this way (34 where a successor is
// the next state's four-byte number, which costs the levels more than that: 1 525 us against 1 489, and memory).
struct DpFinishParams {
    const unsigned char* blob;
    const uint16_t* avail;
    SpaceDesc sp;
    const DpLayout* layouts;
    const DpJob* jobs;
    const uint32_t* live;
    const double* tabs;
    const DpVal* val[2];
    const uint8_t* succ;
    const uint32_t* nxt;             // [vector][TM]
    double* value;                   // indexed by problem index
    DpResult* results;               // indexed by problem index
    DpTabLayout lay;
    uint32_t n_jobs, T, TM;
};

__global__ void __launch_bounds__(DP_FINISH_THREADS) dp_finish_kernel(const __grid_constant__ DpFinishParams fp) {
    __shared__ DpFinishWarp warps[DP_FINISH_WARPS];
    __shared__ uint32_t s_rows[DP_FINISH_WARPS][33 * DP_LIVE_WORDS_MAX];    // live rows of 32 stages and the one after them
    const uint32_t lane = threadIdx.x & 31, x = blockIdx.x * DP_FINISH_WARPS + (threadIdx.x >> 5);
    if (x >= fp.n_jobs) return;
    DpFinishWarp& w = warps[threadIdx.x >> 5];
    uint32_t* rows = s_rows[threadIdx.x >> 5];
    const DpJob job = fp.jobs[x];
    const DpLayout& L = fp.layouts[job.layout];
    DpResult& out = fp.results[job.index];
    const uint32_t T = fp.T, P = job.P, words = dp_live_words(L.nz);
    const uint32_t* live = fp.live + L.live_off;
    const double* tab = fp.tabs + (size_t)job.config * fp.lay.stride();
    const uint32_t* okv = reinterpret_cast<const uint32_t*>(tab + fp.lay.off_ok());
    const double nb = (double)*reinterpret_cast<const uint64_t*>(tab + fp.lay.off_nb());
    const DpVal* lvl0 = fp.val[(P - 1) & 1] + job.val_off;
    double mine_v = make_inf();
    uint32_t mine = DP_NO_STATE, mine_p = 0;
    if (lane < T && ((okv[0] >> lane) & 1u)) {               // stage 0 by first fit from the first zone of the order, a lane per type
        const uint32_t p = L.cap[0][lane] >= 1 ? 0u : L.first_later[0][lane];
        if (p != DP_NONE) {
            const uint32_t slot = live_slot(live, p) + (L.first_vec[p][lane] - live_vec(live, p));
            if (slot < live[0]) {
                const DpVal v = lvl0[(size_t)lane * job.slots + slot];
                if (v.sum < make_inf()) {
                    mine_v = add_rn(add_rn(add_rn(v.sum, mul_rn(nb, v.mx)), v.sy), v.up);
                    mine = slot;
                    mine_p = p;
                }
            }
        }
    }
    double best_v = make_inf();
    uint32_t slot = DP_NO_STATE, g = 0;                      // the state of the stage that the walk is at: slot, type, position
    for (uint32_t g0 = 0; g0 < T; ++g0) {                    // the first of the best
        const double val = __shfl_sync(FULL, mine_v, g0);
        const uint32_t c = __shfl_sync(FULL, mine, g0);
        if (c != DP_NO_STATE && (slot == DP_NO_STATE || val < best_v)) { best_v = val; slot = c; g = g0; }
    }
    if (slot == DP_NO_STATE) return;                         // the value stays at "no plan"
    if (lane == 0) fp.value[job.index] = best_v;
    uint32_t zp = __shfl_sync(FULL, mine_p, g);
    const Config k = config_of(fp.sp, job.config);
    const uint8_t* succ = fp.succ + job.succ_off;
    const uint32_t* nxt = fp.nxt + (size_t)L.nxt_off * fp.TM;
    for (uint32_t at = 0; at < P; at += 32) {
        const uint32_t n = P - at < 32 ? P - at : 32;
        __syncwarp();
        for (uint32_t y = lane; y < (n + (at + n < P ? 1u : 0u)) * words; y += 32) rows[y] = live[(size_t)at * words + y];
        __syncwarp();
        for (uint32_t l = 0; l < n; ++l) {
            const uint32_t *here = rows + l * words, *then = here + words;
            if (lane == 0) w.gz[at + l] = (uint16_t)(g | L.zone[zp] << 8);
            if (at + l + 1 == P) break;
            const uint32_t v = live_vec(here, zp) + (slot - live_slot(here, zp));
            uint32_t got = 0;
            if (lane < fp.TM) got = nxt[(size_t)v * fp.TM + lane];
            else if (lane == 31) got = succ[(live_before(here) + slot) * T + g];
            g = __shfl_sync(FULL, got, 31);
            uint32_t id = __shfl_sync(FULL, got, g) & DP_NO_VEC;
            if (id == DP_NO_VEC) {                           // no room left in this position: the next that has
                zp = L.first_later[zp][g];
                id = L.first_vec[zp][g];
            }
            slot = live_slot(then, zp) + (id - live_vec(then, zp));
        }
    }
    __syncwarp();
    for (uint32_t i = lane; i < P; i += 32) {
        out.type[i] = (uint8_t)(w.gz[i] & 0xffu);
        out.zone[i] = (uint8_t)(w.gz[i] >> 8);
    }
    // the plan written out, through the simulator (Sec. 4.3): what a caller compares with a constraint
    TabView v;
    v.bind(fp.blob, fp.blob);
    const SimOut so = simulate_stages(v, fp.avail, k, w.gz, w.cnt, lane);
    if (lane == 0) {
        out.t_iter = so.t_iter;
        out.cost = so.cost;
        out.peak_mem = so.peak_mem;
        out.status = so.status;
    }
}

// The k best problems by (value, problem index), then the simulator's figures for their plans.
struct DpOut {                       // what a search leaves for the host, in mapped pinned memory
    unsigned long long counters[5];  // [0] problems with a plan, [1] number written to results, [2] plans over the constraint,
                                     // [3], [4] of the budget loop: problems given up, calls
    DeviceSpan span;
    sailor_dp_result results[SAILOR_K_MAX];
};

struct DpSelectParams {
    const double* value;             // [n_problems]
    const DpResult* results;
    const unsigned long long* counters;   // null, or the budget loop's [3] and [4]
    DpOut* out;
    SpaceDesc sp;
    uint32_t n_problems, n_orders, k;
    double budget, min_rate;         // <= 0: none
};

constexpr int DP_SELECT_THREADS = 512;

__global__ void __launch_bounds__(DP_SELECT_THREADS) dp_select_kernel(const __grid_constant__ DpSelectParams sp) {
    __shared__ Hit s_hits[DP_SELECT_THREADS / 32][SAILOR_K_MAX];
    __shared__ uint32_t s_n;
    __shared__ unsigned long long s_solved, s_over;
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = DP_SELECT_THREADS / 32;
    if (tid == 0) { s_solved = 0; s_over = 0; }
    __syncthreads();
    WarpTopK top;
    top.init();
    uint32_t solved = 0, over = 0;
    for (uint32_t base = warp * 32; base < sp.n_problems; base += nw * 32) {
        const uint32_t j = base + lane;
        const double v = j < sp.n_problems ? sp.value[j] : make_inf();
        bool have = v < make_inf();
        solved += have;
        if (have && (sp.budget > 0.0 || sp.min_rate > 0.0)) {  // the planner keeps a plan only within the constraint
            const DpResult& r = sp.results[j];
            const bool out_of = (sp.budget > 0.0 && r.cost > sp.budget) || (sp.min_rate > 0.0 && 1.0 / r.t_iter < sp.min_rate);
            over += out_of;
            have = !out_of;
        }
        const bool want = have && v <= top.thr_score;
        if (__any_sync(FULL, want)) top.offer(want, v, j, sp.k, lane);
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        solved += __shfl_xor_sync(FULL, solved, o);
        over += __shfl_xor_sync(FULL, over, o);
    }
    if (lane == 0 && solved) atomicAdd(&s_solved, (unsigned long long)solved);
    if (lane == 0 && over) atomicAdd(&s_over, (unsigned long long)over);
    s_hits[warp][lane].score = top.score;
    s_hits[warp][lane].flat = top.flat;
    __syncthreads();
    for (uint32_t step = 1; step < nw; step <<= 1) {
        if ((warp & (2 * step - 1)) == 0 && warp + step < nw) {
            top.merge_sorted(s_hits[warp + step][lane].score, s_hits[warp + step][lane].flat, sp.k, lane);
            s_hits[warp][lane].score = top.score;
            s_hits[warp][lane].flat = top.flat;
        }
        __syncthreads();
    }
    if (warp == 0) {
        const uint32_t n = __popc(__ballot_sync(FULL, lane < sp.k && top.flat != ~0ull));
        if (lane == 0) {
            s_n = n;
            sp.out->counters[0] = s_solved;
            sp.out->counters[1] = n;
            sp.out->counters[2] = s_over;
            sp.out->counters[3] = sp.counters ? sp.counters[3] : 0;
            sp.out->counters[4] = sp.counters ? sp.counters[4] : 0;
        }
    }
    __syncthreads();
    for (uint32_t j = warp; j < s_n; j += nw) {
        const uint32_t idx = (uint32_t)s_hits[0][j].flat;
        const DpResult& r = sp.results[idx];
        const uint32_t c = idx / sp.n_orders;
        const Config k = config_of(sp.sp, c);
        sailor_dp_result& o = sp.out->results[j];
        if (lane == 0) {
            o.config = c;
            o.order = idx % sp.n_orders;
            o.value = s_hits[0][j].score;
            o.t_iter = r.t_iter;
            o.cost = r.cost;
            o.peak_mem = r.peak_mem;
            o.status = r.status;
            o.P = (uint8_t)k.P; o.mbs_idx = (uint8_t)k.mi; o.tp_idx = (uint8_t)k.tpi; o.rc = (uint8_t)k.rc; o.D = (uint16_t)k.D;
            o._pad = 0;
        }
        for (uint32_t i = lane; i < SAILOR_P_MAX; i += 32) {
            o.type[i] = i < k.P ? r.type[i] : 0;
            o.zone[i] = i < k.P ? r.zone[i] : 0;
        }
    }
    if (tid == 0) sp.out->span.end = device_ns();
}

}  // namespace sailor
