// Search over plans whose stages mix GPU types among their replicas (Sailor Sec. 4.2.2, "Implementation": per
// stage, the resource combinations of different GPU types that give the stage its D replicas).
//
// A combination is a tuple of units per GPU type (see sailor.h); the host lists the combinations of every degree
// of the space once per space (descending lexicographic order) and the device looks them up.  A candidate is
// (P, mbs, rc, D) and one (zone, combination) per segment.
//
// Whether a candidate is invalid, out of memory or over the availability follows from integers alone, and nearly all
// candidates of a space fall to one of them.  So a space is searched in two steps: mixed_class_kernel (a thread per
// candidate) counts those classes and appends the candidates that are left to a queue; plan_mixed_kernel (a thread per
// queued candidate) evaluates them and keeps top-k lists.  Blocks leave their lists for
// mixed_finish_kernel, which merges them and writes the winners out with their records.
#pragma once

#include "sailor_mixed.cuh"

namespace sailor {

constexpr uint32_t MIX_UNITS_MAX = 16;
static_assert(SAILOR_MIX_P_MAX % 32 == 0, "every lane writes SAILOR_MIX_P_MAX / 32 stages of the record");

struct MixedSpaceDesc {
    uint32_t n_p, n_mbs, n_rc, n_d, seg_max, granularity;
    uint8_t p_values[SAILOR_NP_MAX];
    uint8_t mbs_idx[SAILOR_MBS_MAX];
    uint8_t rc_values[2];
    uint8_t tp_idx_of_type[SAILOR_T_MAX];
    uint16_t d_values[SAILOR_ND_MAX];
    uint32_t n_comb[SAILOR_ND_MAX];          // combinations of each degree of d_values
    uint32_t comb_off[SAILOR_ND_MAX];        // where they start in the table
};

__host__ __device__ inline uint32_t mixed_units(uint32_t granularity, uint32_t D) {
    return (granularity >= 1 && D % granularity == 0) ? granularity : D;
}

// Configuration c = ((p * n_mbs + mbs) * n_rc + rc) * n_d + d (positions in the space's lists).
struct MixedConfig { uint32_t P, mi, rc, D, di, nseg, per_unit; };   // per_unit: replicas in one unit of a combination

__host__ __device__ inline MixedConfig mixed_config_of(const MixedSpaceDesc& s, uint32_t c) {
    MixedConfig k;
    uint32_t x = c;
    k.di = x % s.n_d; x /= s.n_d;
    const uint32_t ri = x % s.n_rc; x /= s.n_rc;
    const uint32_t mi = x % s.n_mbs; x /= s.n_mbs;
    k.P = s.p_values[x];
    k.mi = s.mbs_idx[mi];
    k.rc = s.rc_values[ri];
    k.D = s.d_values[k.di];
    k.nseg = k.P < s.seg_max ? k.P : s.seg_max;
    k.per_unit = k.D / mixed_units(s.granularity, k.D);
    return k;
}

// Stage i of the candidate whose segment digits are `digit` (zone * n_comb + combination): its record.
// `combs` holds one 64-bit word per combination, byte g = units on type g.
__host__ __device__ inline void mixed_build_stage(const MixedSpaceDesc& s, const MixedConfig& k, uint32_t T,
                                                  const uint64_t* combs, const uint32_t* digit, uint32_t i,
                                                  sailor_mixed_stage* out) {
    const uint32_t n_comb = s.n_comb[k.di];
    const uint32_t dg = digit[i * k.nseg / k.P], zone = dg / n_comb;       // a digit is below Z * n_comb < 2^32
    const uint64_t word = combs[s.comb_off[k.di] + (dg - zone * n_comb)];
    // the stage as five 32-bit words (little-endian fields): zone | n_groups << 8, then type | tp_idx << 8 | count << 16
    // per group; the non-empty types in ascending order take the groups
    uint32_t gw[SAILOR_MIX_GROUPS_MAX] = {0, 0, 0, 0}, n_groups = 0;
    for (uint32_t g = 0; g < T; ++g) {
        const uint32_t units = (uint32_t)(word >> (8 * g)) & 0xffu;
        if (!units || n_groups >= SAILOR_MIX_GROUPS_MAX) continue;
        const uint32_t grp = g | (uint32_t)s.tp_idx_of_type[g] << 8 | (units * k.per_unit & 0xffffu) << 16;
        gw[0] = n_groups == 0 ? grp : gw[0];
        gw[1] = n_groups == 1 ? grp : gw[1];
        gw[2] = n_groups == 2 ? grp : gw[2];
        gw[3] = n_groups == 3 ? grp : gw[3];
        n_groups++;
    }
    static_assert(sizeof(sailor_mixed_stage) == 20 && SAILOR_MIX_GROUPS_MAX == 4, "five words a stage");
    uint32_t* w = reinterpret_cast<uint32_t*>(out);
    w[0] = (zone & 0xffu) | n_groups << 8;
    w[1] = gw[0]; w[2] = gw[1]; w[3] = gw[2]; w[4] = gw[3];
}

// Candidates whose class the integers leave open are queued as offsets from the start of their range of the space; a
// range holds at most this many candidates, so the queue (4 bytes each) can never run over.
constexpr uint64_t MIXED_RANGE = 1ull << 23;

// Where the counters stand: the six classes (total, invalid, oom, over_avail, over_constraint, feasible), then these.
enum { MIXC_MIN_COST = 6, MIXC_ERROR = 7, MIXC_FOUND = 8, MIXC_QUEUED = 9, MIXC_N = 10 };

// What a search leaves for the host, written by mixed_finish_kernel into mapped pinned memory.
struct MixedOut {
    unsigned long long counters[MIXC_N];
    DeviceSpan span;
    sailor_mixed_result results[SAILOR_K_MAX];
};

struct MixedSearchParams {
    const unsigned char* blob;
    uint16_t avail[R_MAX];               // the availability snapshot rides in the launch parameters
    const uint64_t* cfg_flat_base;       // [n_config + 1]
    const uint64_t* combs;
    Hit* partial;                        // [grid][SAILOR_K_MAX]
    unsigned long long* counters;        // [MIXC_N]; min cost as bits
    uint32_t* queue;                     // [range_hi - range_lo]
    MixedOut* out;                       // mapped pinned host memory
    MixedSpaceDesc sp;
    uint32_t n_config, k, obj, n_partial;
    uint32_t carry_lists;                // a block goes on from the list it left for the previous range
    uint64_t range_lo, range_hi, n_total;
    double budget, min_rate;             // <= 0: none
};

constexpr int MIXS_THREADS = 256;
constexpr int MIXS_WARPS = MIXS_THREADS / 32;

// The record of candidate `flat` into `plan` (shared memory, one per warp, room for `stages` stages), by all lanes of the
// warp; the stages past the last are all zero, as the host decoder leaves them.
__device__ __forceinline__ void mixed_candidate(const MixedSearchParams& mp, uint32_t T, uint32_t Z, uint64_t flat,
                                                sailor_mixed_plan* plan, uint32_t stages, uint32_t lane) {
    uint32_t lo = 0, hi = mp.n_config;                       // the configuration whose block holds the index
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (mp.cfg_flat_base[mid] <= flat) lo = mid; else hi = mid;
    }
    const MixedConfig k = mixed_config_of(mp.sp, lo);
    const uint64_t radix = (uint64_t)Z * mp.sp.n_comb[k.di];
    uint64_t rem = flat - mp.cfg_flat_base[lo];
    uint32_t digit[SAILOR_SEG_MAX] = {0, 0, 0, 0};
    for (uint32_t s = k.nseg; s-- > 0;) { digit[s] = (uint32_t)(rem % radix); rem /= radix; }
    if (lane == 0) {
        plan->P = (uint8_t)k.P; plan->mbs_idx = (uint8_t)k.mi; plan->rc = (uint8_t)k.rc; plan->_pad = 0;
        plan->D = (uint16_t)k.D; plan->_pad2 = 0;
    }
    for (uint32_t i = lane; i < stages; i += 32) {
        if (i < k.P) mixed_build_stage(mp.sp, k, T, mp.combs, digit, i, &plan->stage[i]);
        else {
            uint32_t* z = reinterpret_cast<uint32_t*>(&plan->stage[i]);
            for (uint32_t x = 0; x < sizeof(sailor_mixed_stage) / 4; ++x) z[x] = 0;
        }
    }
    __syncwarp();
}

// x / d for 32-bit x by one 64-bit multiplication (magic = ceil(2^64 / d), 0 for d = 1).
struct MixedDivisor {
    uint64_t magic;
    uint32_t d;
    __device__ __forceinline__ void set(uint32_t div) { d = div; magic = div > 1 ? ~0ull / div + 1 : 0; }
    __device__ __forceinline__ uint32_t quotient(uint32_t x) const { return d > 1 ? (uint32_t)__umul64hi((uint64_t)x, magic) : x; }
};

// What decides a candidate's class, per configuration: a combination is a word of eight bytes (units per type), so the
// types that cannot host their degree, or do not fit a segment's memory, are byte masks, and the units of a zone are
// added up in 16-bit lanes (a lane holds at most 16 units x 96 stages) and compared with the most the zone can give,
// floor(available / GPUs of one unit): exactly the comparison of the GPU counts.
struct MixedClassTab {
    MixedConfig k;
    uint64_t lo, hi;                     // flat indices of the configuration
    uint32_t valid, stages[SAILOR_SEG_MAX], bad[SAILOR_SEG_MAX];     // bad: bit g, some stage of the segment does not fit type g
    MixedDivisor radix, n_comb;          // radix = zones x combinations (32-bit walk when the configuration allows it)
    uint64_t bad_bytes[SAILOR_SEG_MAX], inv_bytes;
    uint64_t cap[SAILOR_Z_MAX][2];       // 16-bit lanes per type, top bit set
};
constexpr uint64_t MIX_LANE_TOP = 0x8000800080008000ull;

__device__ __forceinline__ uint64_t type_bytes(uint32_t bits) {          // bit g -> byte g
    uint64_t m = 0;
#pragma unroll
    for (uint32_t g = 0; g < SAILOR_T_MAX; ++g) m |= ((bits >> g) & 1u) ? 0xffull << (8 * g) : 0ull;
    return m;
}

// A thread per candidate; a block takes one stretch of consecutive candidates of the range.  Bound: integer issue
// (about 150 instructions a candidate).  Workload 2's model, pipelines of up to four stages, replicas in quarters:
// 1.62e6 candidates, of which three availability snapshots leave 3.5e3 to 1.4e5.  A search that gave every candidate
// a warp (2 960 warp-instructions each) took 5.42 ms; classes first and a warp per candidate left 1.21 ms; classes
// first and a thread per candidate left 0.24 ms (35 us of it here).
__global__ void __launch_bounds__(MIXS_THREADS) mixed_class_kernel(const __grid_constant__ MixedSearchParams mp) {
    __shared__ MixedClassTab t;
    __shared__ unsigned int s_class[3];
    TabView v;
    v.bind(mp.blob, mp.blob);
    const TabHdr* h = v.h;
    const uint32_t T = h->T, Z = h->Z, tid = threadIdx.x, lane = tid & 31u;
    const uint64_t n = mp.range_hi - mp.range_lo, share = (n + gridDim.x - 1) / gridDim.x;
    uint64_t pos = mp.range_lo + share * blockIdx.x;
    const uint64_t stop = pos + share < mp.range_hi ? pos + share : mp.range_hi;
    uint32_t n_inv = 0, n_oom = 0, n_over = 0;
    if (mp.range_lo == 0 && blockIdx.x == 0 && tid == 0) mp.out->span.start = device_ns();
    if (tid < 3) s_class[tid] = 0;
    uint32_t cfg = 0;
    if (pos < stop) {
        uint32_t lo = 0, hi = mp.n_config;
        while (hi - lo > 1) {
            const uint32_t mid = (lo + hi) >> 1;
            if (mp.cfg_flat_base[mid] <= pos) lo = mid; else hi = mid;
        }
        cfg = lo;
    }
    for (; pos < stop; ++cfg) {
        __syncthreads();
        if (tid == 0) {
            t.k = mixed_config_of(mp.sp, cfg);
            t.lo = mp.cfg_flat_base[cfg];
            t.hi = mp.cfg_flat_base[cfg + 1];
            t.valid = h->gbs % ((uint64_t)t.k.D * h->mbs_values[t.k.mi]) == 0 ? 1u : 0u;
            t.radix.set(Z * mp.sp.n_comb[t.k.di]);
            t.n_comb.set(mp.sp.n_comb[t.k.di]);
            uint32_t inv = 0;
            for (uint32_t g = 0; g < T; ++g) {
                const uint32_t tpi = mp.sp.tp_idx_of_type[g];
                if (h->tp_values[tpi] > h->gpn[g] || !((h->heads_ok >> tpi) & 1u)) inv |= 1u << g;
            }
            t.inv_bytes = type_bytes(inv);
        }
        if (tid < SAILOR_SEG_MAX) t.bad[tid] = t.stages[tid] = 0;
        __syncthreads();
        const MixedConfig k = t.k;
        const uint64_t n_b = h->gbs / ((uint64_t)k.D * h->mbs_values[k.mi]);
        const uint32_t base = h->n_blocks / k.P, extra = h->n_blocks - base * k.P;
        for (uint32_t x = tid; x < k.P * T; x += MIXS_THREADS) {          // memory of every stage on every type
            const uint32_t i = x / T, g = x - i * T, seg = i * k.nseg / k.P, tpi = mp.sp.tp_idx_of_type[g];
            const bool e = (i == 0) && h->has_embed, hd = (i == k.P - 1) && h->has_head;
            const uint64_t inflight = (uint64_t)(k.P - i) < n_b ? (uint64_t)(k.P - i) : n_b;
            const size_t comp = (size_t)((e ? 2u : 0u) + (hd ? 1u : 0u)) * h->chain_len + base + (i < extra ? 1u : 0u);
            const uint64_t* mm = v.cmp_mem + (((comp * h->n_tp + tpi) * h->n_mbs + k.mi) * 2 + k.rc) * 2;
            if (mm[0] + inflight * mm[1] + h->reserved[g] > h->capacity[g]) atomicOr(&t.bad[seg], 1u << g);
            if (g == 0) atomicAdd(&t.stages[seg], 1u);
        }
        for (uint32_t x = tid; x < 2 * Z; x += MIXS_THREADS) {
            uint64_t word = MIX_LANE_TOP;
            for (uint32_t q = 0; q < 4; ++q) {
                const uint32_t g = 4 * (x & 1u) + q;
                if (g >= T) break;
                const uint32_t tp = h->tp_values[mp.sp.tp_idx_of_type[g]];
                const uint64_t most = mp.avail[(x >> 1) * T + g] / ((uint64_t)k.per_unit * tp);
                word |= (most < 0x7fffull ? most : 0x7fffull) << (16 * q);
            }
            t.cap[x >> 1][x & 1u] = word;
        }
        __syncthreads();
        if (tid < SAILOR_SEG_MAX) t.bad_bytes[tid] = type_bytes(t.bad[tid]);
        __syncthreads();
        const uint64_t end = t.hi < stop ? t.hi : stop;
        if (!t.valid) {
            if (tid == 0) atomicAdd(&mp.counters[1], (unsigned long long)(end - pos));
            pos = end;
            continue;
        }
        const uint64_t* combs = mp.combs + mp.sp.comb_off[k.di];
        const bool narrow = ((t.hi - t.lo) >> 32) == 0;
        const uint64_t inv_bytes = t.inv_bytes;
        for (uint64_t at = pos; at < end; at += MIXS_THREADS) {
            const uint64_t flat = at + tid;
            bool left = false;
            if (flat < end) {
                uint64_t rem = flat - t.lo, used = 0, misfit = 0;
                uint64_t w0[SAILOR_SEG_MAX], w1[SAILOR_SEG_MAX];          // units x stages per type, 16-bit lanes
                uint32_t zone[SAILOR_SEG_MAX];
#pragma unroll
                for (int q = SAILOR_SEG_MAX - 1; q >= 0; --q) {
                    w0[q] = w1[q] = 0;
                    zone[q] = 0xffffffffu;
                    if ((uint32_t)q >= k.nseg) continue;
                    uint32_t dg;
                    if (narrow) {
                        const uint32_t x = (uint32_t)rem, y = t.radix.quotient(x);
                        dg = x - y * t.radix.d;
                        rem = y;
                    } else {
                        dg = (uint32_t)(rem % t.radix.d);
                        rem /= t.radix.d;
                    }
                    zone[q] = t.n_comb.quotient(dg);
                    const uint64_t word = __ldg(&combs[dg - zone[q] * t.n_comb.d]);
                    used |= word;
                    misfit |= word & t.bad_bytes[q];
                    const uint32_t lo = (uint32_t)word, hi = (uint32_t)(word >> 32);
                    w0[q] = ((uint64_t)__byte_perm(lo, 0, 0x4342) << 32 | __byte_perm(lo, 0, 0x4140)) * t.stages[q];
                    if (T > 4) w1[q] = ((uint64_t)__byte_perm(hi, 0, 0x4342) << 32 | __byte_perm(hi, 0, 0x4140)) * t.stages[q];
                }
                if (used & inv_bytes) ++n_inv;
                else if (misfit) ++n_oom;
                else {
                    bool over = false;
#pragma unroll
                    for (uint32_t q = 0; q < SAILOR_SEG_MAX; ++q) {
                        if (q >= k.nseg) break;
                        uint64_t s0 = 0, s1 = 0;                          // all that the segment's zone has to give
#pragma unroll
                        for (uint32_t p = 0; p < SAILOR_SEG_MAX; ++p)
                            if (zone[p] == zone[q]) { s0 += w0[p]; s1 += w1[p]; }
                        over |= ((t.cap[zone[q]][0] - s0) & MIX_LANE_TOP) != MIX_LANE_TOP;
                        if (T > 4) over |= ((t.cap[zone[q]][1] - s1) & MIX_LANE_TOP) != MIX_LANE_TOP;
                    }
                    if (over) ++n_over;
                    left = !over;
                }
            }
            const uint32_t votes = __ballot_sync(FULL, left);
            if (votes) {
                uint32_t first = 0;
                if (lane == 0) first = (uint32_t)atomicAdd(&mp.counters[MIXC_QUEUED], (unsigned long long)__popc(votes));
                first = __shfl_sync(FULL, first, 0);
                if (left) mp.queue[first + __popc(votes & ((1u << lane) - 1u))] = (uint32_t)(flat - mp.range_lo);
            }
        }
        pos = end;
    }
    n_inv = __reduce_add_sync(FULL, n_inv);
    n_oom = __reduce_add_sync(FULL, n_oom);
    n_over = __reduce_add_sync(FULL, n_over);
    __syncthreads();
    if (lane == 0) {
        if (n_inv) atomicAdd(&s_class[0], n_inv);
        if (n_oom) atomicAdd(&s_class[1], n_oom);
        if (n_over) atomicAdd(&s_class[2], n_over);
    }
    __syncthreads();
    if (tid < 3 && s_class[tid]) atomicAdd(&mp.counters[1 + tid], (unsigned long long)s_class[tid]);
}

// One candidate by one thread.  All stages of a segment split their replicas alike, so a pipeline (one group per
// segment) is walked segment by segment and stretch by stretch, a stretch being consecutive stages of one layer
// make-up: its stage time is one table entry (PieceRec) plus one tabulated message time, and its sums take one addition
// per stage, in stage order.  Operation by operation where roundings are concerned this is simulate_mixed_warp.
// `zone` and `word` (units per type, a byte each) describe the segments; the candidate is known to be valid.
struct MixedScore { double t_iter, cost; };

__device__ __forceinline__ MixedScore mixed_evaluate(const MixedSearchParams& mp, const TabView& v, const MixedConfig& k,
                                                     const uint32_t (&zone)[SAILOR_SEG_MAX], const uint64_t (&word)[SAILOR_SEG_MAX]) {
    const TabHdr* h = v.h;
    const PieceRec* piece = reinterpret_cast<const PieceRec*>(mp.blob + h->off_piece);
    const double* intra2 = reinterpret_cast<const double*>(mp.blob + h->off_lnk_intra2);
    const double* inter2 = reinterpret_cast<const double*>(mp.blob + h->off_lnk_inter2);
    const double* zone2 = reinterpret_cast<const double*>(mp.blob + h->off_lnk_zone2);
    const uint32_t T = h->T, Z = h->Z, n_mbs = h->n_mbs, mi = k.mi, P = k.P, D = k.D, nseg = k.nseg;
    const uint32_t piece_stride = T * h->n_tp * n_mbs * 2;
    const uint64_t n_b = h->gbs / ((uint64_t)D * h->mbs_values[mi]);
    const uint32_t base = h->n_blocks / P, extra = h->n_blocks - base * P;
    const double steps = (double)(2 * (uint64_t)(D - 1)), coef = steps / (double)D;
    auto entry = [&](uint32_t g) { return ((g * h->n_tp + mp.sp.tp_idx_of_type[g]) * n_mbs + mi) * 2 + k.rc; };
    auto seg_end = [&](uint32_t s) { return ((s + 1) * P + nseg - 1) / nseg; };      // stage i is in segment floor(i nseg / P)
    // the stretch that starts at stage i: its make-up, and where it ends (with the segment, after the embedding stage,
    // where the extra blocks run out, before the head stage)
    auto stretch = [&](uint32_t i, uint32_t stop, uint32_t& end) {
        const bool e = (i == 0) && h->has_embed, hd = (i == P - 1) && h->has_head;
        end = stop;
        if (e) end = 1;
        else {
            if (i < extra && extra < end) end = extra;
            if (h->has_head && i < P - 1 && P - 1 < end) end = P - 1;
        }
        return ((e ? 2u : 0u) + (hd ? 1u : 0u)) * h->chain_len + base + (i < extra ? 1u : 0u);
    };

    // price rate (stage after stage, group after group), synchronisation, update, transfer cost
    double rate = 0.0, max_sync = 0.0, max_u = 0.0, c_comm = 0.0;
    const double xbytes = (double)(2 * n_b * (uint64_t)D * v.p2p[mi]);
#pragma unroll 1
    for (uint32_t s = 0, i = 0; s < nseg; ++s) {
        const uint32_t z = s == 0 ? zone[0] : s == 1 ? zone[1] : s == 2 ? zone[2] : zone[3];
        const uint64_t w = s == 0 ? word[0] : s == 1 ? word[1] : s == 2 ? word[2] : word[3];
        const uint32_t stop = seg_end(s);
        double term[SAILOR_MIX_GROUPS_MAX];
        uint32_t ng = 0, tp_least = 0xffffffffu, tpi_least = 0;          // the ring moves the largest shard (smallest tp)
#pragma unroll
        for (uint32_t q = 0; q < SAILOR_MIX_GROUPS_MAX; ++q) term[q] = 0.0;
        for (uint64_t left = w; left;) {
            const uint32_t g = (uint32_t)(__ffsll((long long)left) - 1) >> 3, tpi = mp.sp.tp_idx_of_type[g], tp = h->tp_values[tpi];
            const uint32_t count = ((uint32_t)(w >> (8 * g)) & 0xffu) * k.per_unit;
            const double x = mul_rn((double)(count * tp), v.price_s[z * T + g]);
#pragma unroll
            for (uint32_t q = 0; q < SAILOR_MIX_GROUPS_MAX; ++q) term[q] = q == ng ? x : term[q];
            if (tp < tp_least) { tp_least = tp; tpi_least = tpi; }
            ++ng;
            left &= ~(0xffull << (8 * g));
        }
        for (uint32_t n = i; n < stop; ++n)
#pragma unroll
            for (uint32_t q = 0; q < SAILOR_MIX_GROUPS_MAX; ++q)
                if (q < ng) rate = add_rn(rate, term[q]);
        while (i < stop) {
            uint32_t end;
            const uint32_t comp = stretch(i, stop, end);
            const double gradbytes = v.cmp_grad[(size_t)comp * h->n_tp + tpi_least];
            for (uint64_t left = w; left;) {
                const uint32_t g = (uint32_t)(__ffsll((long long)left) - 1) >> 3, d = z * T + g;
                max_u = dmax(max_u, piece[(size_t)comp * piece_stride + entry(g)].upd);
                if (D > 1) {
                    const bool intra = ng == 1 && (uint64_t)D * h->tp_values[mp.sp.tp_idx_of_type[g]] <= h->gpn[g];
                    max_sync = dmax(max_sync, allreduce_bytes_time(v, d, intra, gradbytes, D, steps, coef));
                }
                left &= ~(0xffull << (8 * g));
            }
            i = end;
        }
        if (s + 1 < nseg) {
            const uint32_t zn = s == 0 ? zone[1] : s == 1 ? zone[2] : zone[3];
            if (zn != z) c_comm = add_rn(c_comm, mul_rn(xbytes, v.egress[z * Z + zn]));
        }
    }

    // the pipelines: from one group boundary (in units) to the next all replicas see the same groups
    const uint32_t units = D / k.per_unit;
    uint64_t rest[SAILOR_SEG_MAX];                       // groups after the current one
    uint32_t type[SAILOR_SEG_MAX], upto[SAILOR_SEG_MAX]; // the current group's type, the unit it ends at
#pragma unroll
    for (uint32_t s = 0; s < SAILOR_SEG_MAX; ++s) { rest[s] = s < nseg ? word[s] : 0ull; type[s] = upto[s] = 0; }
    double max_pp = 0.0;
    for (uint32_t u = 0; u < units;) {
        uint32_t next = units;
#pragma unroll
        for (uint32_t s = 0; s < SAILOR_SEG_MAX; ++s) {
            if (s >= nseg) break;
            if (upto[s] == u) {
                type[s] = (uint32_t)(__ffsll((long long)rest[s]) - 1) >> 3;
                upto[s] += (uint32_t)(rest[s] >> (8 * type[s])) & 0xffu;
                rest[s] &= ~(0xffull << (8 * type[s]));
            }
            next = upto[s] < next ? upto[s] : next;
        }
        double sum_t = 0.0, max_t = 0.0;
#pragma unroll 1
        for (uint32_t s = 0, i = 0; s < nseg; ++s) {
            const uint32_t z = s == 0 ? zone[0] : s == 1 ? zone[1] : s == 2 ? zone[2] : zone[3];
            const uint32_t g = s == 0 ? type[0] : s == 1 ? type[1] : s == 2 ? type[2] : type[3];
            const uint64_t w = s == 0 ? word[0] : s == 1 ? word[1] : s == 2 ? word[2] : word[3];
            const uint32_t stop = seg_end(s), d = z * T + g, tp = h->tp_values[mp.sp.tp_idx_of_type[g]];
            const uint32_t count = ((uint32_t)(w >> (8 * g)) & 0xffu) * k.per_unit;
            const double c2_self = (2 * (uint64_t)count * tp <= h->gpn[g] ? intra2 : inter2)[d * n_mbs + mi];
            const uint32_t ent = entry(g);
            while (i < stop) {
                uint32_t end;
                const double fb = piece[(size_t)stretch(i, stop, end) * piece_stride + ent].fb;
                const uint32_t n_plain = end - i - (end == stop ? 1u : 0u);
                if (n_plain) {
                    const double t = add_rn(fb, c2_self);
                    max_t = dmax(max_t, t);
                    sum_t = add_n(sum_t, t, n_plain);
                }
                if (end == stop) {                       // the segment's last stage sends to the next segment, or is the final stage
                    double t = fb;
                    if (stop < P) {
                        const uint32_t zn = s == 0 ? zone[1] : s == 1 ? zone[2] : zone[3];
                        const uint32_t gn = s == 0 ? type[1] : s == 1 ? type[2] : type[3];
                        const uint64_t wn = s == 0 ? word[1] : s == 1 ? word[2] : word[3];
                        double c2;
                        if (zn != z) c2 = zone2[(z * Z + zn) * n_mbs + mi];
                        else if (gn == g && (uint64_t)count * tp + (uint64_t)(((uint32_t)(wn >> (8 * g)) & 0xffu) * k.per_unit) * tp <= h->gpn[g])
                            c2 = intra2[d * n_mbs + mi];
                        else {
                            c2 = inter2[d * n_mbs + mi];
                            if (gn != g) c2 = dmax(c2, inter2[(z * T + gn) * n_mbs + mi]);
                        }
                        t = add_rn(fb, c2);
                    }
                    max_t = dmax(max_t, t);
                    sum_t = add_rn(sum_t, t);
                }
                i = end;
            }
        }
        max_pp = dmax(max_pp, add_rn(sum_t, mul_rn((double)n_b, max_t)));
        u = next;
    }
    MixedScore o;
    o.t_iter = add_rn(add_rn(max_pp, max_sync), max_u);
    o.cost = add_rn(mul_rn(rate, o.t_iter), c_comm);
    return o;
}

// A thread per queued candidate: evaluation, constraint, top-k list of the warp.  Warps take 32 consecutive entries
// (neighbours in the space: alike), the first ones of all blocks before the second ones, so a short queue spreads over
// the SMs.
__global__ void __launch_bounds__(MIXS_THREADS, 2) plan_mixed_kernel(const __grid_constant__ MixedSearchParams mp) {
    __shared__ Hit s_hits[MIXS_WARPS][SAILOR_K_MAX];
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const uint64_t n = *reinterpret_cast<volatile const unsigned long long*>(&mp.counters[MIXC_QUEUED]);
    Hit* mine = mp.partial + (size_t)blockIdx.x * SAILOR_K_MAX;
    if ((uint64_t)blockIdx.x * 32 >= n) {                      // nothing for this block
        if (!mp.carry_lists && tid == 0) { mine[0].score = make_inf(); mine[0].flat = ~0ull; }
        return;
    }
    TabView v;
    v.bind(mp.blob, mp.blob);
    WarpTopK top;
    top.init();
    if (mp.carry_lists && warp == 0) {
        const Hit had = mine[0].flat != ~0ull && lane < mp.k ? mine[lane] : Hit{make_inf(), ~0ull};
        top.merge_sorted(had.score, had.flat, mp.k, lane);
    }
    uint32_t n_over = 0, n_feasible = 0;                       // a range holds at most 2^23 candidates
    double min_cost = make_inf();
    for (uint64_t e0 = ((uint64_t)warp * gridDim.x + blockIdx.x) * 32; e0 < n; e0 += (uint64_t)gridDim.x * MIXS_WARPS * 32) {
        const uint64_t e = e0 + lane;
        bool good = false;
        double score = make_inf();
        uint64_t flat = 0;
        if (e < n) {
            flat = mp.range_lo + mp.queue[e];
            uint32_t lo = 0, hi = mp.n_config;
            while (hi - lo > 1) {
                const uint32_t mid = (lo + hi) >> 1;
                if (mp.cfg_flat_base[mid] <= flat) lo = mid; else hi = mid;
            }
            const MixedConfig k = mixed_config_of(mp.sp, lo);
            const uint32_t n_comb = mp.sp.n_comb[k.di];
            const uint64_t radix = (uint64_t)v.h->Z * n_comb;
            uint64_t rem = flat - mp.cfg_flat_base[lo], word[SAILOR_SEG_MAX];
            uint32_t zone[SAILOR_SEG_MAX];
            const bool narrow = (rem >> 32) == 0;              // the usual case: 32-bit divisions
#pragma unroll
            for (int s = SAILOR_SEG_MAX - 1; s >= 0; --s) {
                word[s] = 0;
                zone[s] = 0;
                if ((uint32_t)s >= k.nseg) continue;
                uint32_t dg;
                if (narrow) {
                    const uint32_t x = (uint32_t)rem, y = x / (uint32_t)radix;
                    dg = x - y * (uint32_t)radix;
                    rem = y;
                } else {
                    dg = (uint32_t)(rem % radix);
                    rem /= radix;
                }
                zone[s] = dg / n_comb;
                word[s] = mp.combs[mp.sp.comb_off[k.di] + (dg - zone[s] * n_comb)];
            }
            const MixedScore o = mixed_evaluate(mp, v, k, zone, word);
            bool over = false;
            if (mp.budget > 0.0 && o.cost > mp.budget) over = true;
            if (mp.min_rate > 0.0 && 1.0 / o.t_iter < mp.min_rate) over = true;
            if (over) n_over++;
            else {
                n_feasible++;
                good = true;
                min_cost = o.cost < min_cost ? o.cost : min_cost;
                score = mp.obj == SAILOR_OBJ_MAX_THROUGHPUT ? o.t_iter : mp.obj == SAILOR_OBJ_MIN_COST ? o.cost : mul_rn(o.t_iter, o.cost);
            }
        }
        top.offer(good && score <= top.thr_score, score, flat, mp.k, lane);
    }
    n_over = __reduce_add_sync(FULL, n_over);
    n_feasible = __reduce_add_sync(FULL, n_feasible);
    min_cost = warp_min_positive(min_cost);
    if (lane == 0) {
        if (n_over) atomicAdd(&mp.counters[4], (unsigned long long)n_over);
        if (n_feasible) {
            atomicAdd(&mp.counters[5], (unsigned long long)n_feasible);
            atomicMin(&mp.counters[MIXC_MIN_COST], (unsigned long long)__double_as_longlong(min_cost));
        }
    }
    s_hits[warp][lane].score = top.score;
    s_hits[warp][lane].flat = top.flat;
    __syncthreads();
    if (warp == 0) {
        for (uint32_t w = 1; w < MIXS_WARPS; ++w) {
            if (s_hits[w][0].flat == ~0ull) continue;
            top.merge_sorted(s_hits[w][lane].score, s_hits[w][lane].flat, mp.k, lane);
        }
        mine[lane].score = lane < mp.k ? top.score : make_inf();
        mine[lane].flat = lane < mp.k ? top.flat : ~0ull;
    }
}

// Merge the blocks' lists; the winners are built and simulated again for the result records, a warp each.  DEEP: the
// space has pipelines of more than 32 stages.  Results and counters go straight into the host's memory; the counters are
// put back to their starting values for the next search.
template <bool DEEP> constexpr uint32_t MIXF_WARPS = DEEP ? 4 : 16;
template <bool DEEP>
struct MixFinishWarp {                   // what a warp of it keeps in shared memory
    static constexpr uint32_t STAGES = DEEP ? SAILOR_MIX_P_MAX : 32;
    MixScratch<STAGES> scratch;
    uint64_t plan[(offsetof(sailor_mixed_plan, stage) + STAGES * sizeof(sailor_mixed_stage)) / 8];   // the record, cut to STAGES stages
};

template <bool DEEP>
__global__ void __launch_bounds__(32 * MIXF_WARPS<DEEP>) mixed_finish_kernel(const __grid_constant__ MixedSearchParams mp) {
    constexpr uint32_t NW = MIXF_WARPS<DEEP>;
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ uint64_t mbar;
    __shared__ Hit s_hits[NW][SAILOR_K_MAX];
    __shared__ uint32_t s_sel[SAILOR_K_MAX], s_n;
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const uint32_t static_bytes = reinterpret_cast<const TabHdr*>(mp.blob)->static_bytes;
    if (!bulk_load(dyn, mp.blob, static_bytes, &mbar)) {
        if (tid == 0) atomicExch(&mp.counters[MIXC_ERROR], 1ull);
        for (uint32_t x = tid; x < static_bytes / 16; x += 32 * NW)
            reinterpret_cast<uint4*>(dyn)[x] = reinterpret_cast<const uint4*>(mp.blob)[x];
        __syncthreads();
    }
    TabView v;
    v.bind(dyn, mp.blob);
    const uint32_t T = v.h->T, Z = v.h->Z;
    MixFinishWarp<DEEP>& mine = reinterpret_cast<MixFinishWarp<DEEP>*>(dyn + static_bytes)[warp];
    sailor_mixed_plan* plan = reinterpret_cast<sailor_mixed_plan*>(mine.plan);
    const uint32_t n = merge_block_lists<NW>(mp.partial, mp.n_partial, mp.k, s_hits, s_sel, &s_n);
    for (uint32_t j = warp; j < n; j += NW) {
        const uint64_t flat = s_hits[0][j].flat;
        mixed_candidate(mp, T, Z, flat, plan, MixFinishWarp<DEEP>::STAGES, lane);
        const SimOut o = simulate_mixed_warp(v, mp.blob, mp.avail, *plan, mine.scratch, lane);
        __syncwarp();
        sailor_mixed_result* r = mp.out->results + j;
        if (lane == 0) {
            r->flat = flat; r->t_iter = o.t_iter; r->cost = o.cost; r->peak_mem = o.peak_mem;
            r->score = s_hits[0][j].score; r->status = o.status; r->_pad = 0;
        }
        // the record, word by word
        const uint64_t* src = reinterpret_cast<const uint64_t*>(plan);
        uint64_t* dst = reinterpret_cast<uint64_t*>(&r->plan);
        for (uint32_t x = lane; x < sizeof(sailor_mixed_plan) / 8; x += 32) dst[x] = x < sizeof(mine.plan) / 8 ? src[x] : 0ull;
        __syncwarp();
    }
    if (tid < MIXC_N) {
        volatile unsigned long long* live = mp.counters;
        mp.out->counters[tid] = tid == 0 ? mp.n_total : tid == MIXC_FOUND ? n : live[tid];
        live[tid] = tid == MIXC_MIN_COST ? COST_BITS_START : 0ull;
    }
    if (tid == 0) mp.out->span.end = device_ns();
}

}  // namespace sailor
