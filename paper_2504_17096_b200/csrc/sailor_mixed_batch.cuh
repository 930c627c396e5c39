// Batches of plans with mixed replicas (Sailor Sec. 4.2, Sec. 4.3): the kernel behind sailor_simulate_mixed for plans of
// up to 32 stages.
//
// A plan is small (workload 5: 9 stages, 18 groups, 5 different pipelines on average), so a warp that takes one plan at a
// time leaves most of its lanes idle in every step of it.  Here a block takes as many plans at a time as have one stage per
// thread together, orders them by depth, and goes through them in steps with a thread on
//   a stage (of any of them): its record is read and checked, its groups' table entries are read, its memory,
//       synchronisation, update time and transfer cost formed and its items (stage, group) written down;
//   a sum or a maximum over a plan's items or stages, in order;
//   a pipeline (of any of them): a walk over its plan's stages;
//   a plan.
// Bound: issue slots (44 % busy, 456 warp-instructions a plan, 25 of 32 lanes) and barriers between steps.  Random plans of
// workload 5, 2.6e5 of them: 481 us with a warp per plan (1 424 warp-instructions), 245 us this way; 6.0e4 plans of workloads
// 1, 2, 3, 5: 110 144 152 129 -> 56 79 82 63 us.  A warp with plans of its own, 64 stages at a time without barriers, took 328 us
// (steps with a lane per plan ran a few lanes wide); blocks with the batch's plans in input order 281 (each batch waits for its
// deepest plan).  Two blocks of 384 threads 250 us, three of 256 254, three of 320 271, two of 512 262; four steps of a walk side by
// side instead of three, and the window's records asked for at its beginning, 250 -> 245.
// Replica numbers are below 128 (MIXB_D_MAX), so the three group boundaries of a stage are bytes of a word, and the group
// that replica k falls into is one subtraction and a population count.  Of a plan with more replicas only the order of its
// boundaries matters to the pipelines: each takes its place among them as its number (96 at most), after two more barriers
// where such a plan is among those evaluated together (6.0e4 plans of workload 3 with 256 replicas: 175 us by a warp each,
// 117 this way; left to a few warps of the block 436).  Contexts with larger nodes than the packed items can tell apart keep a
// warp per plan.
// Sums whose order of additions is part of the result are one thread's, term after term, as in simulate_mixed_warp.
#pragma once

#include "sailor_mixed.cuh"

namespace sailor {

constexpr uint32_t MIXB_THREADS = 384;
constexpr uint32_t MIXB_WARPS = MIXB_THREADS / 32;
constexpr uint32_t MIXB_BLOCKS = 2;              // of an SM
constexpr uint32_t MIXB_P_MAX = 32;              // stages of a plan
constexpr uint32_t MIXB_D_MAX = 128;             // replicas of a stage whose numbers are kept; of more, boundaries are numbered in order
constexpr uint32_t MIXB_WINDOW = 256;   // plans ordered at a time
constexpr uint32_t MIXB_STAGES = MIXB_THREADS;   // stages evaluated at a time
constexpr uint32_t MIXB_PLANS = 60;              // their plans, at most
constexpr uint32_t MIXB_ITEMS = 5 * MIXB_STAGES / 2;         // their items (stage, group); a plan alone has at most 128
constexpr uint32_t MIXB_COUNTERS = 48 * MIXB_PLANS;          // GPUs taken per (plan, zone, type)
constexpr uint32_t MIXB_PIPES = MIXB_ITEMS + MIXB_PLANS;
constexpr uint32_t MIXB_PIPE_WORDS = (MIXB_PIPES + 31) / 32;
constexpr uint32_t MIXB_WIDE = 1u << 16;         // with a stage's items: its plan has more than MIXB_D_MAX replicas
constexpr uint32_t MIXB_GPUS_MAX = 8191;         // of an item, saturating: 13 bits; a node has fewer
constexpr uint32_t MIXB_AHEAD = 4;               // steps of a walk whose loads are in flight together
static_assert(MIXB_ITEMS >= SAILOR_MIX_GROUPS_MAX * MIXB_P_MAX && MIXB_STAGES >= MIXB_P_MAX && MIXB_COUNTERS >= R_MAX, "a plan fits");
static_assert(SAILOR_T_MAX * SAILOR_TP_MAX <= MIXB_THREADS && SAILOR_T_MAX <= 8 && MIXB_WARPS <= 32 && MIXB_PIPE_WORDS <= 32 && MIXB_PLANS <= 64, "bits and lanes");
static_assert((SAILOR_MIX_GROUPS_MAX - 1) * MIXB_P_MAX < MIXB_D_MAX, "a plan's boundaries, numbered from 1, fit where replica numbers do");

struct alignas(16) MixbHead {        // of a plan of the window, deepest first
    double nb, xbytes;
    uint32_t P, D, mr, nb_cap;       // mr: (mbs index, recomputation) as one index; nb_cap: microbatches in flight, at most
    uint32_t blocks;                 // layers of a stage << 8 | stages with one more
    uint32_t s0;                     // stages of the plans before it
    uint32_t status, at;             // at: its place in the block's share
};
struct MixbPlan {                    // of a plan that is being evaluated
    uint32_t item0, item_end;        // its items
    uint32_t pipe0, pipe_end;        // its pipelines
};
struct alignas(16) MixbStage {       // what a pipeline needs of a stage
    uint32_t ends;                   // replicas before the second, third, fourth group, a byte each: bit 7 set where there is one
    uint32_t first;                  // first item; bit 31: the next stage is in another zone
    double cross2;                   // doubled message time to it
};
struct alignas(16) MixbItem {
    double fb;                       // f + b (+ f with recomputation)
    uint32_t key;                    // type << 13 | GPUs; << 16: one more than the GPUs left on its node, 0 when it does not fit one
    uint32_t digit;
};
struct alignas(16) MixbDigit {       // of a (zone, type)
    double2 ring[2];                 // alpha, 1 / bandwidth: between nodes, inside one
    double price;
    uint32_t avail, _pad;
};
struct alignas(16) MixbShared {
    MixbItem item[MIXB_ITEMS];
    MixbStage stage[MIXB_STAGES];
    double term[4][MIXB_STAGES];                     // of a stage: transfer cost, synchronisation, update, memory (bytes)
    double rate[MIXB_ITEMS];
    double pp[MIXB_PIPES];                           // times of the pipelines
    MixbHead head[MIXB_WINDOW];
    double2 ring[MIXB_WINDOW];                       // 2 (D - 1), 2 (D - 1) / D of its plans
    MixbPlan plan[MIXB_PLANS];
    double total[MIXB_PLANS][5];                     // price rate, transfer cost, synchronisation, update, memory
    uint32_t counter[MIXB_COUNTERS];                 // zero between batches
    uint32_t starts[2][MIXB_PLANS][MIXB_D_MAX / 32]; // bit k: a pipeline starts at replica k (of the plans being evaluated, of the next)
    MixbDigit digit[R_MAX];
    uint4 tp[SAILOR_T_MAX * SAILOR_TP_MAX];          // per (type, tp index): tp (bit 31: the type cannot host it), table entry, GPUs per node
    uint64_t capacity[SAILOR_T_MAX];
    uint64_t p2p[SAILOR_MBS_MAX];
    uint32_t mbs[SAILOR_MBS_MAX];
    uint32_t blocks[MIXB_P_MAX + 1];
    uint32_t pipe_bits[MIXB_PIPE_WORDS];             // bit t: a plan's first pipeline
    uint32_t bin_n[32], bin_plan[32], bin_stage[32]; // by depth, deepest first
    uint32_t warp_sum[MIXB_WARPS];
    uint32_t n_listed, n_stages, n_pipes, fit;
    // The block's share of the batch.  Here and not in registers, which the steps below need (3 to 5 % of a large batch).
    uint64_t lo;                                     // first plan
    const unsigned char* plans;                      // its record
    uint32_t share, windows, pos, size;              // plans, windows left, the next one
    uint64_t next_head[MIXB_WINDOW];                 // its records' heads, each for the thread that asked for it
    uint8_t has_pipes[MIXB_PLANS];                   // the plans that have any
};
static_assert(MIXB_PLANS <= 256 && MIXB_WINDOW <= 256 && MIXB_WINDOW <= MIXB_THREADS, "bytes; a thread per plan");
static_assert(offsetof(MixbShared, starts) % 16 == 0, "read as words of 16 bytes");

// Other batches are evaluated by a warp per plan (simulate_mixed_each_kernel): its blocks lay out fewer tables and pass fewer
// barriers.  What decides is how deep plans can be: a record's room and the model's blocks bound it.  us a call by a warp per
// plan and by blocks, three types, plans of up to so many stages, degrees up to 32 (up to 128):
//    4:  17 6.3 9.3 (6.7 9.3), 1 000 7.2 10.3 (8.2 10.3), 3 500 8.3 10.3 (8.3 10.3)
//    8:  17 8.3 10.3 (8.2 10.3), 2 047 8.3 10.3 (8.3 10.3), 3 500 9.2 10.3 (10.3 10.3)
//   12: 100 8.3 10.3 (8.3 10.3), 1 000 8.3 10.3 (10.3 10.3), 2 047 10.3 10.5 (10.3 10.3)
//   16: 100 9.3 10.3 (10.3 10.3), 1 500 10.3 10.7 (11.0 10.8), 2 500 10.8 11.3 (12.4 11.3)
//   24: 300 10.3 10.3 (14.4 10.6), 1 000 10.7 12.3 (14.9 12.3), 2 500 12.4 12.4 (16.4 12.4)
//   32:  17 12.4 10.3 (16.4 10.3), 1 000 12.4 12.4 (18.3 12.4), 2 500 14.4 12.4 (20.5 12.7)
// Workload 1 (24 blocks, degrees up to 32, one zone with two types) keeps a warp per plan for longer.  Contexts with nodes too
// large for the packed items keep it for batches of any size.
inline bool mixb_takes(const TabHdr& h, uint32_t max_stages, uint64_t n) {
    for (uint32_t g = 0; g < h.T; ++g)
        if (h.gpn[g] >= MIXB_GPUS_MAX) return false;
    const uint32_t deepest = max_stages < h.n_blocks ? max_stages : h.n_blocks;
    return n >= (deepest <= 8 ? 4096 : deepest <= 16 ? 1536 : deepest <= 24 && h.R <= 2 ? 2048 : 17);
}

// All that the kernels with a warp per plan are given: launches take longer with more (one plan, calls back to back: 6.4 to 7.7 us
// with the tables' addresses and small tables as well, 6.2 to 7.2 without).
struct MixbCall {
    const unsigned char* blob;
    const uint16_t* avail;
    const unsigned char* plans;
    uint64_t n;
    double *t_iter, *cost;
    uint64_t* peak_mem;
    uint32_t* status;
    unsigned int *error, *deep_seen;
    uint32_t stride, max_stages, report_bad;
};
static_assert(sizeof(MixbCall) <= 128, "few launch parameters");

struct MixbParams : MixbCall {
    uint64_t gbs;
    const PieceRec* piece;
    const double *zone2, *egress, *grad, *intra_p, *inter_p, *inter_a, *inter_i, *intra_a, *intra_i, *price_s, *inter2, *intra2;
    const uint64_t* p2p;
    uint64_t capacity[SAILOR_T_MAX];
    uint32_t tp_values[SAILOR_TP_MAX], mbs_values[SAILOR_MBS_MAX], gpn[SAILOR_T_MAX], heads_ok;
    uint32_t n_blocks, T, Z, R, n_tp, n_mbs, chain_len, has_embed, has_head, piece_stride;
    uint32_t plans_max;              // plans at a time
};

inline size_t mixb_smem(const TabHdr& h) { return sizeof(MixbShared) + 2 * (size_t)h.R * h.n_mbs * sizeof(double); }

inline MixbParams mixb_params(const MixbCall& call, const TabHdr& h) {
    MixbParams p = {};
    static_cast<MixbCall&>(p) = call;
    const unsigned char* blob = call.blob;
    auto table = [&](uint32_t off) { return off ? reinterpret_cast<const double*>(blob + off) : nullptr; };
    p.gbs = h.gbs;
    p.piece = reinterpret_cast<const PieceRec*>(blob + h.off_piece);
    p.zone2 = table(h.off_lnk_zone2); p.egress = table(h.off_egress); p.grad = table(h.off_cmp_grad);
    p.intra_p = table(h.off_intra_p); p.inter_p = table(h.off_inter_p);
    p.inter_a = table(h.off_inter_a); p.inter_i = table(h.off_inter_i); p.intra_a = table(h.off_intra_a); p.intra_i = table(h.off_intra_i);
    p.price_s = table(h.off_price_s); p.inter2 = table(h.off_lnk_inter2); p.intra2 = table(h.off_lnk_intra2);
    p.p2p = reinterpret_cast<const uint64_t*>(blob + h.off_p2p);
    memcpy(p.capacity, h.capacity, sizeof(p.capacity));
    memcpy(p.tp_values, h.tp_values, sizeof(p.tp_values));
    memcpy(p.mbs_values, h.mbs_values, sizeof(p.mbs_values));
    memcpy(p.gpn, h.gpn, sizeof(p.gpn));
    p.heads_ok = h.heads_ok;
    p.n_blocks = h.n_blocks; p.T = h.T; p.Z = h.Z; p.R = h.R; p.n_tp = h.n_tp; p.n_mbs = h.n_mbs; p.chain_len = h.chain_len;
    p.has_embed = h.has_embed; p.has_head = h.has_head;
    p.piece_stride = h.T * h.n_tp * h.n_mbs * 2;
    p.plans_max = MIXB_COUNTERS / h.R < MIXB_PLANS ? MIXB_COUNTERS / h.R : MIXB_PLANS;
    return p;
}

__device__ __forceinline__ uint32_t warp_scan(uint32_t x, uint32_t lane) {       // inclusive
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t up = __shfl_up_sync(MIX_FULL, x, o);
        if (lane >= (uint32_t)o) x += up;
    }
    return x;
}

// Position of the n-th set bit (from 0) of 128 bits that have more.
__device__ __forceinline__ uint32_t nth_bit(uint4 w, uint32_t n) {
    uint32_t at = 0, m = w.x;
    uint32_t c = __popc(m);
    if (n >= c) { n -= c; at = 32; m = w.y; c = __popc(m);
        if (n >= c) { n -= c; at = 64; m = w.z; c = __popc(m);
            if (n >= c) { n -= c; at = 96; m = w.w; } } }
#pragma unroll
    for (uint32_t half = 16; half; half >>= 1) {
        c = __popc(m & ((1u << half) - 1u));
        if (n >= c) { n -= c; at += half; m >>= half; }
    }
    return at;
}

__device__ __forceinline__ void mixb_store(const MixbCall& p, uint64_t j, const SimOut& o) {
    if (p.t_iter) p.t_iter[j] = o.t_iter;
    if (p.peak_mem) p.peak_mem[j] = o.peak_mem;
    if (p.cost) p.cost[j] = o.cost;
    if (p.status) p.status[j] = o.status;
    if (p.report_bad && (o.status & SAILOR_ST_BAD_RECORD)) atomicOr(p.error, SIM_ERR_BAD_RECORD);
}

// The ring over a link with a bandwidth polynomial (`without`: when it has none).  A call, so that its divisions stay out of
// the loop over a stage's groups.
__device__ __noinline__ double mixb_poly_ring(const double* poly, uint32_t d, double volume, double grad, uint32_t D, double without) {
    return poly ? volume / poly_bw(poly + 4 * d, grad / (double)D) : without;
}

// Boundaries of a stage as mixb_bounds packs them, numbered from 1 by their place among those of the plan's stages: the
// places in the form of MixbStage::ends, their bits set in `starts`.  Equal ones have one place.
__device__ __noinline__ uint32_t mixb_places(const uint2* of_plan, uint32_t P, uint2 mine, uint32_t* starts) {
    const uint32_t b[3] = {mine.x & 0xffffu, mine.x >> 16, mine.y};
    uint32_t place[3] = {1, 1, 1}, ends = 0;
    for (uint32_t y = 0; y < P; ++y) {
        const uint2 o = of_plan[y];
#pragma unroll
        for (uint32_t q = 0; q < 3; ++q) place[q] += ((o.x & 0xffffu) < b[q]) + ((o.x >> 16) < b[q]) + (o.y < b[q]);
    }
#pragma unroll
    for (uint32_t q = 0; q < 3; ++q)
        if (b[q] != 0xffffu) {
            ends |= (place[q] | 0x80u) << (8 * q);
            atomicOr(&starts[place[q] >> 5], 1u << (place[q] & 31u));
        }
    return ends;
}

// The replicas before a stage's second, third and fourth group, 16 bits each (0xffff: there is none; a valid plan has fewer).
__device__ __forceinline__ uint2 mixb_bounds(const uint32_t (&g)[SAILOR_MIX_GROUPS_MAX], uint32_t ng) {
    const uint32_t b1 = g[0] >> 16, b2 = b1 + (g[1] >> 16), b3 = b2 + (g[2] >> 16);
    return make_uint2((ng > 1 ? b1 : 0xffffu) | (ng > 2 ? b2 & 0xffffu : 0xffffu) << 16, ng > 3 ? b3 & 0xffffu : 0xffffu);
}

__global__ void __launch_bounds__(MIXB_THREADS, MIXB_BLOCKS) simulate_mixed_kernel(const __grid_constant__ MixbParams p) {
    extern __shared__ __align__(16) unsigned char dyn[];
    MixbShared& s = *reinterpret_cast<MixbShared*>(dyn);
    double* const s_inter = reinterpret_cast<double*>(dyn + sizeof(MixbShared));       // doubled message time, [mbs][digit]: between nodes
    double* const s_intra = s_inter + p.R * p.n_mbs;                                   // inside one
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    constexpr uint32_t NO_TIME = SAILOR_ST_INVALID | SAILOR_ST_BAD_RECORD;

    // The block's share of the batch, a window at a time (of equal parts).
    const uint64_t lo = p.n / gridDim.x * blockIdx.x + (blockIdx.x < p.n % gridDim.x ? blockIdx.x : p.n % gridDim.x);
    const uint32_t share = (uint32_t)(p.n / gridDim.x) + (blockIdx.x < p.n % gridDim.x ? 1u : 0u);
    const unsigned char* const first_plan = p.plans + lo * p.stride;
    const uint32_t n_windows = (share + MIXB_WINDOW - 1) / MIXB_WINDOW, first_size = share / n_windows;
    auto read_head = [&](const unsigned char* plans, uint32_t x, uint32_t n) {     // (records start at multiples of 8 bytes)
        if (tid < n)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(&s.next_head[tid])),
                         "l"(plans + (size_t)(x + tid) * p.stride) : "memory");
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    read_head(first_plan, 0, first_size);
    {                                                              // (all addresses and small tables are launch parameters: no load waits for another)
        for (uint32_t x = tid; x < p.R * p.n_mbs; x += MIXB_THREADS) {
            const uint32_t d = x / p.n_mbs, to = (x - d * p.n_mbs) * p.R + d;
            s_inter[to] = p.inter2[x];
            s_intra[to] = p.intra2[x];
        }
        for (uint32_t d = tid; d < p.R; d += MIXB_THREADS) {
            MixbDigit& x = s.digit[d];
            x.ring[0] = make_double2(p.inter_a[d], p.inter_i[d]);
            x.ring[1] = make_double2(p.intra_a[d], p.intra_i[d]);
            x.price = p.price_s[d];
            x.avail = p.avail[d];
        }
        if (tid < SAILOR_T_MAX * SAILOR_TP_MAX) {
            const uint32_t g = tid / SAILOR_TP_MAX, ti = tid % SAILOR_TP_MAX;
            if (g < p.T && ti < p.n_tp) {                          // (availability is 16 bits: no count beyond 65 536 matters)
                const uint32_t tp = p.tp_values[ti], gpn = p.gpn[g];
                s.tp[tid] = make_uint4((tp < 65536u ? tp : 65536u) | (tp > gpn || !((p.heads_ok >> ti) & 1u) ? 0x80000000u : 0u),
                                       (g * p.n_tp + ti) * p.n_mbs * 2, gpn, 0u);
            }
        }
        if (tid == 0) {
            s.plans = first_plan;
            s.lo = lo;
            s.pos = 0;
            s.size = first_size;
            s.windows = n_windows;
            s.share = share;
        }
        if (tid < SAILOR_T_MAX) s.capacity[tid] = p.capacity[tid];
        if (tid < p.n_mbs) { s.p2p[tid] = p.p2p[tid]; s.mbs[tid] = p.mbs_values[tid]; }
        if (tid >= 1 && tid <= MIXB_P_MAX) { const uint32_t b = p.n_blocks / tid; s.blocks[tid] = b << 8 | (p.n_blocks - b * tid); }
        for (uint32_t x = tid; x < MIXB_COUNTERS; x += MIXB_THREADS) s.counter[x] = 0;
        if (tid < 2 * MIXB_PLANS) reinterpret_cast<uint4*>(s.starts)[tid] = make_uint4(1, 0, 0, 0);
    }

    uint32_t turn = 0;
    __syncthreads();
    for (;;) {
        // ---- a thread per plan: sort out and order, deepest first (a counting sort; any order gives the same results) ---------
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        const uint32_t size = s.size, pos = s.pos;
        const uint64_t head = tid < size ? s.next_head[tid] : 0ull;
        const uint32_t P0 = (uint32_t)head & 0xff, mi = (uint32_t)(head >> 8) & 0xff, D = (uint32_t)(head >> 32) & 0xffff;
        const bool have = tid < size;
        const uint32_t at = pos + tid;
        if (tid < 32) s.bin_n[tid] = 0;
        __syncthreads();
        uint32_t P = 0, rank = 0;
        if (have) {
            if (P0 < 1 || P0 > p.max_stages || D < 1 || mi >= p.n_mbs) {
                SimOut o;
                o.t_iter = o.cost = make_nan();
                o.peak_mem = 0;
                o.status = SAILOR_ST_BAD_RECORD;
                mixb_store(p, s.lo + at, o);
            } else if (P0 > MIXB_P_MAX) {
                *reinterpret_cast<volatile unsigned int*>(p.deep_seen) = 1u;             // left to the launch for deep plans
            } else {
                P = P0;
                rank = atomicAdd(&s.bin_n[MIXB_P_MAX - P], 1u);
                for (uint32_t x = 0; x < 8 + 20 * P; x += 128)       // its stages are read some batches later
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(s.plans + (size_t)at * p.stride + x));
            }
        }
        __syncthreads();
        if (warp == 0) {                                           // a bin per lane: plans and stages of deeper ones
            const uint32_t n = s.bin_n[lane], depth = MIXB_P_MAX - lane;
            const uint32_t n_plans = warp_scan(n, lane), stages = warp_scan(n * depth, lane);
            s.bin_plan[lane] = n_plans - n;
            s.bin_stage[lane] = stages - n * depth;
            if (lane == 31) { s.n_listed = n_plans; s.n_stages = stages; }
        }
        uint64_t n_b = 0;
        uint32_t status0 = 0;
        if (P) {
            const uint64_t dm = (uint64_t)D * s.mbs[mi];
            if (((p.gbs | dm) >> 32) == 0) {                       // the usual case: a 32-bit division
                const uint32_t q32 = (uint32_t)p.gbs / (uint32_t)dm;
                n_b = q32;
                if (q32 * (uint32_t)dm != (uint32_t)p.gbs) status0 = SAILOR_ST_INVALID;
            } else {
                n_b = p.gbs / dm;
                if (n_b * dm != p.gbs) status0 = SAILOR_ST_INVALID;
            }
        }
        const uint32_t left = s.windows - 1, next_size = left ? (s.share - pos - size) / left : 0u;
        read_head(s.plans, pos + size, next_size);
        __syncthreads();
        if (tid == 0) { s.windows = left; s.pos = pos + size; s.size = next_size; }
        if (P) {
            const uint32_t bin = MIXB_P_MAX - P;
            MixbHead hd;
            hd.nb = (double)n_b;
            hd.xbytes = (double)(2 * n_b * (uint64_t)D * s.p2p[mi]);
            hd.P = P;
            hd.D = D;
            hd.mr = mi * 2 + (((uint32_t)(head >> 16) & 0xff) ? 1u : 0u);
            hd.nb_cap = n_b > MIXB_P_MAX ? MIXB_P_MAX : (uint32_t)n_b;       // no stage holds more than P in flight
            hd.blocks = s.blocks[P];
            hd.s0 = s.bin_stage[bin] + rank * P;
            hd.status = status0;
            hd.at = at;
            s.head[s.bin_plan[bin] + rank] = hd;
            const double steps = (double)(2 * (D - 1));
            s.ring[s.bin_plan[bin] + rank] = make_double2(steps, steps / (double)D);
        }
        __syncthreads();

        // ---- as many plans at a time as have a stage per thread together --------------------------------------------------------
        for (uint32_t r0 = 0; r0 < s.n_listed; turn ^= 1u) {
            const uint32_t n_listed = s.n_listed, all_stages = s.n_stages;
            uint32_t (*const starts)[MIXB_D_MAX / 32] = s.starts[turn];
            // how many of the plans from r0 on, and which plan a thread's stage belongs to: a lane per plan (and per plan + 32)
            const uint32_t base = s.head[r0].s0;
            uint32_t np = 0, n_stages = 0, earlier = 0, begins = 0;
#pragma unroll
            for (uint32_t x = 0; x < MIXB_PLANS; x += 32) {
                const uint32_t r = r0 + x + lane;
                const uint32_t s_begin = r < n_listed ? s.head[r].s0 - base : all_stages - base;
                const uint32_t s_end = r + 1 < n_listed ? s.head[r + 1].s0 - base : all_stages - base;
                const bool in = r < n_listed && x + lane < p.plans_max && s_end <= MIXB_STAGES;
                np += __popc(__ballot_sync(MIX_FULL, in));
                n_stages = max(n_stages, __reduce_max_sync(MIX_FULL, in ? s_end : 0u));
                earlier += __popc(__ballot_sync(MIX_FULL, in && s_begin < 32 * warp));
                begins |= __reduce_or_sync(MIX_FULL, in && s_begin / 32 == warp ? 1u << (s_begin & 31u) : 0u);
            }
            // ---- a thread per stage: its record, checked -----------------------------------------------------------------------------
            const uint32_t rel = earlier + __popc(begins & (MIX_FULL >> (31u - lane))) - 1u;
            uint32_t i = 0, zones = 0, ng = 0, ends = 0, tpi_least = 0, wide = 0, g[SAILOR_MIX_GROUPS_MAX] = {0, 0, 0, 0};
            if (tid < n_stages) {
                MixbHead& hd = s.head[r0 + rel];
                i = tid - (hd.s0 - base);
                const uint32_t* rec = reinterpret_cast<const uint32_t*>(s.plans + (size_t)hd.at * p.stride + 8) + 5 * i;
                const uint32_t w0 = rec[0], zone = w0 & 0xff, next = i + 1 < hd.P ? rec[5] & 0xff : zone;
#pragma unroll
                for (uint32_t q = 0; q < SAILOR_MIX_GROUPS_MAX; ++q) g[q] = rec[1 + q];
                ng = (w0 >> 8) & 0xff;
                bool refuse = zone >= p.Z || ng < 1 || ng > SAILOR_MIX_GROUPS_MAX;
#pragma unroll
                for (uint32_t q = 0; q < SAILOR_MIX_GROUPS_MAX; ++q) refuse |= q < ng && ((g[q] & 0xff) >= p.T || ((g[q] >> 8) & 0xff) >= p.n_tp);
                if (refuse) ng = 0;
                uint32_t status = refuse ? SAILOR_ST_BAD_RECORD : 0u, run = 0, tp_least = 0xffffffffu;
                wide = hd.D > MIXB_D_MAX ? MIXB_WIDE : 0u;
                const uint32_t kept = wide ? 0u : MIXB_D_MAX;
                zones = zone | (next < p.Z ? next : zone) << 8;                // (the next is checked by the thread that has that stage)
#pragma unroll
                for (uint32_t q = 0; q < SAILOR_MIX_GROUPS_MAX; ++q) {
                    if (q >= ng) break;
                    const uint32_t ty = g[q] & 0xff, ti = (g[q] >> 8) & 0xff, cn = g[q] >> 16, tpw = s.tp[ty * SAILOR_TP_MAX + ti].x;
                    if (q && run < kept) {                                   // (a valid plan's are)
                        ends |= (run | 0x80u) << (8 * (q - 1));
                        atomicOr(&starts[rel][run >> 5], 1u << (run & 31u));
                    }
                    run += cn;
                    if (cn == 0 || tpw >> 31) status |= SAILOR_ST_INVALID;
                    if ((tpw & 0x7fffffffu) < tp_least) { tp_least = tpw & 0x7fffffffu; tpi_least = ti; }
                }
                if (run != hd.D) status |= SAILOR_ST_INVALID;
                if (status) atomicOr(&hd.status, status);
            }
            const uint32_t items = warp_scan(ng + wide, lane);
            if (lane == 31) s.warp_sum[warp] = items;
            if (tid < MIXB_PIPE_WORDS) s.pipe_bits[tid] = 0;
            if (tid == 0) s.fit = np;
            __syncthreads();
            const uint32_t of_warp = lane < MIXB_WARPS ? s.warp_sum[lane] : 0u;
            const uint32_t first = (__reduce_add_sync(MIX_FULL, lane < warp ? of_warp : 0u) + items - ng) % MIXB_WIDE;
            const uint32_t all_items = __reduce_add_sync(MIX_FULL, of_warp);
            if (all_items > MIXB_ITEMS) {                          // (the same for all threads; rare)
                if (first + ng > MIXB_ITEMS) atomicMin(&s.fit, rel);         // fewer plans, then
                uint2* const bounds = reinterpret_cast<uint2*>(s.term[0]);   // (not in use at this time)
                if (all_items >= MIXB_WIDE && tid < n_stages) bounds[tid] = mixb_bounds(g, ng);
                __syncthreads();
                np = s.fit;
                if (all_items >= MIXB_WIDE) {                      // numbers its boundaries by their order
                    if (wide) {
                        const MixbHead& hd = s.head[r0 + rel];
                        ends = mixb_places(bounds + (hd.s0 - base), hd.P, bounds[tid], starts[rel]);
                    }
                    __syncthreads();
                }
            }
            if (tid < MIXB_PLANS) *reinterpret_cast<uint4*>(s.starts[turn ^ 1u][tid]) = make_uint4(1, 0, 0, 0);
            if (warp == MIXB_WARPS - 1) {                          // counts the pipelines of the valid plans
                uint32_t n_pipes = 0, n_valid = 0;
                for (uint32_t x = 0; x < np; x += 32) {
                    const uint32_t r = x + lane;
                    const bool valid = r < np && !(s.head[r0 + r].status & NO_TIME);
                    uint32_t n = 0;
                    if (valid) {
                        const uint4 w = *reinterpret_cast<const uint4*>(starts[r]);
                        n = __popc(w.x) + __popc(w.y) + __popc(w.z) + __popc(w.w);
                    }
                    const uint32_t upto_n = warp_scan(n, lane), votes = __ballot_sync(MIX_FULL, valid), from = n_pipes + upto_n - n;
                    if (r < np) { s.plan[r].pipe0 = from; s.plan[r].pipe_end = from + n; }
                    if (valid) {
                        s.has_pipes[n_valid + __popc(votes & ((1u << lane) - 1u))] = (uint8_t)r;
                        atomicOr(&s.pipe_bits[from >> 5], 1u << (from & 31u));
                    }
                    n_pipes += __shfl_sync(MIX_FULL, upto_n, 31);
                    n_valid += __popc(votes);
                }
                if (lane == 0) s.n_pipes = n_pipes;
            }
            // ---- a thread per stage: its items, its terms, what pipelines need of it -------------------------------------------
            if (tid < n_stages && rel < np) {
                MixbHead& hd = s.head[r0 + rel];
                const uint32_t P = hd.P, D = hd.D, mr = hd.mr, zone = zones & 0xff, next = zones >> 8;
                if (i == 0) s.plan[rel].item0 = first;
                if (i + 1 == P) s.plan[rel].item_end = first + ng;
                if (ng) {
                    const bool e = i == 0 && p.has_embed, last = i == P - 1 && p.has_head;
                    const uint32_t comp = ((e ? 2u : 0u) + (last ? 1u : 0u)) * p.chain_len + (hd.blocks >> 8) + (i < (hd.blocks & 0xffu) ? 1u : 0u);
                    const PieceRec* piece = p.piece + (size_t)(comp * p.piece_stride + mr);
                    uint4 tp = s.tp[(g[0] & 0xff) * SAILOR_TP_MAX + ((g[0] >> 8) & 0xff)];
                    PieceRec pr = load_piece(piece + tp.y);
                    const double grad = __ldg(&p.grad[comp * p.n_tp + tpi_least]);           // the ring moves the largest shard (smallest tp)
                    const bool crosses = next != zone;
                    double cross2 = 0.0, comm = 0.0;
                    if (crosses) {
                        cross2 = __ldg(&p.zone2[(zone * p.Z + next) * p.n_mbs + (mr >> 1)]);
                        comm = mul_rn(hd.xbytes, __ldg(&p.egress[zone * p.Z + next]));
                    }
                    const double2 rg = s.ring[r0 + rel];
                    const double steps = rg.x, volume = mul_rn(rg.y, grad);
                    const uint32_t left = P - i, inflight = left < hd.nb_cap ? left : hd.nb_cap;
                    double sync = 0.0, upd = 0.0;
                    uint64_t peak = 0;
                    uint32_t status = 0;
#pragma unroll
                    for (uint32_t q = 0; q < SAILOR_MIX_GROUPS_MAX; ++q) {
                        const uint32_t ty = g[q] & 0xff, cn = g[q] >> 16, d = zone * p.T + ty, tp_now = tp.x & 0x7fffffffu, gpn = tp.z;
                        const PieceRec cur = pr;
                        if (q + 1 < SAILOR_MIX_GROUPS_MAX && q + 1 < ng) {
                            tp = s.tp[(g[q + 1] & 0xff) * SAILOR_TP_MAX + ((g[q + 1] >> 8) & 0xff)];
                            pr = load_piece(piece + tp.y);
                        }
                        const MixbDigit& dg = s.digit[d];
                        const uint32_t gpus = cn * tp_now, taken = gpus > 65536u ? 65536u : gpus;
                        if (atomicAdd(&s.counter[rel * p.R + d], taken) + taken > dg.avail) status |= SAILOR_ST_OVER_AVAIL;
                        MixbItem x;
                        x.fb = cur.fb;
                        x.key = (ty << 13 | (taken < MIXB_GPUS_MAX ? taken : MIXB_GPUS_MAX)) | (taken <= gpn ? gpn - taken + 1 : 0u) << 16;
                        x.digit = d;
                        s.item[first + q] = x;
                        s.rate[first + q] = mul_rn((double)gpus, dg.price);
                        const uint64_t m = cur.mem0r + (uint64_t)inflight * cur.mem1;
                        if (m > s.capacity[ty]) status |= SAILOR_ST_OOM;
                        peak = m > peak ? m : peak;
                        upd = dmax(upd, cur.upd);
                        if (D > 1) {
                            const bool intra = ng == 1 && D * tp_now <= gpn;
                            const double2 ab = dg.ring[intra];
                            double x_t = mul_rn(volume, ab.y);
                            if (p.intra_p || p.inter_p) x_t = mixb_poly_ring(intra ? p.intra_p : p.inter_p, d, volume, grad, D, x_t);
                            sync = dmax(sync, add_rn(x_t, mul_rn(steps, ab.x)));
                        }
                        if (q + 1 >= ng) break;
                    }
                    MixbStage st;
                    st.ends = ends;
                    st.first = first | (crosses ? 0x80000000u : 0u);
                    st.cross2 = cross2;
                    s.stage[tid] = st;
                    s.term[0][tid] = comm;
                    s.term[1][tid] = sync;
                    s.term[2][tid] = upd;
                    reinterpret_cast<uint64_t*>(s.term[3])[tid] = peak;
                    if (status) atomicOr(&hd.status, status);
                }
            }
            __syncthreads();

            // ---- a warp per 32 sums or maxima of plans, from the last warp on, and per 32 pipelines, from the first -------------
            for (uint32_t task = MIXB_WARPS - 1 - warp; task < 5 * ((np + 31) / 32); task += MIXB_WARPS) {
                uint32_t which = task, r = lane;
                for (; which >= 5; which -= 5) r += 32;
                if (r >= np) continue;
                const MixbHead& hd = s.head[r0 + r];
                if (which < 2) {
                    double sum = 0.0;
                    if (!(hd.status & NO_TIME)) {
                        const double* y = which ? &s.term[0][hd.s0 - base] : &s.rate[s.plan[r].item0];
                        const double* const end_y = y + (which ? hd.P : s.plan[r].item_end - s.plan[r].item0);
#pragma unroll 4
                        for (; y < end_y; ++y) sum = add_rn(sum, *y);
                    }
                    s.total[r][which] = sum;
                } else if (!(hd.status & SAILOR_ST_BAD_RECORD)) {
                    const uint64_t* y = reinterpret_cast<const uint64_t*>(&s.term[which - 1][hd.s0 - base]);     // (non-negative: the bits order)
                    const uint64_t* const end_y = y + hd.P;
                    uint64_t most = 0;
#pragma unroll 4
                    for (; y < end_y; ++y) most = *y > most ? *y : most;
                    reinterpret_cast<uint64_t*>(s.total[r])[which] = most;
                }
            }
            const uint32_t n_pipes = s.n_pipes;
            for (uint32_t word = warp; 32 * word < n_pipes; word += MIXB_WARPS) {
                const uint32_t t = 32 * word + lane;
                const uint32_t before = __reduce_add_sync(MIX_FULL, lane < word ? __popc(s.pipe_bits[lane]) : 0);
                const uint32_t r = s.has_pipes[before + __popc(s.pipe_bits[word] & (MIX_FULL >> (31u - lane))) - 1u];
                if (t >= n_pipes) continue;
                const MixbHead& hd = s.head[r0 + r];
                const uint32_t k = nth_bit(*reinterpret_cast<const uint4*>(starts[r]), t - s.plan[r].pipe0);
                const uint32_t n = hd.P, K = (0x80u + k) * 0x010101u;
                const uint4* st = reinterpret_cast<const uint4*>(&s.stage[hd.s0 - base]);
                const double* inter = s_inter + (hd.mr >> 1) * p.R;
                const double* intra = s_intra + (hd.mr >> 1) * p.R;
                // a byte of K less a boundary below 128 keeps its top bit where replica k is not before the boundary
                auto item_of = [&](const uint4& raw) {
                    const uint32_t at = (raw.y & 0xffffu) + __popc((K - (raw.x & 0x7f7f7fu)) & raw.x & 0x808080u);
                    return *reinterpret_cast<const uint4*>(&s.item[at]);
                };
                auto f64 = [](uint32_t x, uint32_t y) { return __hiloint2double((int)y, (int)x); };
                const uint32_t last = n - 1;
                uint4 raw = st[0], cur = item_of(raw);
                double c_cur = inter[cur.w], sum_t = 0.0, max_t = 0.0;
                auto step = [&](const uint4& next_raw, const uint4& nx, double c_next) {
                    double c2 = dmax(c_cur, c_next);                 // unlike types, or not on one node: the slower end counts
                    if ((nx.z & 0xffffu) - (cur.z & 0xe000u) < cur.z >> 16) c2 = intra[cur.w];
                    if (raw.y >> 31) c2 = f64(raw.z, raw.w);
                    const double t_y = add_rn(f64(cur.x, cur.y), c2);
                    sum_t = add_rn(sum_t, t_y);
                    max_t = dmax(max_t, t_y);
                    raw = next_raw;
                    cur = nx;
                    c_cur = c_next;
                };
                uint32_t y = 0;
#pragma unroll 1
                for (; y + MIXB_AHEAD <= last; y += MIXB_AHEAD) {    // the loads of some steps side by side
                    uint4 raws[MIXB_AHEAD], its[MIXB_AHEAD];
                    double cs[MIXB_AHEAD];
#pragma unroll
                    for (uint32_t x = 0; x < MIXB_AHEAD; ++x) raws[x] = st[y + 1 + x];
#pragma unroll
                    for (uint32_t x = 0; x < MIXB_AHEAD; ++x) its[x] = item_of(raws[x]);
#pragma unroll
                    for (uint32_t x = 0; x < MIXB_AHEAD; ++x) cs[x] = inter[its[x].w];
#pragma unroll
                    for (uint32_t x = 0; x < MIXB_AHEAD; ++x) step(raws[x], its[x], cs[x]);
                }
#pragma unroll 1
                for (; y < last; ++y) {
                    const uint4 one = st[y + 1], it = item_of(one);
                    step(one, it, inter[it.w]);
                }
                const double fb = f64(cur.x, cur.y);                 // the final stage sends nothing
                sum_t = add_rn(sum_t, fb);
                max_t = dmax(max_t, fb);
                s.pp[t] = add_rn(sum_t, mul_rn(hd.nb, max_t));
            }
            __syncthreads();

            // ---- a thread per plan ------------------------------------------------------------------------------------------
            if (tid < np) {
                const MixbHead& hd = s.head[r0 + tid];
                const uint32_t status = hd.status;
                SimOut o;
                o.t_iter = o.cost = make_nan();
                o.peak_mem = 0;
                o.status = SAILOR_ST_BAD_RECORD;
                if (!(status & SAILOR_ST_BAD_RECORD)) {
                    o.status = status;
                    o.peak_mem = reinterpret_cast<const uint64_t*>(s.total[tid])[4];
                    if (!(status & SAILOR_ST_INVALID)) {
                        double max_pp = 0.0;
                        for (uint32_t t = s.plan[tid].pipe0; t < s.plan[tid].pipe_end; ++t) max_pp = dmax(max_pp, s.pp[t]);
                        o.t_iter = add_rn(add_rn(max_pp, s.total[tid][2]), s.total[tid][3]);
                        o.cost = add_rn(mul_rn(s.total[tid][0], o.t_iter), s.total[tid][1]);
                    }
                }
                mixb_store(p, s.lo + hd.at, o);
            }
            for (uint32_t x = tid; x < np * p.R; x += MIXB_THREADS) s.counter[x] = 0;
            r0 += np;
        }
        if (s.windows == 0) break;
    }
}

}  // namespace sailor
