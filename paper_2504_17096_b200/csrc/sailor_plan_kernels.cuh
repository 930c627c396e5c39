// Plan search kernels: candidates are generated on the device from their flat index,
// simulated (Sailor Sec. 4.3) and reduced to the k best under the objective (Sec. 4.2).
//
// Work decomposition.  A *configuration* is (P, mbs, tp, rc, D); its candidates differ only
// in the (type, zone) digit of each of its nseg segments.  An *item* is one assignment of
// all segments but the last (a prefix); a thread owns one item and walks the last segment's
// digit, so the running sums of the prefix (in stage order, exactly as a stage-by-stage
// evaluation would add them) are formed once and extended per candidate.  A *chunk* is
// PLAN_THREADS consecutive items of one configuration; blocks take chunks from an atomic
// counter, and rebuild the per-configuration stage tables in shared memory only when the
// configuration changes.  Lanes of a warp hold consecutive prefixes of one configuration,
// so loop trip counts are warp-uniform and per-digit table reads are broadcasts.
#pragma once

#include "sailor_tables.cuh"

namespace sailor {

constexpr int PLAN_THREADS = 256;
constexpr int PLAN_WARPS = PLAN_THREADS / 32;
#ifndef PLAN_DIGITS_PER_STEP
#define PLAN_DIGITS_PER_STEP 4      // candidates evaluated side by side per thread (independent chains)
#endif
#ifndef PLAN_MIN_BLOCKS
#define PLAN_MIN_BLOCKS 2
#endif
#ifndef PLAN_SCREEN_BLOCKS
#define PLAN_SCREEN_BLOCKS 3        // resident blocks per SM the screened kernels are compiled for (binary32 state is half as wide)
#endif
constexpr unsigned FULL = 0xffffffffu;
constexpr uint32_t WAIT_LIMIT = 1u << 22;   // bound of every spin-wait in this file

struct alignas(16) Hit {
    double score;
    uint64_t flat;
};

struct Ctrl {                       // one per context, device memory
    unsigned int work_counter;      // next chunk to hand out (starts at zero in every launch)
    unsigned int blocks_done;       // blocks of the running launch that have handed in their list
    unsigned long long stats[7];    // total, invalid, oom, over_avail, over_constraint, feasible, pruned_tp
    unsigned int wave_chunks;       // chunks of the current wave (searches in degree order)
    unsigned int n_cfg_evaluated;   // configurations selected by the waves so far
    unsigned long long min_cost_bits;   // min C_iter over feasible candidates, as ordered bits
    unsigned long long thr_bits;    // a score no candidate of the final top-k exceeds (ordered bits): the best k-th
                                    // best any warp has seen so far; lets all other warps skip what cannot matter
    double budget;                  // written by the cheapest-plan pass for the next pass
    unsigned int error;             // non-zero: a kernel gave up during this call (bounded wait ran out)
    unsigned int n_found;
    unsigned int no_number;         // a candidate that cannot be chosen cost 0 x infinity: never read (see evaluated())
    unsigned int _pad;
};

// What a pass leaves for the host (one device-to-host copy: the counters, then the k records).  The block that
// finishes a pass writes it and then puts the live counters back to their starting values, so that the next pass
// or the next call needs no clearing from the host.
struct PlanOut {
    Ctrl ctrl;
    DeviceSpan span;
    uint64_t ticket;                   // written last: which call the rest belongs to
    sailor_result results[SAILOR_K_MAX];
};

constexpr unsigned long long COST_BITS_START = 0x7ff0000000000000ull;   // +inf: above every cost

struct PlanParams {
    const unsigned char* blob;
    uint16_t avail[R_MAX];             // the availability snapshot rides in the launch parameters: a search needs no
                                       // copy of its own before it, and 128 bytes are well within the parameter space
    const uint32_t* cfg_chunk_start;   // [n_config + 1]
    const uint64_t* cfg_flat_base;     // [n_config]
    Ctrl* ctrl;
    Hit* partial;                      // [grid][SAILOR_K_MAX]
    uint32_t* partial_n;               // [grid]
    SpaceDesc sp;
    uint32_t n_config;
    uint32_t chunk_lo, chunk_hi, batch;
    uint64_t flat_lo, flat_hi;
    uint32_t k;
    uint32_t budget_from_ctrl;         // read the budget from ctrl->budget
    uint32_t p_max;                    // largest P of the space (sizes the stage tables)
    uint32_t live_mode;                // cfg_chunk_start counts only chunks of prefixes made of usable digits
    uint32_t min_tp_only;              // drop plans that also fit with a smaller tensor-parallel degree (H2)
    uint32_t carry_lists;              // a block starts from the list it left in `partial` (waves of one search)
    const uint32_t* chunk_hi_dev;      // non-null: chunks [0, *chunk_hi_dev) instead of [chunk_lo, chunk_hi)
    unsigned long long* cfg_best;      // non-null: [n_config] best feasible score per configuration (ordered bits)
    PlanOut* out;                      // where the block that finishes the pass leaves the results
    uint64_t ticket;                   // of the call
    uint32_t first;                    // this launch is the call's first: it stamps the start
    uint32_t finish;                   // this launch ends a pass: its last block merges the lists and writes `out`
    double next_budget_factor;         // > 0: the finishing block writes ctrl->budget = factor * best cost (next pass)
    uint32_t cost_only;                // the pass only looks for the cheapest feasible cost (no lists, no result records)
    uint32_t screen;                   // candidates are first evaluated in binary32 (SCREEN kernels): sizes the shared tables
    const uint4* cfg_cache;            // non-null: the per-configuration tables, built once per space (cfg_cache_kernel)
    uint32_t cache_head16, cache_arr16;    // 16-byte words of a cached record: CfgShared head, then the arrays
    double budget;                     // <= 0: none
    double min_rate;                   // <= 0: none
};

// ---- bounded bulk copy global -> shared (non-multicast cp.async.bulk + mbarrier) ------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Copies `bytes` (multiple of 16, both addresses 16-byte aligned) with one bulk-copy
// instruction issued by thread 0 and waits for it with a bounded spin.  Returns false if the
// wait ran out; the caller then falls back to plain loads and raises the error flag.
__device__ __forceinline__ bool bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* mbar) {
    const uint32_t bar = smem_u32(mbar);
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(bar)
                     : "memory");
    }
    uint32_t done = 0;
    for (uint32_t it = 0; it < WAIT_LIMIT && !done; ++it) {
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(bar)
            : "memory");
    }
    return __syncthreads_and((int)done) != 0;
}

// ---- warp-resident sorted top-k list: lane j holds the j-th best (score, flat) -------------
struct WarpTopK {
    double score;      // this lane's element
    uint64_t flat;
    double thr_score;  // element k-1 (warp-uniform): only strictly better candidates enter
    uint64_t thr_flat;

    __device__ __forceinline__ void init() {
        score = thr_score = make_inf();
        flat = thr_flat = ~0ull;
    }
    // Insert one candidate known to every lane.  (score, flat) pairs are unique.
    // Returns false when the candidate is not better than the current k-th (warp-uniform).
    __device__ __forceinline__ bool insert(double s, uint64_t f, uint32_t k, uint32_t lane) {
        if (!(s < thr_score || (s == thr_score && f < thr_flat))) return false;   // warp-uniform
        const bool before = (score < s) || (score == s && flat < f);
        const uint32_t pos = __popc(__ballot_sync(FULL, before));           // sorted: a prefix of lanes
        const double ps = __shfl_up_sync(FULL, score, 1);
        const uint64_t pf = __shfl_up_sync(FULL, flat, 1);
        if (lane > pos) { score = ps; flat = pf; }
        else if (lane == pos) { score = s; flat = f; }
        thr_score = __shfl_sync(FULL, score, k - 1);
        thr_flat = __shfl_sync(FULL, flat, k - 1);
        return true;
    }
    // Merge another ascending list of 32 (lane j passes its j-th element; empty slots are
    // (+inf, ~0)) into this one, keeping the 32 smallest of the union: min(a[j], b[31-j]) is a
    // bitonic sequence holding exactly those, and five compare-exchange stages sort it.
    __device__ __forceinline__ void merge_sorted(double bs, uint64_t bf, uint32_t k, uint32_t lane) {
        const double rs = __shfl_sync(FULL, bs, 31 - lane);
        const uint64_t rf = __shfl_sync(FULL, bf, 31 - lane);
        if (rs < score || (rs == score && rf < flat)) { score = rs; flat = rf; }
#pragma unroll
        for (int stride = 16; stride; stride >>= 1) {
            const double os = __shfl_xor_sync(FULL, score, stride);
            const uint64_t of = __shfl_xor_sync(FULL, flat, stride);
            const bool other_less = os < score || (os == score && of < flat);
            const bool upper = lane & stride;
            if (other_less != upper) { score = os; flat = of; }     // lower lane keeps the smaller, upper the larger
        }
        thr_score = __shfl_sync(FULL, score, k - 1);
        thr_flat = __shfl_sync(FULL, flat, k - 1);
    }
    // Sort the lanes' elements (empty slots are (+inf, ~0)) ascending: a bitonic network, fifteen compare-exchanges.
    __device__ __forceinline__ void sort(uint32_t k, uint32_t lane) {
#pragma unroll
        for (int size = 2; size <= 32; size <<= 1)
#pragma unroll
            for (int stride = size >> 1; stride; stride >>= 1) {
                const double os = __shfl_xor_sync(FULL, score, stride);
                const uint64_t of = __shfl_xor_sync(FULL, flat, stride);
                const bool other_less = os < score || (os == score && of < flat);
                const bool keep_larger = ((lane & stride) != 0) != ((lane & size) != 0);
                if (other_less != keep_larger) { score = os; flat = of; }
            }
        thr_score = __shfl_sync(FULL, score, k - 1);
        thr_flat = __shfl_sync(FULL, flat, k - 1);
    }
    // Offer per-lane candidates: `want` marks lanes whose candidate may qualify.
    __device__ __forceinline__ void offer(bool want, double s, uint64_t f, uint32_t k, uint32_t lane) {
        unsigned m = __ballot_sync(FULL, want);
        while (m) {
            const int src = __ffs(m) - 1;
            m &= m - 1;
            insert(__shfl_sync(FULL, s, src), __shfl_sync(FULL, f, src), k, lane);
        }
    }
};

// ---- per-configuration tables in shared memory ---------------------------------------------
//
// Inside one segment all stages share (type, zone, tp), so their per-microbatch times take at
// most four distinct values, in stage order: stage 0 (embedding), stages with one extra block,
// plain stages, the final stage (head, sends nothing).  A segment is therefore stored as four
// (count, value[digit]) runs; adding `count` copies of `value` one after the other is the same
// sequence of additions as walking the stages.  The last stage of a non-final segment sends to
// the next segment, so its time depends on two digits and is kept apart (fb_last + c2x).
constexpr int N_RUNS = 4;
constexpr uint32_t PLAN_PAD = PLAN_DIGITS_PER_STEP - 1;   // table entries past the last digit that a step may read

struct alignas(16) SegRec {                  // one per (segment, digit); 64 bytes, read as broadcasts
    double v[N_RUNS];            // t_i of each run (f + b + 2c with the next stage on the same digit)
    double tmax;                 // max of v[] over the non-empty runs
    double sync;                 // max all-reduce time over the segment's stages
    double upd;                  // max update time over the segment's stages
    double rate;                 // D * tp * price per second of one stage
};

// The binary32 screen (optional search mode): every candidate is first evaluated in binary32 from rounded copies of
// the tables; an item (a prefix with all its last digits) is evaluated again in binary64, exactly as without the
// screen, only when its best binary32 score comes within SCREEN_BAND of the score a candidate must beat to enter
// the top-k, or its cheapest binary32 cost within SCREEN_BAND of the cheapest cost known.  A binary32 evaluation
// rounds each table entry once (2^-24) and adds at most P + 4 positive terms (each addition 2^-24), multiplies
// twice and, for throughput per cost, once more: a relative error below (P + 12) * 2^-24 < 7e-6 for P <= 96 in time
// and cost, below 1.4e-5 in their product.  The band is 1e-4, so every candidate whose exact score could enter the
// list (or whose exact cost could be the cheapest) is looked at exactly: lists, counts and statistics are the
// exact search's, bit for bit.
constexpr double SCREEN_BAND = 1e-4;

struct alignas(16) SegRec32 {                // SegRec rounded to binary32; 32 bytes
    float v[N_RUNS];
    float tmax, sync, upd, rate;
};

struct alignas(16) CfgShared {
    // scalars (written by thread 0 / the build, read by all)
    Config cfg;
    uint32_t valid;              // gbs % (D*mbs) == 0 and heads % tp == 0
    uint32_t packed;             // prefixes are enumerated over the usable digits of each segment only
    uint32_t g_cnt[SAILOR_SEG_MAX];       // usable digits (valid type, fits in memory) per segment
    uint32_t g_magic[SAILOR_SEG_MAX];     // floor(2^32 / g_cnt) + 1, for division by g_cnt
    uint64_t live_items;         // product of g_cnt over the prefix segments
    uint8_t good_list[SAILOR_SEG_MAX][R_MAX];   // the usable digits of each segment, ascending
    uint32_t need_last;                   // need of the last segment
    uint32_t seg_a[SAILOR_SEG_MAX + 1];   // first stage of each segment; seg_a[nseg] = P
    uint32_t need[SAILOR_SEG_MAX];        // GPUs a segment takes of its digit: D * tp * stages
    uint32_t n_run[SAILOR_SEG_MAX][N_RUNS];   // stages in each run (without a non-final segment's last stage)
    double ar_steps, ar_coef;    // 2(D-1) and 2(D-1)/D of the ring all-reduce
    uint64_t n_b;
    uint64_t n_items;            // R^(nseg-1)
    uint64_t invalid_mask;       // digit d: tp > gpus_per_node[type(d)]
    uint64_t oom_mask[SAILOR_SEG_MAX];    // digit d: some stage of the segment does not fit type(d)
    uint32_t n_lower;            // smaller tensor-parallel degrees of the space that the model accepts (min_tp_only)
    uint32_t lower_tpi[SAILOR_TP_MAX];    // their tp indices
    uint64_t lower_fit[SAILOR_TP_MAX][SAILOR_SEG_MAX];   // digit d: every stage of the segment fits at that degree
    uint64_t flat_base;          // flat index of the configuration's first candidate
    uint32_t by_zone;            // sweeps take the last segment's digits zone by zone (see zones_pay)
    uint32_t _pad_head;
    // ---- everything above depends on the configuration and the context only, not on availability: it is what a
    // ---- cached record holds (with the arrays rec .. fb_last); everything below belongs to the block or the snapshot
    alignas(16) uint64_t avail_last;     // digit d: need[last] <= avail[d]
    uint32_t whole;              // all candidates of the configuration lie in the range searched
    uint32_t magic;              // floor(2^32 / R) + 1: x / R == umulhi(x, magic) for x < 2^26
    uint32_t cur_config;
    uint32_t next_chunk, batch_len;
    unsigned long long oom_stage[SAILOR_P_MAX];   // per stage: bit 8 j + g set when the stage does not fit type g
                                                  // at this configuration's degree (j = 0) or at lower_tpi[j - 1]
    uint64_t params[SAILOR_P_MAX];
    unsigned long long stat[7];
    unsigned long long thr_bits;     // the block's copy of Ctrl::thr_bits, lowered by its own warps as their lists fill
    unsigned long long minc_bits;    // screened search: the cheapest exact cost the block's warps have seen (ordered bits)
    uint64_t mbar;
};

struct CfgArrays {               // pointers into dynamic shared memory
    SegRec* rec;                 // [SEG_MAX][R]
    double* c2x;                 // [R][R]   2 * message time, index [next digit][this digit]
    double* commx;               // [R][Z]   transfer cost of one boundary, index [next digit][this zone]
    double* fb_last;             // [SEG_MAX][T]  f+b of a segment's last stage, per type
    double *fb, *uu;             // [P][T]   build scratch: f+b (+f if rc), update
    uint32_t* availv;            // [R]
    uint32_t* tz;                // [R]      type | zone << 8 of a digit
    uint32_t* chunk_tab;         // [n_config + 1] copy of the chunk offsets (spaces of fewer than PLAN_CFG_SMEM configurations)
    SegRec32* rec32;             // screened search: rec, c2x, commx rounded to binary32 (same shapes and padding)
    float* c2x32;
    float* commx32;
};

constexpr uint32_t PLAN_CFG_SMEM = 4096;

__host__ __device__ inline size_t plan_screen_bytes(uint32_t T, uint32_t Z) {
    const size_t R = (size_t)T * Z;
    return sizeof(SegRec32) * (SAILOR_SEG_MAX * R + PLAN_PAD) + sizeof(float) * ((R + PLAN_PAD) * R + (R + PLAN_PAD) * Z) + 32;
}

__host__ __device__ inline size_t plan_smem_bytes(uint32_t static_bytes, uint32_t p_max, uint32_t T, uint32_t Z, uint32_t n_config,
                                                  bool screen = false) {
    const size_t R = (size_t)T * Z;
    size_t n = static_bytes;
    if (screen) n += plan_screen_bytes(T, Z);
    if (n_config < 4096) n += sizeof(uint32_t) * ((size_t)n_config + 1);
    n += sizeof(SegRec) * (SAILOR_SEG_MAX * R + PLAN_PAD);               // padding digits, see walk_fast
    n += sizeof(double) * ((R + PLAN_PAD) * R + (R + PLAN_PAD) * Z + (size_t)SAILOR_SEG_MAX * T + 2 * (size_t)p_max * T);
    n += sizeof(uint32_t) * 2 * R;
    return (n + 15) & ~(size_t)15;
}

// A cached configuration record: the head of CfgShared up to avail_last, then the arrays rec, c2x, commx, fb_last
// (with their padding entries), both in 16-byte words.
__host__ __device__ inline uint32_t cache_head16() { return (uint32_t)(offsetof(CfgShared, avail_last) / 16); }
__host__ __device__ inline uint32_t cache_arr16(uint32_t T, uint32_t Z) {
    const size_t R = (size_t)T * Z;
    const size_t bytes = sizeof(SegRec) * (SAILOR_SEG_MAX * R + PLAN_PAD) +
                         sizeof(double) * ((R + PLAN_PAD) * R + (R + PLAN_PAD) * Z + (size_t)SAILOR_SEG_MAX * T);
    return (uint32_t)((bytes + 15) / 16);
}

__device__ __forceinline__ void carve(unsigned char* dyn, uint32_t static_bytes, uint32_t p_max, uint32_t T,
                                      uint32_t Z, CfgArrays& a, uint32_t n_config = 0, bool screen = false) {
    const uint32_t R = T * Z;
    a.rec = reinterpret_cast<SegRec*>(dyn + static_bytes);           // static_bytes is a multiple of 16
    double* p = reinterpret_cast<double*>(a.rec + (size_t)SAILOR_SEG_MAX * R + PLAN_PAD);
    a.c2x = p;       p += (size_t)(R + PLAN_PAD) * R;
    a.commx = p;     p += (size_t)(R + PLAN_PAD) * Z;
    a.fb_last = p;   p += (size_t)SAILOR_SEG_MAX * T;
    a.fb = p;        p += (size_t)p_max * T;
    a.uu = p;        p += (size_t)p_max * T;
    a.availv = reinterpret_cast<uint32_t*>(p);
    a.tz = a.availv + R;
    a.chunk_tab = a.tz + R;
    a.rec32 = nullptr;
    a.c2x32 = a.commx32 = nullptr;
    if (screen) {
        uintptr_t at = reinterpret_cast<uintptr_t>(a.chunk_tab + (n_config < PLAN_CFG_SMEM ? n_config + 1 : 0));
        at = (at + 15) & ~(uintptr_t)15;
        a.rec32 = reinterpret_cast<SegRec32*>(at);
        a.c2x32 = reinterpret_cast<float*>(a.rec32 + (size_t)SAILOR_SEG_MAX * R + PLAN_PAD);
        a.commx32 = a.c2x32 + (size_t)(R + PLAN_PAD) * R;
    }
}

// The binary32 copies of the tables of the configuration just built or loaded.  Called by the whole block; ends
// synchronised.
__device__ __forceinline__ void round_config32(const CfgArrays& a, uint32_t R, uint32_t Z) {
    const uint32_t tid = threadIdx.x;
    for (uint32_t x = tid; x < SAILOR_SEG_MAX * R + PLAN_PAD; x += PLAN_THREADS) {
        const SegRec& r = a.rec[x];
        SegRec32 q;
        for (int j = 0; j < N_RUNS; ++j) q.v[j] = __double2float_rn(r.v[j]);
        q.tmax = __double2float_rn(r.tmax); q.sync = __double2float_rn(r.sync);
        q.upd = __double2float_rn(r.upd); q.rate = __double2float_rn(r.rate);
        a.rec32[x] = q;
    }
    for (uint32_t x = tid; x < (R + PLAN_PAD) * R; x += PLAN_THREADS) a.c2x32[x] = __double2float_rn(a.c2x[x]);
    for (uint32_t x = tid; x < (R + PLAN_PAD) * Z; x += PLAN_THREADS) a.commx32[x] = __double2float_rn(a.commx[x]);
    __syncthreads();
}

// Run of stage i: 0 = stage 0 with the embedding, 1 = one extra block, 2 = plain, 3 = final stage.
__device__ __forceinline__ uint32_t run_of(const TabHdr* h, uint32_t P, uint32_t extra, uint32_t i) {
    if (i == P - 1) return 3;
    if (i == 0 && h->has_embed) return 0;
    return i < extra ? 1 : 2;                              // extra = n_blocks % P
}

// Zones that evaluate_only's first group takes besides the prefix's own.
__device__ __forceinline__ uint32_t zone_group(uint32_t Z) { return Z > 7 ? 7u : 4u; }
// Where a type's records are alike in all zones (price rate included), taking a sweep's last digits zone by zone pays if the
// first group is full; the zones beyond it go one at a time, a chain of additions each, which pays for last segments of up
// to five stages.  Sweeps of pipelines of one depth over 8 types, zone by zone against digit by digit, ms, last segments of
// 1, 4, 5, 6, 12 and 24 stages: 5 zones 2.9 4.2, 3.3 5.1, 4.8 7.0, 5.1 6.8, 7.4 8.8, 12.3 12.4; 7 zones 11.6 14.7,
// 17.8 18.1, 23.3 25.0, 25.7 24.3, 41.8 31.5, 74 45; 8 zones 14.7 24.2, 17.6 30.2, 23.3 41.9, 24.8 40.7, 35.8 52.7,
// 57.8 75.5.  Up to 4 zones, one at a time, 1.5 times the digits' time; with a price rate per zone 1.1 (5 zones), 1.06 (8).
__device__ __forceinline__ bool zones_pay(uint32_t Z, uint32_t stages) {
    const uint32_t group = zone_group(Z);
    return Z > group && (Z == group + 1 || stages <= 5);
}

// Build the tables of configuration `c`.  Called by the whole block; ends synchronised.  SWEEP: with `by_zone`, which only
// sweeps of every candidate read.
template <bool SWEEP>
static __device__ void build_config(const PlanParams& pp, const TabView& v, CfgShared& cs, CfgArrays& a, uint32_t c) {
    const TabHdr* h = v.h;
    const uint32_t T = h->T, Z = h->Z, R = h->R, tid = threadIdx.x;
    if (tid < 32) {                    // the first warp sets the configuration up, one segment per lane
        Config k;
        uint32_t valid = 0;
        if (tid == 0) {
            k = config_of(pp.sp, c);
            cs.cfg = k;
            const uint32_t tp0 = h->tp_values[k.tpi];
            const uint64_t dm = (uint64_t)k.D * h->mbs_values[k.mi];
            valid = (k.D >= 1 && h->gbs % dm == 0 && h->heads % tp0 == 0) ? 1u : 0u;
            cs.valid = valid;
            cs.n_b = k.D >= 1 ? h->gbs / dm : 0;
            cs.ar_steps = (double)(2 * (uint64_t)(k.D > 0 ? k.D - 1 : 0));     // ring all-reduce: 2(D-1) messages
            cs.ar_coef = k.D > 0 ? cs.ar_steps / (double)k.D : 0.0;
            cs.n_items = ipow64(R, k.nseg - 1);
            cs.flat_base = pp.cfg_flat_base[c];
            cs.by_zone = 0;
            cs._pad_head = 0;
            cs.packed = 0;             // decided at the end of the build, and only for valid configurations
            cs.cur_config = c;
            uint32_t n_lower = 0;
            if (pp.min_tp_only)
                for (uint32_t j = 0; j < pp.sp.n_tp; ++j) {
                    const uint32_t tj = pp.sp.tp_idx[j], tv = h->tp_values[tj];
                    if (tv < tp0 && h->heads % tv == 0 && n_lower < SAILOR_TP_MAX - 1) cs.lower_tpi[n_lower++] = tj;
                }
            cs.n_lower = n_lower;
        }
        const uint32_t P = __shfl_sync(FULL, k.P, 0), nseg = __shfl_sync(FULL, k.nseg, 0);
        const uint32_t D = __shfl_sync(FULL, k.D, 0), tp = h->tp_values[__shfl_sync(FULL, k.tpi, 0)];
        if (tid <= nseg) cs.seg_a[tid] = (tid * P + nseg - 1) / nseg;
        if (tid < nseg) {              // stages [lo, hi) of segment `tid`, counted per run in closed form
            const uint32_t lo = (tid * P + nseg - 1) / nseg, end = ((tid + 1) * P + nseg - 1) / nseg;
            const uint32_t extra = h->n_blocks % P;
            cs.need[tid] = D * tp * (end - lo);
            if (tid + 1 == nseg) cs.need_last = D * tp * (end - lo);
            cs.oom_mask[tid] = 0;
            for (uint32_t j = 0; j < SAILOR_TP_MAX; ++j) cs.lower_fit[j][tid] = 0;
            uint32_t hi = (tid + 1 < nseg) ? end - 1 : end;      // a non-final segment's last stage is kept apart
            const uint32_t c3 = (hi == P && hi > lo) ? 1u : 0u;   // the final stage
            hi -= c3;
            const uint32_t c0 = (lo == 0 && h->has_embed && hi > lo) ? 1u : 0u;
            const uint32_t lo1 = lo + c0;
            const uint32_t top = hi < extra ? hi : extra;
            const uint32_t c1 = top > lo1 ? top - lo1 : 0u;
            cs.n_run[tid][0] = c0;
            cs.n_run[tid][1] = c1;
            cs.n_run[tid][2] = hi > lo1 ? (hi - lo1) - c1 : 0u;
            cs.n_run[tid][3] = c3;
        }
        uint32_t inv_lo = 0, inv_hi = 0;                          // digits whose type cannot host tp
        {
            const uint32_t d0 = tid, d1 = tid + 32;
            inv_lo = __ballot_sync(FULL, d0 < R && tp > h->gpn[d0 % T]);
            inv_hi = __ballot_sync(FULL, d1 < R && tp > h->gpn[d1 % T]);
        }
        if (tid == 0) cs.invalid_mask = ((uint64_t)inv_hi << 32) | inv_lo;
    }
    for (uint32_t i = tid; i < SAILOR_P_MAX; i += PLAN_THREADS) cs.oom_stage[i] = 0;
    __syncthreads();
    const Config k = cs.cfg;
    const uint32_t P = k.P, tp = h->tp_values[k.tpi];
    if (!cs.valid) return;             // nothing of this configuration is evaluated (block-uniform)

    // phase A: per (stage, type) times and memory
    const uint32_t base = h->n_blocks / P, extra = h->n_blocks % P;
    for (uint32_t x = tid; x < P * T; x += PLAN_THREADS) {
        const uint32_t i = x / T, g = x % T;
        const uint32_t nb = base + (i < extra ? 1u : 0u);
        const bool e = (i == 0) && h->has_embed, hd = (i == P - 1) && h->has_head;
        const StageTimes st = stage_times(v, g, k.tpi, k.mi, nb, e, hd);
        const double b = k.rc ? add_rn(st.b, st.f) : st.b;
        a.fb[x] = add_rn(st.f, b);
        a.uu[x] = st.u;
        const uint64_t inflight = (uint64_t)(P - i) < cs.n_b ? (uint64_t)(P - i) : cs.n_b;
        const StageMem sm = stage_memory(v, k.tpi, k.mi, k.rc, nb, e, hd, inflight);
        if (sm.mem + h->reserved[g] > h->capacity[g]) atomicOr(&cs.oom_stage[i], 1ull << g);
        if (g == 0) cs.params[i] = sm.params;
    }
    for (uint32_t x = tid; x < cs.n_lower * P * T; x += PLAN_THREADS) {      // the same stages at the smaller degrees
        const uint32_t j = x / (P * T), i = (x / T) % P, g = x % T;
        const uint32_t nb = base + (i < extra ? 1u : 0u);
        const bool e = (i == 0) && h->has_embed, hd = (i == P - 1) && h->has_head;
        const uint64_t inflight = (uint64_t)(P - i) < cs.n_b ? (uint64_t)(P - i) : cs.n_b;
        const StageMem sm = stage_memory(v, cs.lower_tpi[j], k.mi, k.rc, nb, e, hd, inflight);
        if (sm.mem + h->reserved[g] > h->capacity[g]) atomicOr(&cs.oom_stage[i], 1ull << (8 * (j + 1) + g));
    }
    for (uint32_t d = tid; d < R; d += PLAN_THREADS) {
        a.availv[d] = pp.avail[d];
        a.tz[d] = (d % T) | ((d / T) << 8);
    }
    __syncthreads();

    // phase B: boundary tables and per-(segment, digit) records
    const double msg = (double)v.p2p[k.mi];
    const uint64_t xbytes = 2 * cs.n_b * (uint64_t)k.D * v.p2p[k.mi];
    for (uint32_t x = tid; x < R * R; x += PLAN_THREADS) {
        const uint32_t dn = x / R, d = x % R;      // [next][this]
        a.c2x[x] = mul_rn(2.0, boundary_time(v, d % T, d / T, tp, dn % T, dn / T, tp, k.D, msg));
    }
    for (uint32_t x = tid; x < R * Z; x += PLAN_THREADS) {
        const uint32_t dn = x / Z, z = x % Z, zn = dn / T;      // [next digit][this zone]
        a.commx[x] = (z != zn) ? mul_rn((double)xbytes, v.egress[z * Z + zn]) : 0.0;
    }
    for (uint32_t x = tid; x < k.nseg * T; x += PLAN_THREADS) {
        const uint32_t s = x / T, g = x % T;
        a.fb_last[x] = a.fb[(cs.seg_a[s + 1] - 1) * T + g];
    }
    for (uint32_t x = tid; x < k.nseg * R; x += PLAN_THREADS) {
        const uint32_t s = x / R, d = x % R, g = d % T, z = d / T;
        const uint32_t sa = cs.seg_a[s], se = cs.seg_a[s + 1];
        // the last stage of a non-final segment talks to the next segment: its t is not in the runs
        const uint32_t t_end = (s + 1 < k.nseg) ? se - 1 : se;
        const double c2self = mul_rn(2.0, boundary_time(v, g, z, tp, g, z, tp, k.D, msg));
        SegRec r;
        for (int q = 0; q < N_RUNS; ++q) r.v[q] = 0.0;
        double tm = 0.0, sy = 0.0, up = 0.0;
        bool oom = false;
        unsigned long long oom_bits = 0;
        for (uint32_t i = sa; i < se; ++i) {
            oom_bits |= cs.oom_stage[i];
            if (i < t_end) {
                const double fbi = a.fb[i * T + g];
                const double t = (i + 1 < P) ? add_rn(fbi, c2self) : fbi;
                r.v[run_of(h, P, extra, i)] = t;
                tm = dmax(tm, t);
            }
            if (k.D > 1) sy = dmax(sy, allreduce_time(v, g, d, tp, k.D, cs.params[i], cs.ar_steps, cs.ar_coef));
            up = dmax(up, a.uu[i * T + g]);
            oom |= (cs.oom_stage[i] >> g) & 1u;
        }
        r.tmax = tm;
        r.sync = sy;
        r.upd = up;
        r.rate = mul_rn((double)(k.D * tp), v.price_s[d]);
        a.rec[x] = r;
        if (oom) atomicOr(reinterpret_cast<unsigned long long*>(&cs.oom_mask[s]), 1ull << d);
        for (uint32_t j = 0; j < cs.n_lower; ++j)
            if (!((oom_bits >> (8 * (j + 1) + g)) & 1ull))
                atomicOr(reinterpret_cast<unsigned long long*>(&cs.lower_fit[j][s]), 1ull << d);
    }
    __syncthreads();                   // the memory masks and the records are complete
    if constexpr (SWEEP) {
        const SegRec* recs = a.rec + (k.nseg - 1) * R;
        bool alike = true;             // the last segment's records of a type are the same bits in every zone
        for (uint32_t d = tid; d < R; d += PLAN_THREADS) {
            const SegRec &x = recs[d], &y = recs[d % T];
            for (int q = 0; q < N_RUNS; ++q) alike &= x.v[q] == y.v[q];
            alike &= x.tmax == y.tmax && x.sync == y.sync && x.upd == y.upd && x.rate == y.rate;
        }
        const int all = __syncthreads_and(alike);
        if (tid == 0) cs.by_zone = all && zones_pay(Z, cs.seg_a[k.nseg] - cs.seg_a[k.nseg - 1]) ? 1u : 0u;
    }
    if (tid < 32) {
        const uint32_t last = k.nseg - 1;
        const uint32_t need_last = cs.need[last];
        const uint32_t a_lo = __ballot_sync(FULL, tid < R && need_last <= a.availv[tid < R ? tid : 0]);
        const uint32_t a_hi = __ballot_sync(FULL, tid + 32 < R && need_last <= a.availv[tid + 32 < R ? tid + 32 : 0]);
        if (tid == 0) {
            cs.avail_last = ((uint64_t)a_hi << 32) | a_lo;
            cs.whole = cs.flat_base >= pp.flat_lo && cs.flat_base + cs.n_items * R <= pp.flat_hi;
        }
        if (pp.live_mode) {
            // usable digits per segment (valid type, fits in memory): only prefixes made of them are
            // enumerated; lane d places digit d (and d + 32) at its rank among the set bits
            const uint64_t full = R == 64 ? ~0ull : ((1ull << R) - 1);
            uint64_t live = 1;
            for (uint32_t sgm = 0; sgm < k.nseg; ++sgm) {
                const uint64_t good = full & ~cs.invalid_mask & ~cs.oom_mask[sgm];
                const uint32_t g_lo = (uint32_t)good, g_hi = (uint32_t)(good >> 32);
                const uint32_t below = (1u << tid) - 1u;
                if ((g_lo >> tid) & 1u) cs.good_list[sgm][__popc(g_lo & below)] = (uint8_t)tid;
                if ((g_hi >> tid) & 1u) cs.good_list[sgm][__popc(g_lo) + __popc(g_hi & below)] = (uint8_t)(tid + 32);
                const uint32_t n = __popcll(good);
                if (tid == 0) {
                    cs.g_cnt[sgm] = n;
                    cs.g_magic[sgm] = n > 1 ? (uint32_t)(0x100000000ull / n) + 1u : 0u;
                }
                if (sgm + 1 < k.nseg) live *= n;
            }
            if (tid == 0) cs.live_items = live;
        }
        if (tid == 0) cs.packed = pp.live_mode;
    }
    __syncthreads();
}

// The tables of configuration `c` from the cache instead of building them: two straight copies, then the availability mask
// of the last segment, which is the only part that follows the snapshot, by the warp that copied the scalars.  Called by the
// whole block; starts and ends synchronised.  `a.availv` holds the snapshot already.  (Bringing the next record into shared
// memory by a bulk copy while a configuration is searched, with the claims of chunks a turn ahead, made searches 2 to 9 %
// slower: what has to be worked out for it sits on the path that every warp waits for.)
static __device__ void load_config(const PlanParams& pp, CfgShared& cs, CfgArrays& a, uint32_t R, uint32_t c) {
    const uint32_t tid = threadIdx.x;
    const uint4* src = pp.cfg_cache + (size_t)c * (pp.cache_head16 + pp.cache_arr16);
    const CfgShared& rec = *reinterpret_cast<const CfgShared*>(src);                       // (its head)
    uint32_t need_last = 0;
    if (tid < 32) need_last = rec.need_last;
    __syncthreads();                                       // the old tables are not used any more
    for (uint32_t x = tid; x < pp.cache_head16; x += PLAN_THREADS) reinterpret_cast<uint4*>(&cs)[x] = src[x];
    for (uint32_t x = tid; x < pp.cache_arr16; x += PLAN_THREADS) reinterpret_cast<uint4*>(a.rec)[x] = src[pp.cache_head16 + x];
    if (tid < 32) {
        const uint32_t a_lo = __ballot_sync(FULL, tid < R && need_last <= a.availv[tid < R ? tid : 0]);
        const uint32_t a_hi = __ballot_sync(FULL, tid + 32 < R && need_last <= a.availv[tid + 32 < R ? tid + 32 : 0]);
        __syncwarp();
        if (tid == 0) {
            cs.avail_last = ((uint64_t)a_hi << 32) | a_lo;
            cs.whole = rec.flat_base >= pp.flat_lo && rec.flat_base + rec.n_items * R <= pp.flat_hi;
            cs.packed = cs.valid ? pp.live_mode : 0u;      // (this warp copied `valid`, and `packed`, which is replaced)
            cs.cur_config = c;
        }
    }
    __syncthreads();
}
static_assert(offsetof(CfgShared, packed) < 32 * 16 && offsetof(CfgShared, valid) < 32 * 16, "copied by warp 0");

// The configuration of chunk `ch`: the last of the n whose first chunk is not beyond it.  By a whole warp, 32 offsets at a
// time (thread by thread a binary search waits for its loads one after another).
__device__ __forceinline__ uint32_t find_config(const uint32_t* chunk_start, uint32_t n, uint32_t ch, uint32_t lane) {
    uint32_t lo = 0, span = n;
    while (span > 1) {
        const uint32_t step = (span + 31) / 32, at = lane * step;
        const uint32_t below = __popc(__ballot_sync(FULL, at < span && chunk_start[lo + (at < span ? at : 0)] <= ch));
        const uint32_t skip = (below - 1) * step;          // the first offset of the span never lies beyond ch
        lo += skip;
        span = min(step, span - skip);
    }
    return lo;
}

__device__ __forceinline__ uint64_t warp_or64(uint64_t x) {
    const uint32_t lo = __reduce_or_sync(FULL, (uint32_t)x);
    const uint32_t hi = __reduce_or_sync(FULL, (uint32_t)(x >> 32));
    return ((uint64_t)hi << 32) | lo;
}

struct Counters {
    uint32_t invalid, oom, over_avail, over_constr, feasible, total, pruned;
    double min_cost;
    double cfg_best;     // best feasible score seen in the current configuration
};

// Hand the block's best feasible score of configuration `c` to the per-configuration table (positive
// doubles order like their bit patterns) and start over.
__device__ __forceinline__ void flush_cfg_best(const PlanParams& pp, Counters& cnt, uint32_t c, uint32_t lane) {
    unsigned long long b = (unsigned long long)__double_as_longlong(cnt.cfg_best);
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        const unsigned long long other = __shfl_xor_sync(FULL, b, o);
        b = other < b ? other : b;
    }
    if (lane == 0 && b < (unsigned long long)__double_as_longlong(make_inf())) atomicMin(&pp.cfg_best[c], b);
    cnt.cfg_best = make_inf();
}

// Add a warp's per-thread counters to the block's 64-bit sums and clear them.
__device__ __forceinline__ void flush_counters(CfgShared& cs, Counters& cnt, uint32_t lane) {
    uint32_t* vals[7] = {&cnt.total, &cnt.invalid, &cnt.oom, &cnt.over_avail, &cnt.over_constr, &cnt.feasible,
                         &cnt.pruned};
#pragma unroll
    for (int j = 0; j < 7; ++j) {
        unsigned long long s = *vals[j];
#pragma unroll
        for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(FULL, s, o);
        if (lane == 0 && s) atomicAdd(&cs.stat[j], s);
        *vals[j] = 0;
    }
}

// The binary32 screen's counterparts of the arithmetic helpers (no NaN occurs).
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float dmax(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ void keep_min(double& least, double x, bool good) { least = (good && x < least) ? x : least; }
__device__ __forceinline__ void keep_min(float& least, float x, bool good) { least = fminf(least, good ? x : least); }

// acc + v if the (warp-uniform) condition holds: a predicated addition, where the compiler would add and select.
__device__ __forceinline__ void add_if(double& acc, double v, bool yes) {
    asm("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p add.rn.f64 %0, %0, %1;\n\t}" : "+d"(acc) : "d"(v), "r"((uint32_t)yes));
}
__device__ __forceinline__ void add_if(float& acc, float v, bool yes) {
    asm("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p add.rn.f32 %0, %0, %1;\n\t}" : "+f"(acc) : "f"(v), "r"((uint32_t)yes));
}
// acc + v + v + ... (n times, n warp-uniform), one rounding per addition: the stage-by-stage sum of a run.  Runs are
// mostly short: the first four additions are straight code.
template <typename F>
__device__ __forceinline__ F add_n(F acc, F v, uint32_t n) {
#pragma unroll
    for (uint32_t j = 0; j < 4; ++j) add_if(acc, v, j < n);
#pragma unroll 1
    for (uint32_t j = 4; j < n; ++j) acc = add_rn(acc, v);
    return acc;
}

// The walk over the last segment's digit is written once for binary64 (F = double) and for the binary32 screen
// (F = float, from the rounded tables).
template <typename F> struct RecOf;
template <> struct RecOf<double> { using type = SegRec; };
template <> struct RecOf<float> { using type = SegRec32; };

// What a lane carries from its prefix into the walk over the last segment's digit.
template <typename F>
struct ItemState {
    F acc, mx, sy, up, rate, cc;         // running sum / maxima / price rate / transfer cost of the prefix
    F fb_b;                              // f+b of the prefix's last stage (its message goes to the last digit)
    uint64_t ok, walk;                   // per last digit: feasible for this lane / worth visiting for the warp
    const typename RecOf<F>::type* recs; // records of the last segment
    const F* c2x_col;                    // c2x[.][d_prev]
    const F* comm_col;                   // commx[.][z_prev]
};

// Time and cost of the W candidates that extend item `it` with last digits d .. d+W-1, evaluated
// side by side (W independent dependency chains; the stage loops run once for all of them).
template <int NSEG, int N2, int W, typename F>
__device__ __forceinline__ void eval_candidates(const CfgShared& cs, const ItemState<F>& it, uint32_t Z, uint32_t R,
                                                uint32_t d, F nb, F (&t_iter)[W], F (&cost)[W]) {
    constexpr uint32_t last = NSEG - 1;
    const typename RecOf<F>::type* rc = it.recs + d;
    F t_sum[W], t_max[W], c_comm[W], r[W];
#pragma unroll
    for (int w = 0; w < W; ++w) {
        t_sum[w] = it.acc; t_max[w] = it.mx; c_comm[w] = it.cc; r[w] = it.rate;
        if (NSEG > 1) {                                   // last stage of the prefix sends to digit d + w
            const F tb = add_rn(it.fb_b, it.c2x_col[(d + w) * R]);
            t_sum[w] = add_rn(t_sum[w], tb);
            t_max[w] = dmax(t_max[w], tb);
            c_comm[w] = add_rn(c_comm[w], it.comm_col[(d + w) * Z]);
        }
    }
    // the segment's stages in order: [stage 0] [stages with an extra block] [plain stages] [final stage];
    // the price-rate sum takes one term per stage alongside
#define SAILOR_STAGE(RUN)                                                          \
    _Pragma("unroll") for (int w = 0; w < W; ++w) {                                \
        t_sum[w] = add_rn(t_sum[w], rc[w].v[RUN]);                                 \
        r[w] = add_rn(r[w], rc[w].rate);                                           \
    }
    if (N2 >= 0) {
#pragma unroll
        for (int j = 0; j < N2; ++j) { SAILOR_STAGE(2) }
        SAILOR_STAGE(3)
    } else {
        const uint32_t n0 = cs.n_run[last][0], n1 = cs.n_run[last][1], n2 = cs.n_run[last][2], n3 = cs.n_run[last][3];
        if (n0) { SAILOR_STAGE(0) }
        for (uint32_t j = 0; j < n1; ++j) { SAILOR_STAGE(1) }
        uint32_t j = n2;
        for (; j >= 4; j -= 4) { SAILOR_STAGE(2) SAILOR_STAGE(2) SAILOR_STAGE(2) SAILOR_STAGE(2) }
        if (j & 2) { SAILOR_STAGE(2) SAILOR_STAGE(2) }
        if (j & 1) { SAILOR_STAGE(2) }
        if (n3) { SAILOR_STAGE(3) }
    }
#undef SAILOR_STAGE
#pragma unroll
    for (int w = 0; w < W; ++w) {
        t_max[w] = dmax(t_max[w], rc[w].tmax);
        const F t_pp = add_rn(t_sum[w], mul_rn(nb, t_max[w]));
        t_iter[w] = add_rn(add_rn(t_pp, dmax(it.sy, rc[w].sync)), dmax(it.up, rc[w].upd));
        cost[w] = add_rn(mul_rn(r[w], t_iter[w]), c_comm[w]);
    }
}

template <int OBJ, typename F>
__device__ __forceinline__ F score_of(F t_iter, F cost) {
    return OBJ == SAILOR_OBJ_MAX_THROUGHPUT ? t_iter : OBJ == SAILOR_OBJ_MIN_COST ? cost : mul_rn(t_iter, cost);
}

template <bool CONSTR>
__device__ __forceinline__ bool within(const PlanParams& pp, double budget, double t_iter, double cost) {
    bool good = true;
    if (CONSTR) {
        if (budget > 0.0) good &= !(cost > budget);
        if (pp.min_rate > 0.0) good &= !(1.0 / t_iter < pp.min_rate);
    }
    return good;
}

// Fast pass over the candidates of one item, several digits per step (independent dependency
// chains per thread): tracks the lane's best score, the feasible count and the cheapest cost.
// No votes, no list updates.  Tables are padded, so a step may read (and mask out) digits >= R.
template <int NSEG, int OBJ, bool CONSTR, int N2, typename F>
__device__ __forceinline__ void walk_fast(const PlanParams& pp, const CfgShared& cs, const ItemState<F>& it,
                                          uint32_t Z, uint32_t R, double budget, F& best, uint32_t& feas,
                                          F& min_cost) {
    const F nb = (F)cs.n_b;
    constexpr uint32_t U = PLAN_DIGITS_PER_STEP;
    for (uint32_t half = 0; half * 32 < R; ++half) {
        const uint32_t wm = (uint32_t)(it.walk >> (32 * half)), om = (uint32_t)(it.ok >> (32 * half));
        const uint32_t d_end = min(R - 32 * half, 32u);
        for (uint32_t dd = 0; dd < d_end; dd += U) {
            if (!((wm >> dd) & ((1u << U) - 1u))) continue;   // warp-uniform
            const uint32_t d = 32 * half + dd;
            F t[U], c[U];
            eval_candidates<NSEG, N2, (int)U>(cs, it, Z, R, d, nb, t, c);
#pragma unroll
            for (uint32_t u = 0; u < U; ++u) {
                const bool g = ((om >> (dd + u)) & 1u) && within<CONSTR>(pp, budget, t[u], c[u]);
                if (CONSTR) feas += (uint32_t)g;
                keep_min(min_cost, c[u], g);
                keep_min(best, score_of<OBJ>(t[u], c[u]), g);
            }
        }
    }
}

// The bulk of every space has four segments: call `walk` with the shape of the last one as a constant where it is a
// common one (N2 >= 0: that many plain stages, then the final stage, nothing else), which makes the candidate loop
// straight-line code; -1 is the general form.
template <int N> struct Shape { static constexpr int value = N; };
template <int NSEG, typename Walk>
__device__ __forceinline__ void by_shape(const CfgShared& cs, Walk walk) {
    if (NSEG == SAILOR_SEG_MAX && cs.n_run[3][0] == 0 && cs.n_run[3][1] == 0 && cs.n_run[3][3] == 1) {
        switch (cs.n_run[3][2]) {
            case 0: walk(Shape<0>()); return;
            case 1: walk(Shape<1>()); return;
            case 2: walk(Shape<2>()); return;
            case 3: walk(Shape<3>()); return;
            default: break;
        }
    }
    walk(Shape<-1>());
}

// ---- items without a feasible candidate, when every candidate's time and cost is asked for ----------------------
//
// SAILOR_FLAG_EVAL_ALL wants the time and the cost of every candidate formed, also of those that are invalid, out of
// memory or over the availability.  Where no lane of the warp has a feasible candidate (98 % of workload 5) nothing is
// selected from them, so no masks and no minima are formed; the values are only looked at for what non-negative tables
// nearly never give, a set sign bit (one three-input OR a candidate): a price rate of zero over an infinite time is a NaN,
// whose sign is set.  It is noted where nobody reads it, as the walk that selects passes over such a candidate too.
__device__ __forceinline__ void evaluated(uint32_t& signs, double t, double c) {
    signs |= (uint32_t)__double2hiint(t) | (uint32_t)__double2hiint(c);
}
__device__ __forceinline__ void evaluated(uint32_t& signs, float t, float c) { signs |= __float_as_uint(t) | __float_as_uint(c); }

// The candidates of W zones that are not the prefix's own and (OWN) of the one that is.  A digit is a (zone, type) pair:
// the message from the prefix, and with it the running sum, the maximum and the transfer cost up to the last segment,
// depend on the zone alone unless it is the prefix's own, so these heads are formed once per zone and kept in registers;
// a type's record is alike in all zones here (CfgShared::by_zone): it is read once for all of them, and the maxima over
// synchronisation and update times and the price-rate sum are formed once.  n_b x max(a, b) is taken as
// max(n_b x a, n_b x b): rounding is monotone, so these are the same bits; a transfer cost of zero is not added.  Every
// candidate still takes its own additions over the segment's stages, in stage order, and its own closing terms: the bits
// are those of eval_candidates.  N2 >= 0: the segment is N2 plain stages and the final stage (straight code); -1: any.
// Bound: issue slots (63 % busy) and the FP64 pipe (52 %): 6 + (stages of the segment) FP64 instructions a candidate
// against 14 + 2 x (stages) digit by digit.  Workload 5, 6.4e9 candidates: 13.89 -> 7.19 ms, 55.9 -> 26.4
// lane-instructions a candidate, about 7 of them what an item costs before its candidates (digits, masks, prefix sums).
template <int N2, int W, bool OWN, typename F>
__device__ __forceinline__ void evaluate_zones(const CfgShared& cs, const ItemState<F>& it, uint32_t T, uint32_t Z, uint32_t R,
                                               uint32_t z_own, uint32_t first, F nb, uint32_t& signs) {
    constexpr uint32_t last = SAILOR_SEG_MAX - 1;
    constexpr int S = W + (OWN ? 1 : 0);
    F hs[S], hm[S], hc[S];
    uint32_t dz[S];
    if (OWN) { dz[S - 1] = z_own * T; hc[S - 1] = it.cc; }
#pragma unroll
    for (int w = 0; w < W; ++w) {
        const uint32_t j = first + w;
        dz[w] = (j + (j >= z_own ? 1u : 0u)) * T;
        const F tb = add_rn(it.fb_b, it.c2x_col[dz[w] * R]);
        hs[w] = add_rn(it.acc, tb);
        hm[w] = mul_rn(nb, dmax(it.mx, tb));
        hc[w] = add_rn(it.cc, it.comm_col[dz[w] * Z]);
    }
    const F* own = it.c2x_col + z_own * T * R;
    // the last of four segments: stages with an extra block, plain stages, the final stage
    const uint32_t n1 = N2 >= 0 ? 0u : cs.n_run[last][1], n2 = N2 >= 0 ? (uint32_t)N2 : cs.n_run[last][2], n = n1 + n2 + 1;
#pragma unroll 1
    for (uint32_t g = 0; g < T; ++g) {
        const typename RecOf<F>::type* rc = it.recs + g;
        const F v1 = rc->v[1], v2 = rc->v[2], v3 = rc->v[3];
        if (OWN) {
            const F tb = add_rn(it.fb_b, own[g * R]);
            hs[S - 1] = add_rn(it.acc, tb);
            hm[S - 1] = mul_rn(nb, dmax(it.mx, tb));
        }
        F t_sum[S], r = it.rate;
        if (N2 >= 0) {
#pragma unroll
            for (int w = 0; w < S; ++w) {
                t_sum[w] = hs[w];
#pragma unroll
                for (int j = 0; j < N2; ++j) t_sum[w] = add_rn(t_sum[w], v2);
                t_sum[w] = add_rn(t_sum[w], v3);
            }
#pragma unroll
            for (int j = 0; j <= N2; ++j) r = add_rn(r, rc->rate);
        } else {
            const F v0 = n1 ? v1 : n2 ? v2 : v3;
#pragma unroll
            for (int w = 0; w < S; ++w) t_sum[w] = add_rn(hs[w], v0);
#pragma unroll 1
            for (uint32_t j = 1; j < n; ++j) {
                const F v = j < n1 ? v1 : j + 1 < n ? v2 : v3;
#pragma unroll
                for (int w = 0; w < S; ++w) t_sum[w] = add_rn(t_sum[w], v);
            }
            r = add_n(r, rc->rate, n);
        }
        const F tm = mul_rn(nb, rc->tmax), sy = dmax(it.sy, rc->sync), up = dmax(it.up, rc->upd);
#pragma unroll
        for (int w = 0; w < S; ++w) {
            const F t = add_rn(add_rn(add_rn(t_sum[w], dmax(hm[w], tm)), sy), up);
            evaluated(signs, t, add_rn(mul_rn(r, t), hc[w]));
        }
    }
}

// All candidates of an item of a four-segment configuration; `z_prev` is the zone the lane's prefix sends from.  Returns
// the values' sign bits (bit 31).
template <typename F>
__device__ __forceinline__ uint32_t evaluate_only(const CfgShared& cs, const ItemState<F>& it, uint32_t T, uint32_t Z, uint32_t R,
                                                  bool active, uint32_t z_prev) {
    constexpr int NSEG = SAILOR_SEG_MAX;
    const F nb = (F)cs.n_b;
    const uint32_t lanes = __ballot_sync(FULL, active);
    const uint32_t z_own = __shfl_sync(FULL, z_prev, lanes ? __ffs(lanes) - 1 : 0);
    uint32_t signs = 0;
    if (!cs.by_zone || __any_sync(FULL, active && z_prev != z_own)) {
        by_shape<NSEG>(cs, [&](auto shape) {
            constexpr uint32_t U = PLAN_DIGITS_PER_STEP;   // (the tables are padded)
            for (uint32_t d = 0; d < R; d += U) {
                F t[U], c[U];
                eval_candidates<NSEG, decltype(shape)::value, (int)U>(cs, it, Z, R, d, nb, t, c);
#pragma unroll
                for (uint32_t u = 0; u < U; ++u) evaluated(signs, t[u], c[u]);
            }
        });
        return signs;
    }
    const uint32_t group = zone_group(Z);                  // the first group takes the prefix's own zone along
    if (group == 7) by_shape<NSEG>(cs, [&](auto shape) { evaluate_zones<decltype(shape)::value, 7, true>(cs, it, T, Z, R, z_own, 0, nb, signs); });
    else by_shape<NSEG>(cs, [&](auto shape) { evaluate_zones<decltype(shape)::value, 4, true>(cs, it, T, Z, R, z_own, 0, nb, signs); });
    for (uint32_t j = group; j + 1 < Z; ++j) evaluate_zones<-1, 1, false>(cs, it, T, Z, R, z_own, j, nb, signs);
    return signs;
}

// Rare second pass over an item: the same arithmetic, one digit at a time, and every candidate that
// may enter the warp's top-k list is offered to it (warp-synchronous).  Nothing is counted.
template <int NSEG, int OBJ, bool CONSTR, int N2>
__device__ __forceinline__ void walk_offer(const PlanParams& pp, const CfgShared& cs, const ItemState<double>& it,
                                           uint32_t Z, uint32_t R, double budget, uint64_t item_flat,
                                           WarpTopK& top, uint32_t lane, double outer_thr, double& min_cost) {
    const double nb = (double)cs.n_b;
    for (uint32_t d = 0; d < R; ++d) {
        if (!((it.walk >> d) & 1ull)) continue;               // warp-uniform
        double t1[1], c1[1];
        eval_candidates<NSEG, N2, 1>(cs, it, Z, R, d, nb, t1, c1);
        const double t = t1[0], c = c1[0];
        const bool good = ((it.ok >> d) & 1ull) && within<CONSTR>(pp, budget, t, c);
        const double score = score_of<OBJ>(t, c);
        min_cost = (good && c < min_cost) ? c : min_cost;      // (the fast pass of the exact search has seen it already)
        const bool want = good && score <= top.thr_score && score <= outer_thr;
        if (__any_sync(FULL, want)) top.offer(want, score, item_flat + d, pp.k, lane);
    }
}

// One item per lane: fixed prefix digits, walk the last segment's digit.
// EVAL: the time and cost of every candidate is wanted (SAILOR_FLAG_EVAL_ALL).
template <int NSEG, int OBJ, bool CONSTR, bool SCREEN, bool EVAL>
__device__ __forceinline__ void run_items(const PlanParams& pp, const CfgShared& cs, const CfgArrays& a,
                                          uint32_t T, uint32_t Z, uint32_t R, uint32_t q, bool active,
                                          double budget, WarpTopK& top, Counters& cnt, uint32_t lane) {
    constexpr uint32_t last = NSEG - 1;
    // ---- prefix: segments 0 .. NSEG-2 --------------------------------------------------------
    // EVAL: the digit of the prefix's last segment varies slowest over the items of a configuration, so that the lanes of
    // a warp nearly always send to the last segment from one zone (evaluate_only relies on it).  Otherwise, and in a
    // configuration that the range holds only a part of (its other chunks are not launched), the items are in flat order
    // and it varies fastest: the lanes' prefixes then share their first digits, and with them most of what makes a prefix fail.
    uint32_t dg[NSEG > 1 ? NSEG - 1 : 1];
    {
        uint32_t x = active ? q : 0;
        auto by_radix = [&]() {                            // the next digit over all digits
            const uint32_t y = R == 1 ? x : __umulhi(x, cs.magic), digit = x - y * R;      // x / R
            x = y;
            return digit;
        };
        if constexpr (EVAL && NSEG > 1) {                  // (every candidate is wanted: never packed)
            uint32_t o[NSEG - 1];
#pragma unroll
            for (int j = 0; j < NSEG - 2; ++j) o[j] = by_radix();
            o[NSEG - 2] = x;
            const bool whole = cs.whole;
#pragma unroll
            for (int s = 0; s < NSEG - 1; ++s) dg[s] = whole ? o[s == NSEG - 2 ? s : NSEG - 3 - s] : o[NSEG - 2 - s];
        } else if (NSEG > 1) {
#pragma unroll
            for (int s = NSEG - 2; s >= 0; --s) {
                if (cs.packed) {                           // mixed radix, over the usable digits of each segment
                    const uint32_t n = cs.g_cnt[s];
                    const uint32_t y = s == 0 ? 0u : n > 1 ? __umulhi(x, cs.g_magic[s]) : x;   // x / n
                    dg[s] = active ? cs.good_list[s][x - y * n] : 0u;
                    x = y;
                } else {
                    dg[s] = s == 0 ? x : by_radix();
                }
            }
        }
    }
    uint64_t item_flat = cs.flat_base;                     // the item's flat index follows from its digits
    {
        uint64_t pf = 0;
#pragma unroll
        for (int s = 0; s < NSEG - 1; ++s) pf = pf * R + dg[s];
        item_flat += pf * R;
    }
    // ---- status of the prefix: node validity and memory (integer work only) -------------------------
    bool p_inv = false, p_oom = false;
#pragma unroll
    for (int s = 0; s < NSEG - 1; ++s) {
        p_inv |= (cs.invalid_mask >> dg[s]) & 1;
        p_oom |= (cs.oom_mask[s] >> dg[s]) & 1;
    }
    // ---- which last digits are in range / valid / fit / available ------------------------------
    uint64_t range = R == 64 ? ~0ull : ((1ull << R) - 1);
    if (!cs.whole) {                                       // (a configuration that lies in the range as a whole skips this)
        if (item_flat < pp.flat_lo) {
            const uint64_t skip = pp.flat_lo - item_flat;
            range = skip >= 64 ? 0 : range & (~0ull << skip);
        }
        if (item_flat + R > pp.flat_hi) {
            const uint64_t keep = pp.flat_hi > item_flat ? pp.flat_hi - item_flat : 0;
            range = keep >= 64 ? range : range & ((1ull << keep) - 1);
        }
    }
    if (!active) range = 0;
    const uint64_t valid_l = range & ~cs.invalid_mask;
    uint64_t ok = 0;
    uint32_t n_ok = 0;
    // exactly one class per candidate: invalid, then oom, then over availability (packed: total, invalid and oom were
    // added in closed form)
    if (!cs.packed) {
        const uint32_t n_range = __popcll(range);
        cnt.total += n_range;
        if (p_inv) cnt.invalid += n_range;
        else {
            const uint32_t n_valid = __popcll(valid_l);
            cnt.invalid += n_range - n_valid;
            cnt.oom += p_oom ? n_valid : (uint32_t)__popcll(valid_l & cs.oom_mask[last]);
        }
    }
    if (__any_sync(FULL, active && !p_inv && !p_oom)) {    // no lane gets further in most warps of an unpruned search
        const uint64_t fit_l = p_inv || p_oom ? 0ull : valid_l & ~cs.oom_mask[last];
        uint64_t drop = 0;        // last digits at which the whole plan also fits with a smaller degree
        if (pp.min_tp_only)
            for (uint32_t j = 0; j < cs.n_lower; ++j) {
                bool pf = true;
#pragma unroll
                for (int s = 0; s < NSEG - 1; ++s) pf &= (cs.lower_fit[j][s] >> dg[s]) & 1;
                if (pf) drop |= cs.lower_fit[j][last];
            }
        const uint64_t good_l = fit_l & ~drop;
        cnt.pruned += __popcll(fit_l) - __popcll(good_l);
        bool p_over = false;
        uint32_t tot[NSEG > 1 ? NSEG - 1 : 1];             // demand of a prefix digit over the prefix
#pragma unroll
        for (int s = 0; s < NSEG - 1; ++s) {
            tot[s] = 0;
#pragma unroll
            for (int s2 = 0; s2 < NSEG - 1; ++s2) tot[s] += (dg[s2] == dg[s]) ? cs.need[s2] : 0u;
            p_over |= tot[s] > a.availv[dg[s]];
        }
        ok = p_over ? 0ull : good_l & cs.avail_last;
        if (__any_sync(FULL, ok != 0)) {
#pragma unroll
            for (int s = 0; s < NSEG - 1; ++s)             // a last digit equal to a prefix digit adds up
                if (cs.need[last] + tot[s] > a.availv[dg[s]]) ok &= ~(1ull << dg[s]);
        }
        n_ok = __popcll(ok);
        cnt.over_avail += __popcll(good_l) - n_ok;
        if (!CONSTR) cnt.feasible += n_ok;
    }

    // ---- the candidates -----------------------------------------------------------------------
    const bool none_ok = !__any_sync(FULL, n_ok != 0);     // then a warp goes on only because every candidate is wanted
    if (none_ok && !(EVAL && __any_sync(FULL, range != 0))) return;
    const uint64_t walk = warp_or64(EVAL ? range : ok);    // warp-uniform: skip dead digits
    // ---- running sums of the prefix, in stage order ---------------------------------------------
    double acc = 0.0, mx = 0.0, sy = 0.0, up = 0.0, rate = 0.0, cc = 0.0;
#pragma unroll
    for (int s = 0; s < NSEG - 1; ++s) {
        const uint32_t d = dg[s];
        const SegRec& rc = a.rec[s * R + d];
        // (run 0 is the stage with the embedding, so the first segment's; run 3 is the final stage)
        if (s == 0 && cs.n_run[0][0]) acc = add_rn(acc, rc.v[0]);
        if (cs.n_run[s][1]) acc = add_n(acc, rc.v[1], cs.n_run[s][1]);
        acc = add_n(acc, rc.v[2], cs.n_run[s][2]);
        mx = dmax(mx, rc.tmax);
        sy = dmax(sy, rc.sync);
        up = dmax(up, rc.upd);
        rate = add_n(rate, rc.rate, cs.seg_a[s + 1] - cs.seg_a[s]);
        if (s < NSEG - 2) {                               // the segment's last stage sends to the next prefix digit
            const uint32_t dn = dg[s + 1];
            const double tb = add_rn(a.fb_last[s * T + (a.tz[d] & 0xff)], a.c2x[dn * R + d]);
            acc = add_rn(acc, tb);
            mx = dmax(mx, tb);
            cc = add_rn(cc, a.commx[dn * Z + (a.tz[d] >> 8)]);
        }
    }
    ItemState<double> it;
    it.acc = acc; it.mx = mx; it.sy = sy; it.up = up; it.rate = rate; it.cc = cc;
    it.ok = ok;
    it.walk = walk;
    it.fb_b = 0.0;
    uint32_t d_prev = 0, z_prev = 0;
    if (NSEG > 1) {
        d_prev = dg[NSEG > 1 ? NSEG - 2 : 0];
        z_prev = a.tz[d_prev] >> 8;
        it.fb_b = a.fb_last[(NSEG > 1 ? NSEG - 2 : 0) * T + (a.tz[d_prev] & 0xff)];
    }
    it.recs = a.rec + last * R;
    it.c2x_col = a.c2x + d_prev;
    it.comm_col = a.commx + z_prev;

    if (SCREEN) {
        // binary32 first; the item is walked exactly only if it may hold a member of the top-k or the cheapest plan
        ItemState<float> s32;
        s32.acc = __double2float_rn(acc); s32.mx = __double2float_rn(mx); s32.sy = __double2float_rn(sy);
        s32.up = __double2float_rn(up); s32.rate = __double2float_rn(rate); s32.cc = __double2float_rn(cc);
        s32.fb_b = __double2float_rn(it.fb_b);
        s32.ok = ok;
        s32.walk = walk;
        s32.recs = a.rec32 + last * R;
        s32.c2x_col = a.c2x32 + d_prev;
        s32.comm_col = a.commx32 + z_prev;
        if (EVAL && NSEG == SAILOR_SEG_MAX && none_ok) {
            if ((int)evaluate_only(cs, s32, T, Z, R, active, z_prev) < 0) pp.ctrl->no_number = 1u;
            return;
        }
        const float f_inf = __int_as_float(0x7f800000);
        float best32 = f_inf, minc32 = f_inf;
        uint32_t none = 0;
        by_shape<NSEG>(cs, [&](auto shape) {
            walk_fast<NSEG, OBJ, false, decltype(shape)::value>(pp, cs, s32, Z, R, budget, best32, none, minc32);
        });
        const double outer_thr = __longlong_as_double((long long)*reinterpret_cast<const volatile unsigned long long*>(&cs.thr_bits));
        const double outer_minc = __longlong_as_double((long long)*reinterpret_cast<const volatile unsigned long long*>(&cs.minc_bits));
        const double thr = top.thr_score < outer_thr ? top.thr_score : outer_thr;
        const bool need = best32 < f_inf && ((double)best32 <= thr * (1.0 + SCREEN_BAND) || (double)minc32 <= outer_minc * (1.0 + SCREEN_BAND));
        if (__any_sync(FULL, need)) {
            const double before = top.thr_score, mc_before = cnt.min_cost;
            by_shape<NSEG>(cs, [&](auto shape) {
                walk_offer<NSEG, OBJ, CONSTR, decltype(shape)::value>(pp, cs, it, Z, R, budget, item_flat, top, lane, outer_thr, cnt.min_cost);
            });
            if (lane == 0 && top.thr_score < before)
                atomicMin(const_cast<unsigned long long*>(&cs.thr_bits), (unsigned long long)__double_as_longlong(top.thr_score));
            if (cnt.min_cost < mc_before)
                atomicMin(const_cast<unsigned long long*>(&cs.minc_bits), (unsigned long long)__double_as_longlong(cnt.min_cost));
        }
        return;
    }
    if (EVAL && NSEG == SAILOR_SEG_MAX && none_ok) {
        if ((int)evaluate_only(cs, it, T, Z, R, active, z_prev) < 0) pp.ctrl->no_number = 1u;
        return;
    }
    // fast pass: no votes, no list updates; each lane keeps its item's best score
    double best = make_inf();
    uint32_t feas = 0;
    by_shape<NSEG>(cs, [&](auto shape) {
        walk_fast<NSEG, OBJ, CONSTR, decltype(shape)::value>(pp, cs, it, Z, R, budget, best, feas, cnt.min_cost);
    });
    cnt.cfg_best = best < cnt.cfg_best ? best : cnt.cfg_best;
    if (CONSTR) {
        cnt.feasible += feas;
        cnt.over_constr += n_ok - feas;
    }
    // rare: some lane's item holds a candidate that may enter the warp's list; walk again and offer
    // (a candidate worse than the k-th best of ANY warp's list cannot be among the k best overall: the block keeps
    // the lowest such score its warps and the other blocks have reached; equal scores still pass, the list decides)
    const double outer_thr = __longlong_as_double((long long)*reinterpret_cast<const volatile unsigned long long*>(&cs.thr_bits));
    if (!pp.cost_only && __any_sync(FULL, best < make_inf() && best <= top.thr_score && best <= outer_thr)) {   // best == inf: no feasible candidate
        const double before = top.thr_score;
        by_shape<NSEG>(cs, [&](auto shape) {
            walk_offer<NSEG, OBJ, CONSTR, decltype(shape)::value>(pp, cs, it, Z, R, budget, item_flat, top, lane, outer_thr, cnt.min_cost);
        });
        if (lane == 0 && top.thr_score < before)
            atomicMin(const_cast<unsigned long long*>(&cs.thr_bits), (unsigned long long)__double_as_longlong(top.thr_score));
    }
}

// The k best of `n_lists` sorted lists of SAILOR_K_MAX slots (all k slots written, empty ones as (+inf, ~0)), merged by a
// whole block of NW warps into s_hits[0]; returns how many there are (at most k).  `sel` (SAILOR_K_MAX words) and `s_n`
// are scratch in shared memory.  Ends synchronised.
template <uint32_t NW>
__device__ __forceinline__ uint32_t merge_block_lists(const Hit* partial, uint32_t n_lists, uint32_t k, Hit (*s_hits)[SAILOR_K_MAX],
                                                      uint32_t* sel, uint32_t* s_n) {
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // The k best of all lists lie in the k lists with the best first elements: k elements (those heads) are at
    // least as good as the k-th best head, and a list whose head is worse holds nothing better than its head.
    // So: the k best heads first (one element per list, all loads in flight together), then only those lists.
    // (Other SMs wrote the lists: read them in L2.)
    auto load_hit = [&](uint32_t b, uint32_t slot, double& sc, uint64_t& fl) {
        const double2 raw = __ldcg(reinterpret_cast<const double2*>(&partial[(size_t)b * SAILOR_K_MAX + slot]));
        sc = raw.x;
        fl = (uint64_t)__double_as_longlong(raw.y);
    };
    constexpr uint32_t PER_WARP = (SAILOR_K_MAX + NW - 1) / NW;
    WarpTopK top;
    top.init();
    auto tree_merge = [&]() {          // the warps' lists into warp 0's, through shared memory
        s_hits[warp][lane].score = top.score;
        s_hits[warp][lane].flat = top.flat;
        __syncthreads();
        for (uint32_t step = 1; step < NW; step <<= 1) {
            if ((warp & (2 * step - 1)) == 0 && warp + step < NW) {
                top.merge_sorted(s_hits[warp + step][lane].score, s_hits[warp + step][lane].flat, k, lane);
                s_hits[warp][lane].score = top.score;
                s_hits[warp][lane].flat = top.flat;
            }
            __syncthreads();
        }
    };
    WarpTopK more;
    double hs[2];                                          // the heads of up to 64 * NW lists stay in registers
    uint64_t hf[2];
    const uint32_t rounds = (n_lists + 32 * NW - 1) / (32 * NW);
    for (uint32_t r = 0; r < rounds; ++r) {
        const uint32_t b = r * 32 * NW + tid;
        more.init();
        if (b < n_lists) load_hit(b, 0, more.score, more.flat);
        if (more.flat == ~0ull) more.score = make_inf();   // an empty list (only its first slot need be written)
        if (r == 0) { hs[0] = more.score; hf[0] = more.flat; }
        if (r == 1) { hs[1] = more.score; hf[1] = more.flat; }
        more.sort(k, lane);
        if (r == 0) top = more;
        else top.merge_sorted(more.score, more.flat, k, lane);
    }
    tree_merge();
    const double cut_s = s_hits[0][k - 1].score;           // the k-th best head (or (+inf, ~0): fewer than k lists hold anything)
    const uint64_t cut_f = s_hits[0][k - 1].flat;
    if (tid == 0) *s_n = 0;
    __syncthreads();
    for (uint32_t r = 0; r < rounds; ++r) {
        const uint32_t b = r * 32 * NW + tid;
        double h_s = make_inf();
        uint64_t h_f = ~0ull;
        if (r == 0) { h_s = hs[0]; h_f = hf[0]; }
        else if (r == 1) { h_s = hs[1]; h_f = hf[1]; }
        else if (b < n_lists) load_hit(b, 0, h_s, h_f);
        if (h_f != ~0ull && (h_s < cut_s || (h_s == cut_s && h_f <= cut_f))) sel[atomicAdd(s_n, 1u)] = b;
    }
    __syncthreads();
    top.init();
    const uint32_t n_sel = *s_n;                               // at most k
    double ls[PER_WARP];
    uint64_t lf[PER_WARP];
#pragma unroll
    for (uint32_t x = 0; x < PER_WARP; ++x) {                  // all loads in flight before the first merge
        const uint32_t y = warp + x * NW;
        ls[x] = make_inf();
        lf[x] = ~0ull;
        if (y < n_sel && lane < k) load_hit(sel[y], lane, ls[x], lf[x]);
    }
#pragma unroll
    for (uint32_t x = 0; x < PER_WARP; ++x)
        if (warp + x * NW < n_sel) top.merge_sorted(ls[x], lf[x], k, lane);
    __syncthreads();                                           // `sel` has been read by everyone
    tree_merge();
    if (warp == 0) {
        const bool have = lane < k && top.flat != ~0ull;
        const uint32_t n = __popc(__ballot_sync(FULL, have));
        if (lane == 0) *s_n = n;
    }
    __syncthreads();
    return *s_n;
}

// The result records of the `n` winners, side by side: a group of G lanes per winner, lane i of it taking stage i (then
// i + G, ...), G as large as lets every winner have a group.  Per-stage terms are formed side by side; the sums whose order is
// part of the result run over the lanes' terms in stage order (a stage or message that is not there adds zero), so the bits
// are those of simulate_runs.  Bound by latency: a thread alone waits for one table after another (9.4 us from decoding to the
// record for plans of up to 24 stages, 5.0 us by a warp); 32 winners of up to 48 stages four to a warp, one after the other:
// 19.5 us, side by side 8.  By the whole block.
__device__ __forceinline__ void write_results(const PlanParams& pp, const TabView& v, const Hit* hits, uint32_t n, sailor_result* results) {
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t G = 32;
    while (G > 1 && n > PLAN_WARPS * (32 / G)) G /= 2;
    const uint32_t mine = lane & (G - 1), group = lane / G, j = warp * (32 / G) + group;
    if (warp * (32 / G) >= n) return;
    const bool real = j < n;
    const Hit hit = hits[real ? j : n - 1];
    sailor_result* out = results + j;
    const TabHdr* h = v.h;
    const SpaceDesc& sp = pp.sp;
    const uint32_t T = h->T, Z = h->Z, R = h->R;
    // the sub-space (number of stages) that holds the index: lane j knows the size of the j-th
    const uint32_t per_p = sp.n_mbs * sp.n_tp * sp.n_rc * sp.n_d;
    uint64_t size = 0;
    if (lane < sp.n_p) size = (uint64_t)per_p * ipow64(R, nseg_of(sp.p_values[lane], sp.seg_max));
    uint64_t end = size;
#pragma unroll 1
    for (int o = 1; o < 32; o <<= 1) {
        const uint64_t up = __shfl_up_sync(FULL, end, o);
        if (lane >= (uint32_t)o) end += up;
    }
    uint32_t sub = 0;
#pragma unroll 1
    for (uint32_t q = 0; q < 32 / G; ++q) {
        const uint64_t flat = __shfl_sync(FULL, hit.flat, q * G);
        const uint32_t at = __ffs(__ballot_sync(FULL, lane < sp.n_p && flat < end)) - 1;
        if (group == q) sub = at;
    }
    const uint64_t rem = hit.flat - __shfl_sync(FULL, end - size, sub);
    const uint32_t nseg = nseg_of(sp.p_values[sub], sp.seg_max);
    const uint32_t block = (uint32_t)ipow64(R, nseg);       // candidates of a configuration: at most 64^4
    const uint32_t cfg = (uint32_t)(rem / block);
    uint32_t x = (uint32_t)(rem - (uint64_t)cfg * block), dg[SAILOR_SEG_MAX];
#pragma unroll
    for (int q = SAILOR_SEG_MAX - 1; q >= 0; --q) {
        dg[q] = 0;
        if ((uint32_t)q < nseg) { const uint32_t y = x / R; dg[q] = x - y * R; x = y; }
    }
    const Config k = config_of(sp, sub * per_p + cfg);
    const uint32_t P = k.P, D = k.D, mi = k.mi, tp = h->tp_values[k.tpi];
    uint32_t seg_end[SAILOR_SEG_MAX], gz[SAILOR_SEG_MAX];   // per segment: past its last stage; type | zone << 8
#pragma unroll
    for (uint32_t q = 0; q < SAILOR_SEG_MAX; ++q) {
        seg_end[q] = q < nseg ? ((q + 1) * P + nseg - 1) / nseg : P;
        gz[q] = dg[q] / T;
        gz[q] = (dg[q] - gz[q] * T) | gz[q] << 8;
    }
    auto of_stage = [&](uint32_t i, const uint32_t (&seg)[SAILOR_SEG_MAX]) {
        return i < seg_end[0] ? seg[0] : i < seg_end[1] ? seg[1] : i < seg_end[2] ? seg[2] : seg[3];
    };
    const uint64_t dm = (uint64_t)D * h->mbs_values[mi], n_b = h->gbs / dm;
    uint32_t status = (n_b * dm != h->gbs || !((h->heads_ok >> k.tpi) & 1u)) ? SAILOR_ST_INVALID : 0u;
#pragma unroll
    for (uint32_t q = 0; q < SAILOR_SEG_MAX; ++q) {         // GPUs of every (zone, type) used, over all segments that use it
        uint32_t stages = 0;
#pragma unroll
        for (uint32_t q2 = 0; q2 < SAILOR_SEG_MAX; ++q2)
            if (q2 < nseg && dg[q2] == dg[q]) stages += seg_end[q2] - (q2 ? seg_end[q2 - 1] : 0u);
        if (q < nseg && (uint64_t)stages * D * tp > pp.avail[dg[q]]) status |= SAILOR_ST_OVER_AVAIL;
    }
    const uint32_t base = h->n_blocks / P, extra = h->n_blocks - base * P;
    const double msg = (double)v.p2p[mi], steps = (double)(2 * (uint64_t)(D - 1)), coef = steps / (double)D;
    const double xbytes = (double)(2 * n_b * (uint64_t)D * v.p2p[mi]);
    double sum_t = 0.0, max_t = 0.0, max_sync = 0.0, max_u = 0.0, rate = 0.0, c_comm = 0.0;
    uint64_t peak = 0;
    const uint32_t P_most = __reduce_max_sync(FULL, P);
    for (uint32_t at = 0; at < P_most; at += G) {
        const uint32_t i = at + mine;
        double t = 0.0, gpu_rate = 0.0, comm = 0.0;
        bool crosses = false;
        if (i < P) {
            const uint32_t x_i = of_stage(i, gz), g = x_i & 0xff, z = x_i >> 8, d = z * T + g;
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
            peak = m > peak ? m : peak;
            if (D > 1) max_sync = dmax(max_sync, allreduce_bytes_time(v, d, (uint64_t)D * tp <= h->gpn[g], v.cmp_grad[ct], D, steps, coef));
            gpu_rate = mul_rn((double)(D * tp), v.price_s[d]);
            if (i + 1 < P) {
                const uint32_t x_n = of_stage(i + 1, gz), zn = x_n >> 8;
                t = add_rn(t, mul_rn(2.0, boundary_time(v, g, z, tp, x_n & 0xff, zn, tp, D, msg)));
                crosses = zn != z;
                if (crosses) comm = mul_rn(xbytes, v.egress[z * Z + zn]);
            }
            max_t = dmax(max_t, t);
        }
        const uint32_t m = P_most - at < G ? P_most - at : G;
        for (uint32_t l = 0; l < m; ++l) {                   // in stage order
            sum_t = add_rn(sum_t, __shfl_sync(FULL, t, l, G));
            rate = add_rn(rate, __shfl_sync(FULL, gpu_rate, l, G));
        }
        uint32_t some = __ballot_sync(FULL, crosses);        // the stages at which any of the warp's plans changes zones
        for (uint32_t o = 16; o >= G; o >>= 1) some |= some >> o;
        for (some &= G == 32 ? FULL : (1u << G) - 1u; some; some &= some - 1)
            c_comm = add_rn(c_comm, __shfl_sync(FULL, comm, __ffs(some) - 1, G));
    }
#pragma unroll 1
    for (uint32_t o = G / 2; o; o >>= 1) {
        max_t = dmax(max_t, __shfl_xor_sync(FULL, max_t, o));
        max_sync = dmax(max_sync, __shfl_xor_sync(FULL, max_sync, o));
        max_u = dmax(max_u, __shfl_xor_sync(FULL, max_u, o));
        const uint64_t other = __shfl_xor_sync(FULL, peak, o);
        peak = other > peak ? other : peak;
        status |= __shfl_xor_sync(FULL, status, o);
    }
    if (!real) return;
    const double t_iter = add_rn(add_rn(add_rn(sum_t, mul_rn((double)n_b, max_t)), max_sync), max_u);
    if (mine == 0) {
        out->flat = hit.flat;
        out->score = hit.score;
        out->t_iter = t_iter;
        out->cost = add_rn(mul_rn(rate, t_iter), c_comm);
        out->peak_mem = peak;
        out->status = status;
        out->_pad = 0;
    }
    for (uint32_t y = mine; y < sizeof(sailor_plan_rec) / 4; y += G) {      // the record word by word: header, then a run per segment
        uint32_t word = 0;
        if (y == 0) word = P | mi << 8 | k.rc << 16 | nseg << 24;
        else if (y == 1) word = D;
        else if (y - 2 < nseg) {
            const uint32_t q = y - 2, x_q = q == 0 ? gz[0] : q == 1 ? gz[1] : q == 2 ? gz[2] : gz[3];
            const uint32_t a = q == 0 ? 0u : q == 1 ? seg_end[0] : q == 2 ? seg_end[1] : seg_end[2];
            const uint32_t e = q == 0 ? seg_end[0] : q == 1 ? seg_end[1] : q == 2 ? seg_end[2] : seg_end[3];
            word = x_q | k.tpi << 16 | (e - a) << 24;
        }
        reinterpret_cast<uint32_t*>(&out->plan)[y] = word;
    }
}

// End of a pass, run by the one block that hands in its list last (no block waits for another: every block
// adds one to Ctrl::blocks_done after its list is written, and the block that reads gridDim.x - 1 knows all the
// lists are in memory).  Merges the blocks' lists, simulates the winners in full for the result records, copies
// the counters next to them, hands `factor x best cost` to a following pass, and puts the counters back to
// their starting values.  `v` is the block's own view of the static tables (already in shared memory); `s_hits`
// (PLAN_WARPS lists) and `s_cnt` (SAILOR_K_MAX words) are scratch in shared memory.
static __device__ __noinline__ void finish_pass(const PlanParams& pp, const TabView& v, Hit (*s_hits)[SAILOR_K_MAX],
                                         uint32_t* s_cnt, uint32_t* s_n, uint32_t n_partial) {
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (pp.cost_only) {
        // the cheapest-plan pass of a budget-factor search: all the next pass needs is factor x the cheapest feasible
        // cost, which every block has already folded into Ctrl::min_cost_bits (the same bits a full simulation of
        // that plan gives: one operation order everywhere)
        if (tid == 0) {
            volatile Ctrl* live = pp.ctrl;
            const bool any = live->stats[5] != 0;
            const double cheapest = __longlong_as_double((long long)live->min_cost_bits);
            pp.ctrl->budget = any ? mul_rn(pp.next_budget_factor, cheapest) : make_inf();
            Ctrl* c = pp.ctrl;
            c->work_counter = 0;
            for (int q = 0; q < 7; ++q) c->stats[q] = 0;
            c->wave_chunks = 0;
            c->n_cfg_evaluated = 0;
            c->min_cost_bits = COST_BITS_START;
            c->thr_bits = COST_BITS_START;
            c->n_found = 0;
        }
        return;
    }
    // The counters as they stand (every block's contribution is in: atomics, then its blocks_done increment), a lane of the last
    // warp per word; they are asked for now and looked at when the merge is done.
    constexpr uint32_t WORDS = sizeof(Ctrl) / 4;
    static_assert(WORDS <= 32, "a lane per word");
    volatile uint32_t* live = reinterpret_cast<volatile uint32_t*>(pp.ctrl);
    const bool counts = warp == PLAN_WARPS - 1 && lane < WORDS;
    uint32_t word = 0;
    if (counts) word = live[lane];
    const uint32_t n = merge_block_lists<PLAN_WARPS>(pp.partial, n_partial, pp.k, s_hits, s_cnt, s_n);
    if (counts) {                      // to the host, and back to their starting values; the budget stays for the next pass
        const uint32_t at = 4 * lane;
        const bool cost = at >= offsetof(Ctrl, min_cost_bits) && at < offsetof(Ctrl, min_cost_bits) + 16;   // and thr_bits
        if (at != offsetof(Ctrl, n_found)) reinterpret_cast<uint32_t*>(&pp.out->ctrl)[lane] = word;
        if (!(at >= offsetof(Ctrl, budget) && at < offsetof(Ctrl, budget) + 8) && at != offsetof(Ctrl, blocks_done))
            live[lane] = cost && (at & 4) ? (uint32_t)(COST_BITS_START >> 32) : 0u;
    }
    if (n) write_results(pp, v, s_hits[0], n, pp.out->results);     // the winners are simulated in full for the result records
    __syncthreads();
    if (tid == 0) {
        pp.out->ctrl.n_found = n;
        pp.out->span.end = device_ns();
        __threadfence_system();        // the host may be looking: everything above is there before the ticket is
        *const_cast<volatile uint64_t*>(&pp.out->ticket) = pp.ticket;
    }
}

// FUSED: the block that hands in its list last also ends the pass (one launch per pass: what small searches, bound
// by launch and hand-over latencies, want).  Not FUSED: the lists are left for finish_kernel (the call inside the
// kernel costs the candidate loop a few registers, which long searches would pay for in every iteration).
// SCREEN: candidates are evaluated in binary32 first (unconstrained searches; see SCREEN_BAND).
template <int OBJ, bool CONSTR, bool FUSED, bool EVAL, bool SCREEN = false>
__global__ void __launch_bounds__(PLAN_THREADS, SCREEN ? PLAN_SCREEN_BLOCKS : PLAN_MIN_BLOCKS) plan_kernel(const __grid_constant__ PlanParams pp) {
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ CfgShared cs;
    __shared__ Hit s_hits[PLAN_WARPS][SAILOR_K_MAX];

    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const TabHdr* gh = reinterpret_cast<const TabHdr*>(pp.blob);
    const uint32_t static_bytes = gh->static_bytes;
    if (pp.first && blockIdx.x == 0 && tid == 0) pp.out->span.start = device_ns();

    // stage the static tables: one bulk copy, bounded wait, plain-load fallback
    if (!bulk_load(dyn, pp.blob, static_bytes, &cs.mbar)) {
        if (tid == 0) atomicExch(&pp.ctrl->error, 1u);
        for (uint32_t x = tid; x < static_bytes / 16; x += PLAN_THREADS)
            reinterpret_cast<uint4*>(dyn)[x] = reinterpret_cast<const uint4*>(pp.blob)[x];
        __syncthreads();
    }
    TabView v;
    v.bind(dyn, pp.blob);
    const uint32_t T = v.h->T, Z = v.h->Z, R = v.h->R;
    CfgArrays a;
    carve(dyn, static_bytes, pp.p_max, T, Z, a, pp.n_config, SCREEN);

    if (tid == 0) {
        cs.cur_config = 0xffffffffu;
        cs.minc_bits = COST_BITS_START;
        cs.magic = (uint32_t)(0x100000000ull / (gh->R ? gh->R : 1u)) + 1u;      // for x / R, see CfgShared
    }
    if (tid < 7) cs.stat[tid] = 0;
    if (tid == 7) cs.thr_bits = *reinterpret_cast<volatile unsigned long long*>(&pp.ctrl->thr_bits);
    // the padding digit of the tables is read (and masked out) by the two-digit steps: keep it finite
    for (uint32_t x = tid; x < PLAN_PAD * sizeof(SegRec) / 8; x += PLAN_THREADS)
        reinterpret_cast<double*>(a.rec + (size_t)SAILOR_SEG_MAX * R)[x] = 0.0;
    for (uint32_t x = tid; x < PLAN_PAD * R; x += PLAN_THREADS) a.c2x[(size_t)R * R + x] = 0.0;
    for (uint32_t x = tid; x < PLAN_PAD * Z; x += PLAN_THREADS) a.commx[(size_t)R * Z + x] = 0.0;
    for (uint32_t d = tid; d < R; d += PLAN_THREADS) {      // what does not depend on the configuration
        a.availv[d] = pp.avail[d];
        a.tz[d] = (d % T) | ((d / T) << 8);
    }
    // the chunk offsets are searched once per run of chunks and read once per chunk: keep a copy next to the tables
    // (the waves of a degree-order search rewrite them between launches, so every launch copies them afresh)
    const bool tab_local = pp.n_config < PLAN_CFG_SMEM;
    if (tab_local)
        for (uint32_t x = tid; x <= pp.n_config; x += PLAN_THREADS) a.chunk_tab[x] = pp.cfg_chunk_start[x];
    const uint32_t* chunk_start = tab_local ? a.chunk_tab : pp.cfg_chunk_start;
    WarpTopK top;
    top.init();
    if (pp.carry_lists && warp == 0) {     // a later wave of one search: go on from the list this block left behind
        if (lane < pp.partial_n[blockIdx.x]) {
            top.score = pp.partial[(size_t)blockIdx.x * SAILOR_K_MAX + lane].score;
            top.flat = pp.partial[(size_t)blockIdx.x * SAILOR_K_MAX + lane].flat;
        }
        top.thr_score = __shfl_sync(FULL, top.score, pp.k - 1);
        top.thr_flat = __shfl_sync(FULL, top.flat, pp.k - 1);
    }
    Counters cnt = {0, 0, 0, 0, 0, 0, 0, make_inf(), make_inf()};
    const double budget = pp.budget_from_ctrl ? pp.ctrl->budget : pp.budget;
    const uint32_t chunk_lo = pp.chunk_hi_dev ? 0u : pp.chunk_lo;
    const uint32_t chunk_hi = pp.chunk_hi_dev ? *pp.chunk_hi_dev : pp.chunk_hi;
    __syncthreads();

    uint32_t c = 0;     // configuration of the current chunk (monotone within a batch)
    bool first_round = true;
    for (;;) {
        if (tid == 0) {
            // every block starts with the chunk of its own number (no counter involved: small searches are bound by
            // such round trips); the rest is handed out by guided self-scheduling: long runs of consecutive chunks
            // first (a block then stays inside one configuration and changes its tables rarely), single chunks at
            // the end (even finish)
            const uint32_t n_chunks = chunk_hi - chunk_lo;
            if (first_round) {
                cs.next_chunk = chunk_lo + min(blockIdx.x, n_chunks);
                cs.batch_len = 1;
            } else if (n_chunks <= gridDim.x) {
                cs.next_chunk = chunk_hi;                    // every chunk had a block of its own
                cs.batch_len = 1;
            } else {
                const uint32_t rest = n_chunks - gridDim.x;
                const uint32_t seen = *reinterpret_cast<volatile unsigned int*>(&pp.ctrl->work_counter);
                const uint32_t left = seen < rest ? rest - seen : 0u;
                const uint32_t len = max(1u, left / (gridDim.x * 4u));
                const uint32_t got = atomicAdd(&pp.ctrl->work_counter, len);
                // trade thresholds with the other blocks in the meantime
                const unsigned long long theirs = *reinterpret_cast<volatile unsigned long long*>(&pp.ctrl->thr_bits);
                const unsigned long long ours = *reinterpret_cast<volatile unsigned long long*>(&cs.thr_bits);
                if (ours < theirs) atomicMin(&pp.ctrl->thr_bits, ours);
                else if (theirs < ours) atomicMin(&cs.thr_bits, theirs);
                cs.next_chunk = got < rest ? chunk_lo + gridDim.x + got : chunk_hi;
                cs.batch_len = len;
            }
        }
        first_round = false;
        __syncthreads();
        const uint32_t first = cs.next_chunk;
        if (first >= chunk_hi) break;
        const uint32_t end = min(first + cs.batch_len, chunk_hi);
        c = find_config(chunk_start, pp.n_config, first, lane);
        for (uint32_t ch = first; ch < end; ++ch) {
            while (ch >= chunk_start[c + 1]) ++c;
            if (cs.cur_config != c) {
                if (pp.cfg_best && cs.cur_config != 0xffffffffu) flush_cfg_best(pp, cnt, cs.cur_config, lane);
                if (pp.cfg_cache) load_config(pp, cs, a, R, c);
                else {
                    __syncthreads();
                    build_config<EVAL>(pp, v, cs, a, c);
                }
                if (SCREEN) round_config32(a, R, Z);
            }
            const uint32_t q = (ch - chunk_start[c]) * PLAN_THREADS + tid;    // < R^3 + 256 <= 2^18 + 256
            const bool active = q < (cs.packed ? cs.live_items : cs.n_items);
            if (!cs.valid) {
                // every candidate of the configuration is invalid; count those in range
                if (active) {
                    const uint64_t item_flat = cs.flat_base + (uint64_t)q * R;
                    const uint64_t lo = item_flat > pp.flat_lo ? item_flat : pp.flat_lo;
                    const uint64_t hi = item_flat + R < pp.flat_hi ? item_flat + R : pp.flat_hi;
                    const uint32_t n = hi > lo ? (uint32_t)(hi - lo) : 0u;
                    cnt.total += n;
                    cnt.invalid += n;
                }
                continue;
            }
            switch (cs.cfg.nseg) {
                case 1: run_items<1, OBJ, CONSTR, SCREEN, EVAL>(pp, cs, a, T, Z, R, q, active, budget, top, cnt, lane); break;
                case 2: run_items<2, OBJ, CONSTR, SCREEN, EVAL>(pp, cs, a, T, Z, R, q, active, budget, top, cnt, lane); break;
                case 3: run_items<3, OBJ, CONSTR, SCREEN, EVAL>(pp, cs, a, T, Z, R, q, active, budget, top, cnt, lane); break;
                default: run_items<4, OBJ, CONSTR, SCREEN, EVAL>(pp, cs, a, T, Z, R, q, active, budget, top, cnt, lane); break;
            }
        }
        // per-thread counters are 32 bits wide: hand them to the block's 64-bit sums in time
        if (__any_sync(FULL, cnt.total > (1u << 30))) flush_counters(cs, cnt, lane);
        __syncthreads();     // next_chunk and the tables are reused
    }

    // ---- block reduction: counters, then the warps' lists ---------------------------------------
    if (pp.cfg_best && cs.cur_config != 0xffffffffu) flush_cfg_best(pp, cnt, cs.cur_config, lane);
    flush_counters(cs, cnt, lane);
    {
        unsigned long long mc = (unsigned long long)__double_as_longlong(cnt.min_cost);   // positive: bits order
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            const unsigned long long other = __shfl_xor_sync(FULL, mc, o);
            mc = other < mc ? other : mc;
        }
        if (lane == 0) atomicMin(&pp.ctrl->min_cost_bits, mc);
    }
    s_hits[warp][lane].score = top.score;
    s_hits[warp][lane].flat = top.flat;
    __syncthreads();
    if (tid < 7 && cs.stat[tid]) atomicAdd(&pp.ctrl->stats[tid], cs.stat[tid]);
    if (warp == 0) {
        for (uint32_t w = 1; w < PLAN_WARPS; ++w) {
            if (s_hits[w][0].flat == ~0ull) continue;    // an empty list
            top.merge_sorted(s_hits[w][lane].score, s_hits[w][lane].flat, pp.k, lane);
        }
        const uint32_t n = __popc(__ballot_sync(FULL, top.flat != ~0ull && lane < pp.k));
        if (lane < pp.k) {
            pp.partial[(size_t)blockIdx.x * SAILOR_K_MAX + lane].score = top.score;
            pp.partial[(size_t)blockIdx.x * SAILOR_K_MAX + lane].flat = top.flat;
        }
        if (lane == 0) pp.partial_n[blockIdx.x] = n;
    }
    if (FUSED) {
        // hand the list in; the block that does so last ends the launch (and, in a pass's final launch, the pass)
        __threadfence();
        __syncthreads();
        if (tid == 0) {
            const unsigned int before = atomicAdd(&pp.ctrl->blocks_done, 1u);
            cs.next_chunk = (before == gridDim.x - 1) ? 1u : 0u;
            if (before == gridDim.x - 1) {
                pp.ctrl->blocks_done = 0;                    // the next launch counts from zero
                if (!pp.finish) pp.ctrl->work_counter = 0;   // (a finishing launch resets all counters below)
            }
        }
        __syncthreads();
        if (cs.next_chunk && pp.finish) {
            __threadfence();
            finish_pass(pp, v, s_hits, reinterpret_cast<uint32_t*>(a.rec), &cs.batch_len, gridDim.x);
        }
    }
}

using PlanKernel = void (*)(const PlanParams);

// The search kernels of one objective.  Each objective is compiled in a file of its own (sailor_plan_obj*.cu), side
// by side: the straight-line variants of the candidate loop are what the library takes longest to compile.
template <int OBJ, bool EVAL>
PlanKernel plan_kernel_with(bool constr, bool fused, bool screen) {
    if (screen) return plan_kernel<OBJ, false, false, EVAL, true>;     // unconstrained searches only; they end their pass in finish_kernel
    if (fused) return constr ? plan_kernel<OBJ, true, true, EVAL> : plan_kernel<OBJ, false, true, EVAL>;
    return constr ? plan_kernel<OBJ, true, false, EVAL> : plan_kernel<OBJ, false, false, EVAL>;
}
template <int OBJ>
PlanKernel plan_kernel_of(bool constr, bool fused, bool screen, bool eval_all) {
    return eval_all ? plan_kernel_with<OBJ, true>(constr, fused, screen) : plan_kernel_with<OBJ, false>(constr, fused, screen);
}

}  // namespace sailor
