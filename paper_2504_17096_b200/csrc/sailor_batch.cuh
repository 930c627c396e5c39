// Explicit batches of plan records (Sailor Sec. 4.3): the kernel behind sailor_simulate.
//
// A record costs 72 bytes in and 28 bytes out; what bounds the batch is the instructions a record takes (issue slots 64 %
// busy, HBM 12 %).  4.2e6 random records of workload 5 (19 stages, 4.3 runs, 5.7 pieces on average): 850 us -> 396 us
// (110 -> 67 warp-instructions a record).  What keeps them few:
//   - everything a stretch of equal stages needs (f + b, update time, memory with and without an in-flight microbatch)
//     sits in ONE 32-byte table entry (one memory sector, one load) per (stage make-up, GPU type, tp, mbs, rc), the gradient
//     bytes in a table per (stage make-up, tp), both formed once per context with the same functions and operation order as
//     a stage-by-stage walk;
//   - the doubled one-way message time of every link (inside a node, between nodes, between zones) is tabulated
//     per microbatch size, "fits into a node" as the largest D for which it does, so a stage boundary is one or two loads
//     and at most one maximum;
//   - a lane walks its record once, piece by piece: each run is unpacked and checked when the walk enters it, and leaves
//     behind what the plan has taken of its zone and type, for the rare run that repeats them;
//   - what is the same for all records are launch parameters (operands from the constant bank): kept in shared memory they
//     were held in registers, and the spills that followed pushed the table entries out of a small L1 (617 -> 495 us).
// The sums whose order of additions is part of the result (stage times, price rate, transfer cost) are still
// added one stage after the other, exactly as simulate_runs does, so both give the same bits.
#pragma once

#include "sailor_plan_kernels.cuh"

namespace sailor {

struct alignas(32) PieceRec {        // one per (composition, type, tp index, mbs index, rc): one 32-byte sector
    double fb;                       // f + b (+ f with recomputation) of a stage of this make-up
    double upd;                      // its update time
    uint64_t mem0r;                  // model + working bytes + the type's reserved bytes
    uint64_t mem1;                   // bytes kept per in-flight microbatch
};
static_assert(sizeof(PieceRec) == 32, "two 16-byte loads from one sector");

__host__ __device__ inline size_t piece_count(const TabHdr& h) {
    return (size_t)4 * h.chain_len * h.T * h.n_tp * h.n_mbs * 2;
}

// One thread per table entry; then the link tables (2 x one-way time per digit or zone pair and mbs index).
__global__ void batch_tables_kernel(unsigned char* blob) {
    TabView v;
    v.bind(blob, blob);
    const TabHdr* h = v.h;
    const size_t total = piece_count(*h);
    PieceRec* out = reinterpret_cast<PieceRec*>(blob + h->off_piece);
    for (size_t x = (size_t)blockIdx.x * blockDim.x + threadIdx.x; x < total; x += (size_t)gridDim.x * blockDim.x) {
        size_t y = x;
        const uint32_t rc = y % 2; y /= 2;
        const uint32_t mi = y % h->n_mbs; y /= h->n_mbs;
        const uint32_t tpi = y % h->n_tp; y /= h->n_tp;
        const uint32_t g = y % h->T; y /= h->T;
        const size_t comp = y;
        const uint32_t nb = (uint32_t)(comp % h->chain_len), eh = (uint32_t)(comp / h->chain_len);
        const bool e = eh & 2u, hd = eh & 1u;
        const StageTimes st = stage_times(v, g, tpi, mi, nb, e, hd);
        const double b = rc ? add_rn(st.b, st.f) : st.b;
        const StageMem one = stage_memory(v, tpi, mi, rc, nb, e, hd, 1);     // model + 1 * kept + work
        const StageMem zero = stage_memory(v, tpi, mi, rc, nb, e, hd, 0);    // model + work
        PieceRec r;
        r.fb = add_rn(st.f, b);
        r.upd = st.u;
        r.mem0r = zero.mem + h->reserved[g];
        r.mem1 = one.mem - zero.mem;
        out[x] = r;
    }
    double* intra2 = reinterpret_cast<double*>(blob + h->off_lnk_intra2);
    double* inter2 = reinterpret_cast<double*>(blob + h->off_lnk_inter2);
    double* zone2 = reinterpret_cast<double*>(blob + h->off_lnk_zone2);
    const uint32_t n_d = h->R * h->n_mbs, n_z = h->Z * h->Z * h->n_mbs;
    for (uint32_t x = blockIdx.x * blockDim.x + threadIdx.x; x < 2 * n_d + n_z; x += gridDim.x * blockDim.x) {
        if (x < 2 * n_d) {
            const uint32_t y = x < n_d ? x : x - n_d, d = y / h->n_mbs, mi = y % h->n_mbs;
            const double msg = (double)v.p2p[mi];
            if (x < n_d) intra2[y] = mul_rn(2.0, link_time(v.intra_a[d], v.intra_i[d], v.intra_p, d, msg));
            else inter2[y] = mul_rn(2.0, link_time(v.inter_a[d], v.inter_i[d], v.inter_p, d, msg));
        } else {
            const uint32_t y = x - 2 * n_d, zz = y / h->n_mbs, mi = y % h->n_mbs;
            zone2[y] = mul_rn(2.0, link_time(v.zone_a[zz], v.zone_i[zz], v.zone_p, zz, (double)v.p2p[mi]));
        }
    }
}

// What every lane of the batch kernel needs of the context: launch parameters, so that they are operands from the constant
// bank and take no registers.
struct BatchParams {
    const unsigned char* blob;
    const PieceRec* piece;
    const double *grad, *intra_p, *inter_p;          // global memory; grad: null when it is kept in shared memory
    uint64_t gbs;
    uint32_t T, Z, n_tp, n_mbs, chain_len, has_embed, has_head;
    uint32_t piece_stride;           // entries per composition: T * n_tp * n_mbs * 2
    uint32_t link_inter;             // entries of the link table inside a node (those between nodes follow)
    uint32_t s_grad, s_link, s_zone2;                // where these tables are in dynamic shared memory
    uint32_t smem;                   // its size
};

// What it keeps in shared memory of it (the tables whose size depends on the workload are in dynamic shared memory).
struct BatchConst {
    uint32_t mbs_values[SAILOR_MBS_MAX];
    uint64_t p2p[SAILOR_MBS_MAX];
    uint64_t cap[SAILOR_T_MAX];
    uint32_t blocks[SAILOR_P_MAX + 1];                           // per P: layers of a stage << 8 | stages with one more
    uint2 tpt[SAILOR_T_MAX * SAILOR_TP_MAX];                     // per (type, tp index): tp; largest D whose stage fits a node (0:
                                                                 // invalid) | largest D with which two such stages do << 16
    uint16_t pair[SAILOR_T_MAX * SAILOR_TP_MAX * SAILOR_TP_MAX]; // largest D with which two stages of these tp share a node
    uint32_t avail[R_MAX];
    double price_s[R_MAX];
    double2 ring[2 * R_MAX];                                     // alpha, 1 / bandwidth: between nodes, then inside one
    double egress[SAILOR_Z_MAX * SAILOR_Z_MAX];
};

constexpr unsigned int SIM_ERR_DEVICE = 1u, SIM_ERR_BAD_RECORD = 2u;   // bits of the batch kernels' error word
constexpr uint32_t REC_WORDS = sizeof(sailor_plan_rec) / 8;
constexpr uint32_t BATCH_WARPS = 19;                 // evaluating warps of a block; one more loads and orders
constexpr uint32_t BATCH_THREADS = 32 * (BATCH_WARPS + 1);
constexpr uint32_t BATCH_POOL = 768;                 // records ordered at a time, at most
constexpr uint32_t BATCH_RING = 2;                   // pools in shared memory
constexpr uint32_t BATCH_GRAD_SMEM = 24 * 1024;      // gradient tables of up to this size are kept in shared memory

struct alignas(16) BatchPool {
    uint64_t rec[BATCH_POOL * REC_WORDS + 2];        // (a batch that starts 8 bytes past a 16-byte line keeps that phase)
    uint16_t perm[BATCH_POOL];                       // records in the order of their work
};
struct BatchRing {
    BatchPool pool[BATCH_RING];
    uint32_t hist[256];
    uint16_t rank[BATCH_POOL];                       // of a record among those of its bin
    uint32_t run[BATCH_WARPS][SAILOR_RUN_MAX][32];   // runs of the records that a warp is evaluating
    uint64_t loaded[BATCH_RING], ready[BATCH_RING], drained[BATCH_RING];     // barriers
    uint32_t ticket;                                 // next group of records, counted over all pools of the block
};

inline BatchParams batch_params(const TabHdr& h, const unsigned char* blob) {
    BatchParams p;
    auto table = [&](size_t off) { return off ? reinterpret_cast<const double*>(blob + off) : nullptr; };
    p.blob = blob;
    p.piece = reinterpret_cast<const PieceRec*>(blob + h.off_piece);
    p.intra_p = table(h.off_intra_p); p.inter_p = table(h.off_inter_p);
    p.gbs = h.gbs;
    p.T = h.T; p.Z = h.Z; p.n_tp = h.n_tp; p.n_mbs = h.n_mbs; p.chain_len = h.chain_len;
    p.has_embed = h.has_embed; p.has_head = h.has_head;
    p.piece_stride = h.T * h.n_tp * h.n_mbs * 2;
    p.link_inter = h.R * h.n_mbs;
    uint32_t at = (uint32_t)((sizeof(BatchRing) + 15) / 16 * 16);
    const uint32_t grad_bytes = 4 * h.chain_len * h.n_tp * 8;
    const bool keep = grad_bytes <= BATCH_GRAD_SMEM;
    p.grad = keep ? nullptr : table(h.off_cmp_grad);
    p.s_grad = at; at += keep ? grad_bytes : 0u;
    p.s_link = at; at += 2 * h.R * h.n_mbs * 8;      // doubled message time per (digit, mbs): inside a node, then between nodes
    p.s_zone2 = at; at += h.Z * h.Z * h.n_mbs * 8;
    p.smem = at;
    return p;
}

struct BatchOut {
    double t_iter, cost;
    uint64_t peak;
    uint32_t status;
};

// The table entry of a stage make-up, one 32-byte load.
__device__ __forceinline__ PieceRec load_piece(const PieceRec* p) {
    PieceRec r;
    uint64_t fb, upd;
    asm("ld.global.nc.v4.b64 {%0, %1, %2, %3}, [%4];" : "=l"(fb), "=l"(upd), "=l"(r.mem0r), "=l"(r.mem1) : "l"(p));
    r.fb = __longlong_as_double((long long)fb);
    r.upd = __longlong_as_double((long long)upd);
    return r;
}

// One record: its first word and its runs (shared memory, 32 words apart; each is replaced by what the plan has taken of
// its zone and type when the walk has entered it).  Follows simulate_runs operation by operation where roundings are concerned.
// The stages are taken piece by piece (equal stages of one run): the first stage, then pieces that end with their run or
// where the extra layers run out, in one loop whose turn also moves on to the next run; then the final stage.
__device__ __forceinline__ BatchOut simulate_batch_record(const BatchParams& p, const BatchConst& k, const double* s_grad, const double* s_link,
                                                          const double* s_zone2, uint64_t w0, uint32_t* run) {
    BatchOut o;
    o.t_iter = o.cost = make_nan();
    o.peak = 0;
    o.status = SAILOR_ST_BAD_RECORD;
    const uint32_t P = (uint32_t)w0 & 0xff, mi = (uint32_t)(w0 >> 8) & 0xff;
    const uint32_t n_runs = (uint32_t)(w0 >> 24) & 0xff, D = (uint32_t)(w0 >> 32) & 0xffff;
    if (P < 1 || P > SAILOR_P_MAX || n_runs < 1 || n_runs > SAILOR_RUN_MAX || D < 1 || mi >= p.n_mbs) return o;
    const uint32_t mr = mi * 2 + (((uint32_t)(w0 >> 16) & 0xff) ? 1u : 0u);

    uint32_t status = 0;
    const uint64_t dm = (uint64_t)D * k.mbs_values[mi];
    uint64_t n_b;
    if (((p.gbs | dm) >> 32) == 0) {                        // the usual case: a 32-bit division
        const uint32_t q32 = (uint32_t)p.gbs / (uint32_t)dm;
        n_b = q32;
        if (q32 * (uint32_t)dm != (uint32_t)p.gbs) status |= SAILOR_ST_INVALID;
    } else {
        n_b = p.gbs / dm;
        if (n_b * dm != p.gbs) status |= SAILOR_ST_INVALID;
    }
    const uint32_t nb_cap = n_b > SAILOR_P_MAX ? SAILOR_P_MAX : (uint32_t)n_b;      // no stage holds more than P in flight
    const uint32_t base = k.blocks[P] >> 8, extra = k.blocks[P] & 0xffu;
    const double steps = (double)(2 * (D - 1));
    const double coef = D > 1 ? steps / (double)D : 0.0;    // ring all-reduce: 2(D-1)/D
    double sum_t = 0.0, max_t = 0.0, max_sync = 0.0, max_u = 0.0, rate = 0.0, c_comm = 0.0;
    uint64_t peak = 0;

    // the run that the walk is in (r: type, zone, tp index), and what follows from it
    uint32_t r, run_end = 0, q = 0, ent, seen_lo = 0, seen_hi = 0;
    uint32_t ring;
    double gpu_rate, c2_self;
    // Unpacks and checks run q before any table is read through it; GPUs taken per (zone, type) on the way.
    auto enter = [&]() -> bool {
        r = run[32 * q];
        const uint32_t g = r & 0xff, z = (r >> 8) & 0xff, tpi = (r >> 16) & 0xff, n = r >> 24;
        run_end += n;
        if (g >= p.T || z >= p.Z || tpi >= p.n_tp || n == 0 || run_end > P) return false;
        const uint32_t d = z * p.T + g, gt = g * SAILOR_TP_MAX + tpi;
        const uint2 tl = k.tpt[gt];
        if ((tl.y & 0xffffu) == 0) status |= SAILOR_ST_INVALID;
        uint64_t sum = (uint64_t)(D * n) * tl.x;            // GPUs this run takes of its (zone, type) ...
        const uint32_t bit = 1u << (d & 31u), seen = d < 32 ? seen_lo : seen_hi;
        if (seen & bit) {                                    // ... and earlier runs took of the same: the latest one says
            uint32_t q2 = q, r2;
#pragma unroll 1
            do {
                r2 = run[32 * --q2];
            } while ((r2 ^ r) & 0xffffu);
            sum += r2 >> 16;
        }
        if (d < 32) seen_lo |= bit; else seen_hi |= bit;
        if (sum > k.avail[d]) status |= SAILOR_ST_OVER_AVAIL;          // the total only grows from run to run
        run[32 * q] = (r & 0xffffu) | (sum < 0xffffull ? (uint32_t)sum : 0xffffu) << 16;   // (availability is 16 bits)
        gpu_rate = mul_rn((double)(D * tl.x), k.price_s[d]);
        const uint32_t lnk = d * p.n_mbs + mi;
        c2_self = s_link[D <= tl.y >> 16 ? lnk : lnk + p.link_inter];   // two neighbouring stages of the run
        ring = D <= (tl.y & 0xffffu) ? R_MAX + d : d;
        ent = (g * p.n_tp + tpi) * p.n_mbs * 2 + mr;         // entry within a composition
        return true;
    };
    // Order-free terms of a piece whose first stage is i; returns its f + b.
    auto piece = [&](uint32_t comp, uint32_t i) {
        const PieceRec pr = load_piece(p.piece + (size_t)(comp * p.piece_stride + ent));
        if (D > 1) {
            const uint32_t x = comp * p.n_tp + ((r >> 16) & 0xff);
            const double grad = p.grad ? __ldg(&p.grad[x]) : s_grad[x];
            const double volume = mul_rn(coef, grad);
            const double2 ab = k.ring[ring];
            double t = mul_rn(volume, ab.y);
            if (p.intra_p || p.inter_p) {
                const uint32_t g = r & 0xff, d = ((r >> 8) & 0xff) * p.T + g;
                const double* poly = ring >= R_MAX ? p.intra_p : p.inter_p;
                if (poly) t = volume / poly_bw(poly + 4 * d, grad / (double)D);
            }
            max_sync = dmax(max_sync, add_rn(t, mul_rn(steps, ab.x)));
        }
        const uint32_t left = P - i, inflight = left < nb_cap ? left : nb_cap;
        const uint64_t m = pr.mem0r + (uint64_t)inflight * pr.mem1;
        if (m > k.cap[r & 0xff]) status |= SAILOR_ST_OOM;
        peak = m > peak ? m : peak;
        max_u = dmax(max_u, pr.upd);
        return pr.fb;
    };

    if (!enter()) return o;
    uint32_t i = 0;
#pragma unroll 1
    while (i + 1 < P) {
        // the piece ends with its run, after the first stage, where the extra layers run out, before the final stage
        uint32_t end = run_end < P ? run_end : P - 1;
        if (i == 0) end = 1;
        else if (i < extra && extra < end) end = extra;
        const uint32_t comp = (i == 0 && p.has_embed ? 2 * p.chain_len : 0u) + base + (i < extra ? 1u : 0u);
        const double fb = piece(comp, i);
        const bool closes = end == run_end;                  // its last stage sends to the next run
        uint32_t n = end - i - (closes ? 1u : 0u);
        if (n) {
            const double t_self = add_rn(fb, c2_self);
            max_t = dmax(max_t, t_self);
            auto stage = [&]() { sum_t = add_rn(sum_t, t_self); rate = add_rn(rate, gpu_rate); };
            if (n & 1) stage();
            if (n & 2) { stage(); stage(); }
#pragma unroll 1
            for (n >>= 2; n; --n) { stage(); stage(); stage(); stage(); }
        }
        i = end;
        if (closes) {
            rate = add_rn(rate, gpu_rate);
            const uint32_t r1 = r;
            if (++q >= n_runs || !enter()) return o;
            const uint32_t g1 = r1 & 0xff, z1 = (r1 >> 8) & 0xff, g = r & 0xff, z = (r >> 8) & 0xff;
            const uint32_t lnk1 = (z1 * p.T + g1) * p.n_mbs + mi;
            double c2;
            if (z != z1) {
                c2 = s_zone2[(z1 * p.Z + z) * p.n_mbs + mi];
                c_comm = add_rn(c_comm, mul_rn((double)(2 * n_b * (uint64_t)D * k.p2p[mi]), k.egress[z1 * p.Z + z]));
            } else if (g == g1 && D <= k.pair[(g * SAILOR_TP_MAX + ((r1 >> 16) & 0xff)) * SAILOR_TP_MAX + ((r >> 16) & 0xff)]) {
                c2 = s_link[lnk1];
            } else {
                c2 = dmax(s_link[lnk1 + p.link_inter], s_link[(z * p.T + g) * p.n_mbs + mi + p.link_inter]);
            }
            const double t = add_rn(fb, c2);
            sum_t = add_rn(sum_t, t);
            max_t = dmax(max_t, t);
        }
    }
    if (q + 1 != n_runs || run_end != P) return o;           // runs left over, or too short for P stages
    {
        const uint32_t comp = ((i == 0 && p.has_embed ? 2u : 0u) + (p.has_head ? 1u : 0u)) * p.chain_len + base + (i < extra ? 1u : 0u);
        const double fb = piece(comp, i);                    // the final stage sends nothing
        sum_t = add_rn(sum_t, fb);
        max_t = dmax(max_t, fb);
        rate = add_rn(rate, gpu_rate);
    }
    o.peak = peak;
    o.status = status;
    if (status & SAILOR_ST_INVALID) return o;
    const double t_pp = add_rn(sum_t, mul_rn((double)n_b, max_t));
    o.t_iter = add_rn(add_rn(t_pp, max_sync), max_u);
    o.cost = add_rn(mul_rn(rate, o.t_iter), c_comm);
    return o;
}

__device__ __forceinline__ void bar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void bar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool bar_test(uint64_t* bar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return done != 0;
}
// Bounded wait of a whole warp; false when it ran out.
__device__ __forceinline__ bool bar_wait(uint64_t* bar, uint32_t parity) {
    bool done = false;
    for (uint32_t it = 0; it < WAIT_LIMIT && !done; ++it) done = bar_test(bar, parity);
    return __all_sync(FULL, done);
}

// Orders the `cnt` records of a pool by their work, most first: by run count (byte 3 of a record), then by stage count
// (byte 0).  A counting sort by one warp; any order gives the same results.
__device__ __forceinline__ void order_pool(const uint64_t* rec, uint16_t* perm, uint32_t* hist, uint16_t* rank, uint32_t cnt,
                                           uint32_t lane) {
    if (cnt <= 32) {                                           // one group
        if (lane < cnt) perm[lane] = (uint16_t)lane;
        __syncwarp();
        return;
    }
    auto bin_of = [&](uint32_t x) {
        const uint32_t w0 = (uint32_t)rec[x * REC_WORDS], P = w0 & 0xff, nr = w0 >> 24;
        return 255u - ((nr > 15u ? 15u : nr) * 16u + (P > 95u ? 15u : P / 6u));
    };
#pragma unroll
    for (int u = 0; u < 8; ++u) hist[lane + 32 * u] = 0;
    __syncwarp();
#pragma unroll 4
    for (uint32_t x = lane; x < cnt; x += 32) rank[x] = (uint16_t)atomicAdd(&hist[bin_of(x)], 1u);
    __syncwarp();
    uint32_t h8[8], sum = 0;                                   // exclusive scan of the 256 bins
#pragma unroll
    for (int u = 0; u < 8; ++u) { h8[u] = hist[lane * 8 + u]; sum += h8[u]; }
    uint32_t incl = sum;
#pragma unroll
    for (int x = 1; x < 32; x <<= 1) {
        const uint32_t up = __shfl_up_sync(FULL, incl, x);
        if (lane >= (uint32_t)x) incl += up;
    }
    uint32_t at = incl - sum;
#pragma unroll
    for (int u = 0; u < 8; ++u) { hist[lane * 8 + u] = at; at += h8[u]; }
    __syncwarp();
#pragma unroll 4
    for (uint32_t x = lane; x < cnt; x += 32) perm[hist[bin_of(x)] + rank[x]] = (uint16_t)x;
    __syncwarp();
}

// One block an SM; the batch goes through it in pools of `pool_size` records (a multiple of 32).  One warp brings pools into
// a ring in shared memory (one bulk copy each) and orders them by work; the others take groups of 32 similar records, longest
// first, copy their runs aside and hand the slot on before they evaluate them, so that nobody waits for the slowest group (an
// order of 512 records with barriers around it cost 3 of 11 stall cycles an instruction; slots held until evaluated: 626 us).
// 19 warps of 96 registers: 23 of 80 spill (461 us), 15 of 107 leave latencies open (461); pools of 768: 411 us when
// this was tried, 512 446, 640 419, 896 and 1 024 the same.  Results leave as four structure-of-arrays streams.
__global__ void __launch_bounds__(BATCH_THREADS, 1)
simulate_kernel(const __grid_constant__ BatchParams p, const uint16_t* __restrict__ avail,
                const sailor_plan_rec* __restrict__ plans, uint64_t n, uint32_t pool_size, uint32_t lanes, double* __restrict__ t_iter,
                uint64_t* __restrict__ peak_mem, double* __restrict__ cost, uint32_t* __restrict__ status, unsigned int* error,
                uint32_t report_bad) {                         // report_bad: set SIM_ERR_BAD_RECORD when a record is refused
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ BatchConst k;
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    BatchRing& ring = *reinterpret_cast<BatchRing*>(dyn);
    TabView v;
    v.bind(p.blob, p.blob);                                    // everything read through it comes from global memory
    const TabHdr* h = v.h;
    const uint64_t n_pools = (n + pool_size - 1) / pool_size;
    const uint32_t mine = n_pools > blockIdx.x ? (uint32_t)((n_pools - blockIdx.x - 1) / gridDim.x) + 1 : 0;     // pools of this block
    const uint32_t phase = (uint32_t)((uintptr_t)plans & 8u) / 8;           // words by which the records miss a 16-byte line

    // Pool `it` of this block into its slot: the part between 16-byte lines by a bulk copy, the rest by plain loads.
    auto load_pool = [&](uint32_t it) {                        // lane 0 of the loading warp
        const uint64_t first = (blockIdx.x + (uint64_t)it * gridDim.x) * pool_size;
        const uint32_t words = (uint32_t)(n - first < pool_size ? n - first : pool_size) * REC_WORDS;
        const uint32_t slot = it % BATCH_RING, bar = smem_u32(&ring.loaded[slot]);
        const uint64_t* src = reinterpret_cast<const uint64_t*>(plans) + first * REC_WORDS;
        uint64_t* dst = ring.pool[slot].rec + phase;
        const uint32_t even = (words - phase) & ~1u;
        if (phase) dst[0] = src[0];
        if (phase + even < words) dst[words - 1] = src[words - 1];
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(even * 8) : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"(smem_u32(dst + phase)), "l"(src + phase), "r"(even * 8), "r"(bar)
                     : "memory");
    };
    uint32_t issued = 0;
    if (tid == 32 * BATCH_WARPS) {
        for (uint32_t s = 0; s < BATCH_RING; ++s) {
            bar_init(&ring.loaded[s], 1);
            bar_init(&ring.ready[s], 1);
            bar_init(&ring.drained[s], pool_size / lanes);
        }
        ring.ticket = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        for (; issued < BATCH_RING && issued < mine; ++issued) load_pool(issued);
    }
    issued = mine < BATCH_RING ? mine : BATCH_RING;

    if (tid < SAILOR_MBS_MAX) { k.mbs_values[tid] = h->mbs_values[tid]; k.p2p[tid] = tid < h->n_mbs ? v.p2p[tid] : 0; }
    if (tid < SAILOR_T_MAX) k.cap[tid] = h->capacity[tid];
    if (tid >= 1 && tid <= SAILOR_P_MAX) { const uint32_t b = h->n_blocks / tid; k.blocks[tid] = b << 8 | (h->n_blocks - b * tid); }
    for (uint32_t x = tid; x < h->T * SAILOR_TP_MAX * SAILOR_TP_MAX; x += BATCH_THREADS) {
        const uint32_t t2 = x % SAILOR_TP_MAX, t1 = x / SAILOR_TP_MAX % SAILOR_TP_MAX, g = x / (SAILOR_TP_MAX * SAILOR_TP_MAX);
        if (t1 < h->n_tp && t2 < h->n_tp) {
            const uint32_t tp = h->tp_values[t1], both = tp + h->tp_values[t2], gpn = h->gpn[g];
            const uint32_t lim = both ? gpn / both : 0xffffu;
            k.pair[x] = (uint16_t)(lim < 0xffffu ? lim : 0xffffu);
            if (t1 == t2) {
                const uint32_t one = (h->heads_ok >> t1) & 1u ? gpn / tp : 0u;
                k.tpt[x / SAILOR_TP_MAX] = make_uint2(tp, (one < 0xffffu ? one : 0xffffu) | (uint32_t)k.pair[x] << 16);
            }
        }
    }
    for (uint32_t x = tid; x < h->R; x += BATCH_THREADS) {
        k.avail[x] = avail[x];
        k.price_s[x] = v.price_s[x];
        k.ring[x] = make_double2(v.inter_a[x], v.inter_i[x]);
        k.ring[R_MAX + x] = make_double2(v.intra_a[x], v.intra_i[x]);
    }
    for (uint32_t x = tid; x < h->Z * h->Z; x += BATCH_THREADS) k.egress[x] = v.egress[x];
    double* s_grad = reinterpret_cast<double*>(dyn + p.s_grad);
    double* s_link = reinterpret_cast<double*>(dyn + p.s_link);
    double* s_zone2 = reinterpret_cast<double*>(dyn + p.s_zone2);
    {
        const uint32_t n_link = h->R * h->n_mbs, n_zone = h->Z * h->Z * h->n_mbs, n_grad = 4 * h->chain_len * h->n_tp;
        for (uint32_t x = tid; x < n_link; x += BATCH_THREADS) {
            s_link[x] = reinterpret_cast<const double*>(p.blob + h->off_lnk_intra2)[x];
            s_link[n_link + x] = reinterpret_cast<const double*>(p.blob + h->off_lnk_inter2)[x];
        }
        for (uint32_t x = tid; x < n_zone; x += BATCH_THREADS) s_zone2[x] = reinterpret_cast<const double*>(p.blob + h->off_lnk_zone2)[x];
        if (!p.grad)
            for (uint32_t x = tid; x < n_grad; x += BATCH_THREADS) s_grad[x] = v.cmp_grad[x];
    }
    __syncthreads();

    if (warp == BATCH_WARPS) {                                 // loads and orders
        for (uint32_t it = 0; it < mine; ++it) {
            const uint32_t slot = it % BATCH_RING;
            // the next loads, as far as their slots have been drained (this pool's own has to be)
            while (issued < mine && issued < it + BATCH_RING) {
                const uint32_t s = issued % BATCH_RING, parity = (issued / BATCH_RING - 1) & 1u;
                if (issued > it && !__all_sync(FULL, bar_test(&ring.drained[s], parity))) break;
                if (issued == it && !bar_wait(&ring.drained[s], parity)) { if (lane == 0) atomicOr(error, SIM_ERR_DEVICE); return; }
                if (lane == 0) load_pool(issued);
                ++issued;
            }
            if (!bar_wait(&ring.loaded[slot], (it / BATCH_RING) & 1u)) { if (lane == 0) atomicOr(error, SIM_ERR_DEVICE); return; }
            const uint64_t first = (blockIdx.x + (uint64_t)it * gridDim.x) * pool_size;
            order_pool(ring.pool[slot].rec + phase, ring.pool[slot].perm, ring.hist, ring.rank, (uint32_t)(n - first < pool_size ? n - first : pool_size), lane);
            if (lane == 0) bar_arrive(&ring.ready[slot]);
        }
        return;
    }
    uint32_t* run = &ring.run[warp][0][lane];
    const uint32_t groups = pool_size / lanes;
    for (uint32_t it = 0, base = 0;;) {
        uint32_t grp = 0;
        if (lane == 0) grp = atomicAdd(&ring.ticket, 1u);
        grp = __shfl_sync(FULL, grp, 0);
        for (; grp - base >= groups; base += groups) ++it;
        if (it >= mine) break;
        const uint32_t slot = it % BATCH_RING;
        if (!bar_wait(&ring.ready[slot], (it / BATCH_RING) & 1u)) { if (lane == 0) atomicOr(error, SIM_ERR_DEVICE); return; }
        const uint64_t first = (blockIdx.x + (uint64_t)it * gridDim.x) * pool_size;
        const uint32_t x = (grp - base) * lanes + lane;
        const bool live = lane < lanes && first + x < n;
        // take the records along, so that the slot can be filled again before they are evaluated
        uint64_t w0 = 0;
        uint32_t r = 0;
        if (live) {
            r = ring.pool[slot].perm[x];
            const uint64_t* rec = ring.pool[slot].rec + phase + r * REC_WORDS;
            w0 = rec[0];
            const uint32_t pairs = ((uint32_t)(w0 >> 24) & 0xffu) + 1 >> 1;
            for (uint32_t y = 0; y < SAILOR_RUN_MAX / 2 && y < pairs; ++y) {
                const uint64_t two = rec[1 + y];
                run[64 * y] = (uint32_t)two;
                run[64 * y + 32] = (uint32_t)(two >> 32);
            }
        }
        __syncwarp();
        if (lane == 0) bar_arrive(&ring.drained[slot]);
        if (live) {
            const BatchOut o = simulate_batch_record(p, k, s_grad, s_link, s_zone2, w0, run);
            const uint64_t j = first + r;
            if (t_iter) __stcs(&t_iter[j], o.t_iter);
            if (peak_mem) __stcs(&peak_mem[j], o.peak);
            if (cost) __stcs(&cost[j], o.cost);
            if (status) __stcs(&status[j], o.status);
            if (report_bad && (o.status & SAILOR_ST_BAD_RECORD)) atomicOr(error, SIM_ERR_BAD_RECORD);
        }
        __syncwarp();
    }
}

}  // namespace sailor
