// Simulator for plans whose stages mix GPU types among their D replicas (Sailor Sec. 4.2, Sec. 4.3).
//
// Pipeline k runs on replica k of every stage, replicas being numbered group after group.  Two
// pipelines that use the same group in every stage are identical, so a plan has at most
// 1 + sum_i (groups_i - 1) different pipelines: one per interval between group boundaries (of any stage).
//
// One warp evaluates one plan, three times with its lanes on something else: first a lane per stage (reads the
// record, splits it into (stage, group) items), then a lane per item (memory, availability, synchronisation, update,
// price rate, and what a pipeline through the item needs: f + b, message time), then a lane per pipeline, which walks
// the stages with everything it needs in the warp's shared memory.  Every sum whose order of additions is part of the
// result is one lane's or runs over the lanes' terms in order (price rate: stage after stage, group after group;
// transfer cost: stage after stage).
// Bound: issue slots (67 % busy).  Random plans of workload 5 (mean 9.4 stages, 1.9 groups a stage, 5.4 pipelines), 2.6e5
// of them: 1 003 us with a lane per stage throughout and one pipeline after the other (2 960 warp-instructions a plan);
// 479 us this way (1 424).  Four blocks of 64 registers an SM: with 80 registers and three blocks 540 us.
#pragma once

#include "sailor_batch.cuh"

namespace sailor {

constexpr uint32_t MIX_FULL = 0xffffffffu;

// Largest of the warp's 64-bit values by two 32-bit warp maxima: the high words, then the low words of the lanes
// that hold the largest high word.
__device__ __forceinline__ uint64_t warp_max_u64(uint64_t x) {
    const uint32_t hi = (uint32_t)(x >> 32), lo = (uint32_t)x;
    const uint32_t mh = __reduce_max_sync(MIX_FULL, hi);
    const uint32_t ml = __reduce_max_sync(MIX_FULL, hi == mh ? lo : 0u);
    return (uint64_t)mh << 32 | ml;
}

// Largest of the warp's non-negative binary64 values (they order like their bit patterns).
__device__ __forceinline__ double warp_max_positive(double x) {
    return __longlong_as_double((long long)warp_max_u64((uint64_t)__double_as_longlong(x)));
}

// Smallest of the warp's positive binary64 values.
__device__ __forceinline__ double warp_min_positive(double x) {
    const uint64_t b = (uint64_t)__double_as_longlong(x);
    const uint32_t hi = (uint32_t)(b >> 32), lo = (uint32_t)b;
    const uint32_t mh = __reduce_min_sync(MIX_FULL, hi);
    const uint32_t ml = __reduce_min_sync(MIX_FULL, hi == mh ? lo : 0xffffffffu);
    return __longlong_as_double((long long)((uint64_t)mh << 32 | ml));
}

struct MixItem {                     // a group of a stage
    double fb;                       // f + b (+ f with recomputation) of the stage on the group's GPUs
    double inter2;                   // doubled message time between nodes
    uint32_t gpus, type;             // GPUs of the group (saturating), their type
};
struct alignas(16) MixStage {
    uint64_t ends;                   // replicas before the second, third, fourth group (16 bits each; 0xffff: there is none)
    double cross2;                   // doubled message time to the next stage when that is in another zone, else -1
    double grad;                     // gradient bytes of one worker: the ring moves the largest shard (smallest tp)
    uint32_t first;                  // first item | zone << 16 | groups << 24
    uint32_t comp;                   // layer make-up
};

// What a warp keeps in shared memory of the plan it evaluates (at most PM stages).
template <uint32_t PM>
struct alignas(16) MixScratch {
    MixItem item[SAILOR_MIX_GROUPS_MAX * PM];
    MixStage stage[PM];
    uint32_t cnt[R_MAX];             // GPUs taken per (zone, type)
    uint16_t start[(SAILOR_MIX_GROUPS_MAX - 1) * PM + 2];     // first replica of every interval
    uint8_t stage_of[SAILOR_MIX_GROUPS_MAX * PM];
};

// Every lane of the warp calls with the same record and gets the same result.
template <uint32_t PM>
__device__ inline SimOut simulate_mixed_warp(const TabView& v, const unsigned char* __restrict__ blob, const uint16_t* __restrict__ avail,
                                             const sailor_mixed_plan& r, MixScratch<PM>& s, uint32_t lane) {
    constexpr uint32_t TILES = PM / 32;
    static_assert(PM % 32 == 0 && SAILOR_MIX_GROUPS_MAX * PM < 65536, "a lane owns a stage of every tile");
    const TabHdr* h = v.h;
    SimOut o;
    o.t_iter = o.cost = make_nan();
    o.peak_mem = 0;
    o.status = SAILOR_ST_BAD_RECORD;
    const uint32_t P = r.P, D = r.D, mi = r.mbs_idx, rc = r.rc ? 1u : 0u, T = h->T, Z = h->Z, n_mbs = h->n_mbs;
    if (P < 1 || P > PM || D < 1 || mi >= n_mbs) return o;
    const PieceRec* piece = reinterpret_cast<const PieceRec*>(blob + h->off_piece);
    const double* intra2 = reinterpret_cast<const double*>(blob + h->off_lnk_intra2);
    const double* inter2 = reinterpret_cast<const double*>(blob + h->off_lnk_inter2);
    const double* zone2 = reinterpret_cast<const double*>(blob + h->off_lnk_zone2);

    // ---- a lane per stage: read, check, split into items ---------------------------------------
    uint32_t status = 0, n_items = 0;
    uint64_t n_b;
    {
        const uint64_t dm = (uint64_t)D * h->mbs_values[mi];
        if (((h->gbs | dm) >> 32) == 0) {                        // the usual case: a 32-bit division
            const uint32_t q32 = (uint32_t)h->gbs / (uint32_t)dm;
            n_b = q32;
            if (q32 * (uint32_t)dm != (uint32_t)h->gbs) status |= SAILOR_ST_INVALID;
        } else {
            n_b = h->gbs / dm;
            if (n_b * dm != h->gbs) status |= SAILOR_ST_INVALID;
        }
    }
    const uint32_t base = h->n_blocks / P, extra = h->n_blocks - base * P;
    uint64_t ends_of[TILES];
#pragma unroll
    for (uint32_t tl = 0; tl < TILES; ++tl) {
        if (tl && 32 * tl >= P) { ends_of[tl] = ~0ull; continue; }
        const uint32_t i = lane + 32 * tl;
        uint32_t zone = 0, ng = 0, gw[SAILOR_MIX_GROUPS_MAX] = {0, 0, 0, 0};
        bool bad = false;
        if (i < P) {
            const uint32_t* w = reinterpret_cast<const uint32_t*>(&r.stage[i]);      // five words a stage
            const uint32_t w0 = w[0];
            gw[0] = w[1]; gw[1] = w[2]; gw[2] = w[3]; gw[3] = w[4];
            zone = w0 & 0xff;
            ng = (w0 >> 8) & 0xff;
            bad = zone >= Z || ng < 1 || ng > SAILOR_MIX_GROUPS_MAX;
#pragma unroll
            for (uint32_t q = 0; q < SAILOR_MIX_GROUPS_MAX; ++q)
                bad = bad || (q < ng && ((gw[q] & 0xff) >= T || ((gw[q] >> 8) & 0xff) >= h->n_tp));
        }
        if (__any_sync(MIX_FULL, bad)) return o;
        uint32_t incl = ng;                                      // items of the stages before this one
#pragma unroll
        for (int x = 1; x < 32; x <<= 1) {
            const uint32_t up = __shfl_up_sync(MIX_FULL, incl, x);
            if (lane >= (uint32_t)x) incl += up;
        }
        const uint32_t first = n_items + incl - ng;
        n_items += __shfl_sync(MIX_FULL, incl, 31);
        uint64_t ends = ~0ull;
        if (i < P) {
            uint32_t run = 0, tp_least = 0xffffffffu, tpi_least = 0;
#pragma unroll
            for (uint32_t q = 0; q < SAILOR_MIX_GROUPS_MAX; ++q) {
                if (q >= ng) break;
                const uint32_t ty = gw[q] & 0xff, ti = (gw[q] >> 8) & 0xff, cn = gw[q] >> 16, tp = h->tp_values[ti];
                if (q) ends = (ends & ~(0xffffull << (16 * (q - 1)))) | (uint64_t)(run & 0xffffu) << (16 * (q - 1));
                run += cn;
                if (cn == 0 || tp > h->gpn[ty] || !((h->heads_ok >> ti) & 1u)) status |= SAILOR_ST_INVALID;
                if (tp < tp_least) { tp_least = tp; tpi_least = ti; }
                s.item[first + q].type = gw[q];                  // completed below
                s.stage_of[first + q] = (uint8_t)i;
            }
            if (run != D) status |= SAILOR_ST_INVALID;
            const bool e = (i == 0) && h->has_embed, hd = (i == P - 1) && h->has_head;
            MixStage st;
            st.comp = ((e ? 2u : 0u) + (hd ? 1u : 0u)) * h->chain_len + base + (i < extra ? 1u : 0u);
            st.ends = ends;
            st.cross2 = -1.0;
            st.grad = v.cmp_grad[(size_t)st.comp * h->n_tp + tpi_least];
            st.first = first | zone << 16 | ng << 24;
            s.stage[i] = st;
        }
        ends_of[tl] = ends;
    }
    for (uint32_t d = lane; d < h->R; d += 32) s.cnt[d] = 0;
    __syncwarp();
    const uint64_t xbytes = 2 * n_b * (uint64_t)D * v.p2p[mi];
    double c_comm = 0.0;
#pragma unroll
    for (uint32_t tl = 0; tl < TILES; ++tl) {
        if (tl && 32 * tl >= P) break;
        const uint32_t i = lane + 32 * tl;
        bool crosses = false;
        double cost = 0.0;
        if (i + 1 < P) {
            const uint32_t z = (s.stage[i].first >> 16) & 0xff, zn = (s.stage[i + 1].first >> 16) & 0xff;
            crosses = z != zn;
            if (crosses) {
                s.stage[i].cross2 = zone2[(z * Z + zn) * n_mbs + mi];
                cost = mul_rn((double)xbytes, v.egress[z * Z + zn]);
            }
        }
        for (uint32_t m = __ballot_sync(MIX_FULL, crosses); m; m &= m - 1)    // boundaries in stage order
            c_comm = add_rn(c_comm, __shfl_sync(MIX_FULL, cost, __ffs(m) - 1));
    }

    // ---- a lane per item -------------------------------------------------------------------------
    const uint32_t piece_stride = T * h->n_tp * n_mbs * 2;
    const double steps = (double)(2 * (uint64_t)(D - 1)), coef = steps / (double)D;
    double max_sync = 0.0, max_u = 0.0, rate = 0.0;
    uint64_t peak = 0;
    for (uint32_t at = 0; at < n_items; at += 32) {
        const uint32_t it = at + lane;
        double term = 0.0;
        if (it < n_items) {
            const uint32_t gq = s.item[it].type, ty = gq & 0xff, ti = (gq >> 8) & 0xff, cn = gq >> 16;
            const uint32_t i = s.stage_of[it];
            const MixStage& st = s.stage[i];
            const uint32_t zone = (st.first >> 16) & 0xff, ng = st.first >> 24, d = zone * T + ty, tp = h->tp_values[ti];
            const PieceRec* pr = piece + (size_t)st.comp * piece_stride + ((ty * h->n_tp + ti) * n_mbs + mi) * 2 + rc;
            const double2 a0 = __ldg(reinterpret_cast<const double2*>(pr));                // fb, upd
            const ulonglong2 a1 = __ldg(reinterpret_cast<const ulonglong2*>(pr) + 1);      // mem0r, mem1
            const uint64_t gpus = (uint64_t)cn * tp;
            MixItem x;
            x.fb = a0.x;
            x.inter2 = __ldg(&inter2[d * n_mbs + mi]);
            x.gpus = gpus > 0x7fffffffull ? 0x7fffffffu : (uint32_t)gpus;
            x.type = ty;
            s.item[it] = x;
            atomicAdd(&s.cnt[d], gpus > 65536 ? 65536u : (uint32_t)gpus);                  // (availability is 16 bits)
            const uint64_t inflight = (uint64_t)(P - i) < n_b ? (uint64_t)(P - i) : n_b;
            const uint64_t m = a1.x + inflight * a1.y;
            if (m > h->capacity[ty]) status |= SAILOR_ST_OOM;
            peak = m > peak ? m : peak;
            max_u = dmax(max_u, a0.y);
            if (D > 1) {
                const bool intra = ng == 1 && (uint64_t)D * tp <= h->gpn[ty];
                max_sync = dmax(max_sync, allreduce_bytes_time(v, d, intra, st.grad, D, steps, coef));
            }
            term = mul_rn((double)(cn * tp), v.price_s[d]);
        }
        const uint32_t n = n_items - at < 32 ? n_items - at : 32;
        for (uint32_t l = 0; l < n; ++l) rate = add_rn(rate, __shfl_sync(MIX_FULL, term, l));
    }
    __syncwarp();                                                // the counters and the items are complete
    for (uint32_t it = lane; it < n_items; it += 32) {
        const uint32_t d = ((s.stage[s.stage_of[it]].first >> 16) & 0xff) * T + s.item[it].type;
        if (s.cnt[d] > avail[d]) status |= SAILOR_ST_OVER_AVAIL;
    }
    status = __reduce_or_sync(MIX_FULL, status);
    o.peak_mem = warp_max_u64(peak);
    o.status = status;
    if (status & SAILOR_ST_INVALID) return o;
    max_sync = warp_max_positive(max_sync);
    max_u = warp_max_positive(max_u);

    // ---- where the intervals start ------------------------------------------------------------------
    uint32_t n_start;
    if (D <= 64) {                                               // a bit per replica
        uint32_t lo = 0, hi = 0;
#pragma unroll
        for (uint32_t tl = 0; tl < TILES; ++tl)
#pragma unroll
            for (uint32_t q = 0; q + 1 < SAILOR_MIX_GROUPS_MAX; ++q) {
                const uint32_t e = (uint32_t)(ends_of[tl] >> (16 * q)) & 0xffffu;
                lo |= e < 32 ? 1u << e : 0u;
                hi |= e >= 32 && e < 64 ? 1u << (e - 32) : 0u;
            }
        lo = __reduce_or_sync(MIX_FULL, lo) | 1u;
        hi = D > 32 ? __reduce_or_sync(MIX_FULL, hi) : 0u;
        const uint32_t below = (1u << lane) - 1u;
        if ((lo >> lane) & 1u) s.start[__popc(lo & below)] = (uint16_t)lane;
        if ((hi >> lane) & 1u) s.start[__popc(lo) + __popc(hi & below)] = (uint16_t)(lane + 32);
        n_start = __popc(lo) + __popc(hi);
    } else {                                                     // from one boundary to the next
        n_start = 0;
        for (uint32_t k = 0; k < D;) {
            if (lane == 0) s.start[n_start] = (uint16_t)k;
            ++n_start;
            uint32_t next = D;
#pragma unroll
            for (uint32_t tl = 0; tl < TILES; ++tl)
#pragma unroll
                for (uint32_t q = 0; q + 1 < SAILOR_MIX_GROUPS_MAX; ++q) {
                    const uint32_t e = (uint32_t)(ends_of[tl] >> (16 * q)) & 0xffffu;
                    if (e > k && e < next) next = e;
                }
            k = __reduce_min_sync(MIX_FULL, next);
        }
    }
    __syncwarp();

    // ---- a lane per pipeline -----------------------------------------------------------------------
    auto item_of = [&](const MixStage& st, uint32_t k) {
        const uint32_t lo = (uint32_t)st.ends, hi = (uint32_t)(st.ends >> 32);
        return (st.first & 0xffffu) + (k >= (lo & 0xffffu) ? 1u : 0u) + (k >= (lo >> 16) ? 1u : 0u) + (k >= (hi & 0xffffu) ? 1u : 0u);
    };
    double max_pp = 0.0;
    for (uint32_t at = 0; at < n_start; at += 32) {
        const uint32_t k = s.start[at + lane < n_start ? at + lane : n_start - 1];
        MixItem cur = s.item[item_of(s.stage[0], k)];
        double sum_t = 0.0, max_t = 0.0;
        for (uint32_t i = 0; i + 1 < P; ++i) {
            const MixItem nx = s.item[item_of(s.stage[i + 1], k)];
            const double cross2 = s.stage[i].cross2;
            const bool intra = cur.type == nx.type && cur.gpus + nx.gpus <= h->gpn[cur.type];
            double c2 = dmax(cur.inter2, nx.inter2);             // unlike types: the slower end counts
            if (intra) c2 = __ldg(&intra2[(((s.stage[i].first >> 16) & 0xff) * T + cur.type) * n_mbs + mi]);
            c2 = cross2 >= 0.0 ? cross2 : c2;
            const double t = add_rn(cur.fb, c2);
            sum_t = add_rn(sum_t, t);
            max_t = dmax(max_t, t);
            cur = nx;
        }
        sum_t = add_rn(sum_t, cur.fb);                           // the final stage sends nothing
        max_t = dmax(max_t, cur.fb);
        max_pp = dmax(max_pp, add_rn(sum_t, mul_rn((double)n_b, max_t)));
    }
    max_pp = warp_max_positive(max_pp);
    o.t_iter = add_rn(add_rn(max_pp, max_sync), max_u);
    o.cost = add_rn(mul_rn(rate, o.t_iter), c_comm);
    return o;
}

}  // namespace sailor
