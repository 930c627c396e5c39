// The per-stage recursion under a cost limit (Sailor Sec. 4.2.3, "Adding a monetary cost constraint", and the
// second half of the listing in Sec. 4.2.2).
//
// A stage is charged  C_i = rate_i * (N_b * t_straggler) + C_comm_i  with an ASSUMED straggler: first its own
// time; the stages after it are solved with what is left of the limit, and when their straggler turns out
// slower the stage is charged again with that one and they are solved again, until the assumption holds,
// nothing is left, or they have no plan.  The remaining limit is an argument of the recursion, so a state has no
// single value and the tables of the unlimited search do not apply: every problem (configuration x zone order) is
// walked depth-first with an explicit stack.  Problems, and the types of a problem's first two stages, are independent, which
// is where the parallelism is; a walk itself is sequential by nature (each call's limit depends on the charges before
// it).  A branch is cut when what is left cannot pay even the cheapest conceivable rest of the
// pipeline (every later stage alone on its cheapest GPUs, charged for its own compute time): such a branch has no
// plan, so the cut changes nothing but the work.  A problem that would take more than `node_limit` calls is given
// up and reported as unfinished.
#pragma once

#include "sailor_dp.cuh"

namespace sailor {

constexpr uint32_t DP_BUDGET_P_MAX = 32;     // deepest pipeline the limited recursion takes

struct DpProblem {                   // what first fit needs of a (configuration, zone order)
    uint32_t config, order, index;   // index = config * n_orders + order
    uint32_t P, nz, need;            // need = D * tp GPUs per stage
    uint8_t zone[SAILOR_Z_MAX];      // zone of each position of the order
    uint8_t cap[SAILOR_Z_MAX][SAILOR_T_MAX];       // stages a (position, type) can host, saturated at 255
    uint8_t first_later[SAILOR_Z_MAX][SAILOR_T_MAX];   // first position after zp that can host a stage of the type
};

// What first fit needs of every problem, from the availability last set.  A thread per problem (formed and copied by the
// host it took 60 us for 1 344).
__global__ void __launch_bounds__(128)
dp_budget_problems_kernel(const unsigned char* __restrict__ blob, const uint16_t* __restrict__ avail, SpaceDesc sp,
                          const sailor_zone_order* __restrict__ orders, uint32_t n_orders, uint32_t n_problems, DpProblem* __restrict__ out,
                          unsigned long long* counters) {
    const TabHdr* h = reinterpret_cast<const TabHdr*>(blob);
    const uint32_t x = blockIdx.x * blockDim.x + threadIdx.x, T = h->T;
    if (x < 5) counters[x] = 0;
    if (x >= n_problems) return;
    const uint32_t c = x / n_orders, q = x - c * n_orders;
    const Config k = config_of(sp, c);
    const uint64_t need = (uint64_t)k.D * h->tp_values[k.tpi];
    const sailor_zone_order& order = orders[q];
    DpProblem& pb = out[x];
    pb.config = c; pb.order = q; pb.index = x;
    pb.P = k.P; pb.nz = order.n; pb.need = (uint32_t)(need > 0xffffffffull ? 0xffffffffull : need);
    uint32_t later = 0;                                      // per type (4 bits each): the first position after this one, or none
    for (uint32_t g = 0; g < T; ++g) later |= 15u << (4 * g);
    for (uint32_t zp = pb.nz; zp-- > 0;) {
        const uint32_t z = order.zone[zp];
        pb.zone[zp] = (uint8_t)z;
        for (uint32_t g = 0; g < T; ++g) {
            const uint32_t a = avail[z * T + g], first = (later >> (4 * g)) & 15u;
            const uint32_t cap = need > a ? 0u : a / (uint32_t)need;
            pb.cap[zp][g] = (uint8_t)(cap > 255 ? 255 : cap);
            pb.first_later[zp][g] = first == 15u ? DP_NONE : (uint8_t)first;
            if (cap >= 1) later = (later & ~(15u << (4 * g))) | zp << (4 * g);
        }
    }
}
static_assert(SAILOR_Z_MAX < 15 && SAILOR_T_MAX * 4 <= 32, "a position fits four bits");

struct DpbFrame {                    // one call of the recursion: stage `level` on type g at zone position zp
    double limit;                    // what stages level.. may be charged
    double rate, sync, fb, upd;      // of this stage on its GPUs
    double t, comm, assumed, charge; // the candidate being tried: stage time with its message, transfer cost, ...
    double b_sum, b_mx, b_sy, b_up, b_cost;      // best plan of stages level.. so far (b_found)
    uint8_t g, zp, g2, zp2;          // g2: type tried for the next stage, zp2: where first fit puts it
    uint8_t b_found, _pad[3];
    uint64_t u;                      // stages per type (a byte each) in zone position zp, this stage included
    uint64_t u2;                     // the same for the next stage's position after the move
    union {                          // types of stages level.. of the best plan (indexed by stage)
        uint8_t b_type[DP_BUDGET_P_MAX];
        uint64_t b_word[DP_BUDGET_P_MAX / 8];
    };
};
static_assert(SAILOR_T_MAX <= 8 && DP_BUDGET_P_MAX < 256, "a byte per type holds every count");

struct DpbRoot {                     // what the walk from one type of stage 0 (and one of stage 1, where it is split) found
    double value;                    // +inf: no plan
    unsigned long long nodes;        // calls of the recursion; above the limit: given up
    uint8_t type[DP_BUDGET_P_MAX];
};

struct DpBudgetParams {
    const unsigned char* blob;
    const uint16_t* avail;
    SpaceDesc sp;
    const DpProblem* problems;
    const double* tabs;
    double* value;                   // indexed by problem index; +inf: no plan
    DpResult* results;
    DpbRoot* roots;                  // [n_walks]
    unsigned long long* counters;    // [3] += problems given up, [4] += calls of the recursion
    DpTabLayout lay;
    uint32_t n_problems, T, p_max;
    uint32_t n_walks;
    uint32_t per_length;             // problems of each pipeline length in the space's list: problem / per_length is its place there
    uint32_t split;                  // bit: problems of this length have a walk per type of stage 1 as well
    uint32_t first[SAILOR_NP_MAX];   // the first walk of a length (deep ones first; all in the problems' order where none is split)
    double limit;
    unsigned long long node_limit;

    __host__ __device__ uint32_t walks_of_type(uint32_t length) const { return (split >> length) & 1u ? T : 1u; }
};
static_assert(SAILOR_NP_MAX <= 32, "a bit per length");

__device__ __forceinline__ double dpb_value(double nb, double sum, double mx, double sy, double up) {
    return add_rn(add_rn(add_rn(sum, mul_rn(nb, mx)), sy), up);
}

// A warp per (problem, type of stage 0) or, where walks are split, (problem, type of stage 0, type of stage 1): what the first stage
// has to give to a type of the second does not depend on the others, so the best of them is found afterwards
// (dp_budget_finish_kernel), the lowest among equals as in one walk.
// The walk is one lane's: problems differ too much in what they try to share instructions (a thread per problem ran a warp's 32
// walks one after the other), and its stack sits in shared memory.
// Bound by the latency of one chain of calls.  Workload 2, pipelines of up to eight stages, all orders, budget 1.2 x
// cheapest (1 344 problems, up to 4 700 calls, hundreds of them in one walk): 2.76 -> 0.44 ms a call with a warp per first type; a
// frame's counts as bytes of one word and the walk's tables brought near beforehand took its share from 459 to 408 us.
// Warps of a block.  Where walks are split a block is one warp and the kernel compiled for that: the longest walk decides then
// (workload 2, up to 8 stages, and up to 16: 324 us and 13.7 ms a call; blocks of four 347 us and 14.7 ms, of two 361 us and 15.4
// ms; frames of a block's warps side by side instead of each warp's own in one piece 367 us).
template <bool SPLIT> constexpr uint32_t DPB_WARPS = SPLIT ? 1 : 4;
// Where walks are split, by the length of their pipelines, deepest first: as long as the walks this adds, for all lengths split so
// far, are at most DPB_SPLIT_WORTH times the calls that one walk from a first type can make without charging again.  A walk costs
// about 0.5 ns (its block, and reading that there is nothing to do), and where the limit is tight most of them end at once; what a
// long one saves grows with its calls.  us a call, unsplit and split, limits of 1.2 and 1.01 x the cheapest plan:
//   workload 3, up to 4 stages (85 calls):  7 680 walks more 117 97, 79 80; 11 520 more 119 102, 84 83; 19 200 more 128 111, 90 93
//   workload 3, up to 3 stages (21 calls):  3 840 more 73 70, 65 66; 15 360 more 86 85, 75 80
//   workload 5, up to 4 stages: the deepest (259 calls), 14 400 more 97 85, 82 80; with the second (43 calls), 28 800 more 89, 87
//   eight types, up to 3 stages (73 calls): 16 128 more 153 102
// All lengths split (workload 3, up to 2 stages, 51 000 walks): 75 -> 95 us.  Fewer than DPB_SPLIT_CALLS calls (two types, three
// stages: 7; three types: 13) are not worth a walk of their own; two types, four stages, 15 calls: 89 -> 76 us.
constexpr uint64_t DPB_SPLIT_CALLS = 15, DPB_SPLIT_WORTH = 224;
// Most walks of a search that splits any (their records' memory).
constexpr uint64_t DPB_SPLIT_WALKS = 1u << 16;
constexpr size_t DPB_NEAR_BYTES = 16 * 1024;      // tables of up to this size are brought near before a walk

inline size_t dpb_smem(uint32_t p_max, uint32_t warps) {
    return warps * (p_max * sizeof(DpbFrame) + (p_max + 1) * sizeof(double));
}

template <bool SPLIT>
__global__ void __launch_bounds__(32 * DPB_WARPS<SPLIT>) dp_budget_kernel(const __grid_constant__ DpBudgetParams bp) {
    extern __shared__ __align__(16) unsigned char dyn[];
    constexpr uint32_t WARPS = DPB_WARPS<SPLIT>;
    const uint32_t lane = threadIdx.x & 31u, warp = WARPS > 1 ? threadIdx.x >> 5 : 0u;
    const uint32_t unit = blockIdx.x * WARPS + warp, T = bp.T;
    if (unit >= bp.n_walks) return;
    uint32_t length = 0, split = SPLIT ? bp.walks_of_type(0) : 1u, first = 0;
    if (SPLIT) {
        while (unit - bp.first[length] >= bp.per_length * T * split) split = bp.walks_of_type(++length);
        first = bp.first[length];
    }
    const uint32_t nth = (unit - first) / split, of_length = nth / T, x = length * bp.per_length + of_length;
    const uint32_t g0 = nth - of_length * T, g1 = unit - first - nth * split;
    const uint32_t g1_end = split > 1 ? g1 + 1 : T;              // types of stage 1 that this walk tries
    DpbFrame* const fr = reinterpret_cast<DpbFrame*>(dyn) + warp * bp.p_max;
    double* const lb = reinterpret_cast<double*>(reinterpret_cast<DpbFrame*>(dyn) + WARPS * bp.p_max) + warp * (bp.p_max + 1);
    const DpProblem& pb = bp.problems[x];
    DpbRoot& root = bp.roots[unit];
    if (lane == 0) { root.value = make_inf(); root.nodes = 0; }
    const uint32_t P = pb.P;
    const double* tab = bp.tabs + (size_t)pb.config * bp.lay.stride();
    if (*reinterpret_cast<const uint32_t*>(tab + bp.lay.off_nb() + 1) == 0 || P > DP_BUDGET_P_MAX) return;   // no valid plan here
    TabView v;
    v.bind(bp.blob, bp.blob);
    const TabHdr* h = v.h;
    const uint32_t R = h->R, Z = h->Z;
    const uint32_t* okv = reinterpret_cast<const uint32_t*>(tab + bp.lay.off_ok());
    if (!((okv[0] >> g0) & 1u)) return;
    if (g1 && (P == 1 || !((okv[1] >> g1) & 1u))) return;
    const uint32_t p0 = pb.cap[0][g0] >= 1 ? 0u : pb.first_later[0][g0];     // by first fit from the first zone of the order
    if (p0 == DP_NONE) return;
    const uint64_t n_b = *reinterpret_cast<const uint64_t*>(tab + bp.lay.off_nb());
    const double nb = (double)n_b;
    const Config k = config_of(bp.sp, pb.config);
    const double gpus = (double)(k.D * h->tp_values[k.tpi]);
    const double xbytes = (double)(2 * n_b * (uint64_t)k.D * v.p2p[k.mi]);
    const double* fbt = tab + bp.lay.off_fb();
    const double* updt = tab + bp.lay.off_upd();
    const double* synct = tab + bp.lay.off_sync();
    const double* c2x = tab + bp.lay.off_c2x();

    // one thread walks below: what it reads is brought near by all of them first (a walk of a few dozen calls otherwise
    // waits for one line after another)
    auto bring = [&](const void* first, size_t bytes) {
        const uintptr_t at = reinterpret_cast<uintptr_t>(first) & ~(uintptr_t)127, end = reinterpret_cast<uintptr_t>(first) + bytes;
        for (uintptr_t a = at + 128 * lane; a < end; a += 128 * 32) asm volatile("prefetch.global.L1 [%0];" ::"l"(a));
    };
    bring(&pb, sizeof(pb));
    bring(v.price_s, R * sizeof(double));
    bring(v.egress, Z * Z * sizeof(double));
    if (bp.lay.stride() * sizeof(double) <= DPB_NEAR_BYTES) bring(tab, bp.lay.stride() * sizeof(double));

    // the least any plan of stages j.. can be charged: every stage alone on the cheapest GPUs it fits, for its own
    // compute time; added up from the last stage backwards, as the recursion adds its charges
    if (lane < P) {
        double least = make_inf();
        for (uint32_t g = 0; g < T; ++g) {
            if (!((okv[lane] >> g) & 1u)) continue;
            for (uint32_t q = 0; q < pb.nz; ++q) {
                const double c = mul_rn(mul_rn(gpus, v.price_s[pb.zone[q] * T + g]), mul_rn(nb, fbt[lane * T + g]));
                least = c < least ? c : least;
            }
        }
        lb[lane] = least;
    }
    __syncwarp();
    if (lane != 0) return;
    lb[P] = 0.0;
    for (uint32_t j = P; j-- > 0;) lb[j] = add_rn(lb[j], lb[j + 1]);
    if (bp.limit < lb[0]) return;

    unsigned long long nodes = g1 ? ~0ull : 0ull;                // (the call for the first stage counts once)
    bool gave_up = false;
    // result of the call that has just returned
    bool r_found = false;
    double r_sum = 0.0, r_mx = 0.0, r_sy = 0.0, r_up = 0.0, r_cost = 0.0;
    int level = 0;
    {
        DpbFrame& f = fr[0];
        f.g = (uint8_t)g0; f.zp = (uint8_t)p0; f.limit = bp.limit;
        f.u = 1ull << (8 * g0);
    }
    enum { ENTER, NEXT_TYPE, CHARGE, RESUME } state = ENTER;
    while (level >= 0) {
        DpbFrame& f = fr[level];
        const uint32_t i = (uint32_t)level, g = f.g, z = pb.zone[f.zp], d = z * T + g;
        if (state == ENTER) {
            if (++nodes > bp.node_limit) { gave_up = true; break; }
            f.b_found = 0;
            f.rate = mul_rn(gpus, v.price_s[d]);
            f.sync = synct[i * R + d];
            f.fb = fbt[i * T + g];
            f.upd = updt[i * T + g];
            if (i == P - 1) {                    // the last stage sends nothing and is its own straggler
                const double charge = mul_rn(f.rate, mul_rn(nb, f.fb));
                r_found = charge <= f.limit;
                r_sum = f.fb; r_mx = f.fb; r_sy = f.sync; r_up = f.upd; r_cost = charge;
                f.b_type[i] = (uint8_t)g;
                --level;
                state = RESUME;
                continue;
            }
            f.g2 = (uint8_t)(level ? 0u : g1);
            state = NEXT_TYPE;
        }
        if (state == NEXT_TYPE) {
            bool placed = false;
            for (const uint32_t g2_end = level ? T : g1_end; f.g2 < g2_end;) {
                const uint32_t g2 = f.g2;
                if ((okv[i + 1] >> g2) & 1u) {
                    // first fit: this zone while it has room for one more stage of the type, else the next that has
                    uint32_t zp2 = f.zp;
                    if (!(((uint32_t)(f.u >> (8 * g2)) & 0xffu) < pb.cap[f.zp][g2])) zp2 = pb.first_later[f.zp][g2];
                    if (zp2 != DP_NONE) {
                        f.zp2 = (uint8_t)zp2;
                        f.u2 = (zp2 == f.zp ? f.u : 0ull) + (1ull << (8 * g2));
                        const uint32_t z2 = pb.zone[zp2], dn = z2 * T + g2;
                        f.t = add_rn(f.fb, c2x[dn * R + d]);
                        f.comm = z2 != z ? mul_rn(xbytes, v.egress[z * Z + z2]) : 0.0;
                        f.assumed = f.t;                 // first: this stage is the straggler
                        placed = true;
                        break;
                    }
                }
                ++f.g2;
            }
            if (!placed) {                               // every type tried: hand the best plan back
                r_found = f.b_found != 0;
                r_sum = f.b_sum; r_mx = f.b_mx; r_sy = f.b_sy; r_up = f.b_up; r_cost = f.b_cost;
                --level;
                state = RESUME;
                continue;
            }
            state = CHARGE;
        }
        if (state == CHARGE) {
            f.charge = add_rn(mul_rn(f.rate, mul_rn(nb, f.assumed)), f.comm);
            const double rest = f.limit - f.charge;
            if (!(rest > 0.0) || rest < lb[i + 1]) {    // nothing left, or not enough for any rest of the pipeline
                ++f.g2;
                state = NEXT_TYPE;
                continue;
            }
            DpbFrame& c = fr[level + 1];
            c.g = f.g2; c.zp = f.zp2; c.limit = rest;
            c.u = f.u2;
            ++level;
            state = ENTER;
            continue;
        }
        // RESUME: the call for stages i + 1.. has returned
        if (!r_found) {
            ++f.g2;
            state = NEXT_TYPE;
            continue;
        }
        if (r_mx <= f.assumed) {                         // the assumption holds
            const double all = add_rn(f.charge, r_cost);
            if (all <= f.limit) {
                const double c_sum = add_rn(f.t, r_sum), c_mx = dmax(f.t, r_mx), c_sy = dmax(f.sync, r_sy),
                             c_up = dmax(f.upd, r_up);
                if (!f.b_found || dpb_value(nb, c_sum, c_mx, c_sy, c_up) < dpb_value(nb, f.b_sum, f.b_mx, f.b_sy, f.b_up)) {
                    f.b_found = 1;
                    f.b_sum = c_sum; f.b_mx = c_mx; f.b_sy = c_sy; f.b_up = c_up; f.b_cost = all;
                    const DpbFrame& c = fr[level + 1];
#pragma unroll
                    for (uint32_t j = 0; j < DP_BUDGET_P_MAX / 8; ++j) f.b_word[j] = c.b_word[j];
                    f.b_type[i] = (uint8_t)g;
                }
            }
            ++f.g2;
            state = NEXT_TYPE;
            continue;
        }
        f.assumed = r_mx;                                // charge again with the straggler that was found
        state = CHARGE;
    }
    root.nodes = nodes;
    if (gave_up || !r_found) return;
    root.value = dpb_value(nb, r_sum, r_mx, r_sy, r_up);
    for (uint32_t j = 0; j < P; ++j) root.type[j] = fr[0].b_type[j];
}

// Per problem the best of its walks (the lowest types among equals), written out and simulated; a warp each.
__global__ void __launch_bounds__(DP_FINISH_THREADS) dp_budget_finish_kernel(const __grid_constant__ DpBudgetParams bp) {
    __shared__ DpFinishWarp warps[DP_FINISH_WARPS];
    const uint32_t lane = threadIdx.x & 31, x = blockIdx.x * DP_FINISH_WARPS + (threadIdx.x >> 5);
    if (x >= bp.n_problems) return;
    DpFinishWarp& w = warps[threadIdx.x >> 5];
    const DpProblem& pb = bp.problems[x];
    const uint32_t T = bp.T, P = pb.P;
    const uint32_t length = x / bp.per_length, n_roots = T * bp.walks_of_type(length);
    const DpbRoot* roots = bp.roots + bp.first[length] + (size_t)(x - length * bp.per_length) * n_roots;
    unsigned long long nodes = 0;
    double best_v = make_inf();
    uint32_t best = DP_NONE;
    for (uint32_t g = 0; g < n_roots; ++g) {
        nodes += roots[g].nodes;
        if (roots[g].value < best_v) { best_v = roots[g].value; best = g; }
    }
    if (lane == 0 && nodes) atomicAdd(&bp.counters[4], nodes);
    if (nodes > bp.node_limit) {
        if (lane == 0) atomicAdd(&bp.counters[3], 1ull);
        return;
    }
    if (best == DP_NONE) return;
    if (lane == 0) bp.value[pb.index] = best_v;
    const uint8_t* best_type = roots[best].type;
    DpResult& out = bp.results[pb.index];
    TabView v;
    v.bind(bp.blob, bp.blob);
    const Config k = config_of(bp.sp, pb.config);
    // zones by first fit, as the recursion placed them; then the plan through the simulator (Sec. 4.3)
    const uint32_t my_type = lane < P ? best_type[lane] : 0u;
    static_assert(DP_BUDGET_P_MAX <= 32, "a lane per stage");
    if (lane < SAILOR_T_MAX) w.used[lane] = 0;
    __syncwarp();
    for (uint32_t i = 0, zp = 0; i < P; ++i) {
        const uint32_t g = __shfl_sync(FULL, my_type, i);
        const uint32_t zp2 = w.used[g] < pb.cap[zp][g] ? zp : (uint32_t)pb.first_later[zp][g];
        __syncwarp();
        if (lane < SAILOR_T_MAX) w.used[lane] = (uint8_t)((zp2 != zp ? 0u : w.used[lane]) + (lane == g ? 1u : 0u));
        zp = zp2;
        if (lane == i) w.gz[i] = (uint16_t)(g | pb.zone[zp] << 8);
        __syncwarp();
    }
    if (lane < P) {
        out.type[lane] = (uint8_t)my_type;
        out.zone[lane] = (uint8_t)(w.gz[lane] >> 8);
    }
    const SimOut so = simulate_stages(v, bp.avail, k, w.gz, w.cnt, lane);
    if (lane == 0) {
        out.t_iter = so.t_iter;
        out.cost = so.cost;
        out.peak_mem = so.peak_mem;
        out.status = so.status;
    }
}

}  // namespace sailor
