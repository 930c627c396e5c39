// C ABI of the library (see include/sailor.h): context management, argument checks, launches.
// Every simulation step runs in the kernels; the host only validates, packs tables and
// enqueues work on the caller's stream.
#include <atomic>
#include <chrono>
#include <cmath>
#include <cstddef>
#include <cstdlib>
#include <cstring>
#include <memory>
#include <new>
#include <vector>

#include <algorithm>
#include <array>
#include <map>
#include <mutex>

#include "sailor_batch.cuh"
#include "sailor_dp.cuh"
#include "sailor_dp_budget.cuh"
#include "sailor_mixed.cuh"
#include "sailor_mixed_batch.cuh"
#include "sailor_mixed_search.cuh"
#include "sailor_peaks.cuh"
#include "sailor_plan_setup.cuh"

using namespace sailor;

namespace {

constexpr int PLAN_SMEM_CEILING = 200 * 1024;    // dynamic shared memory any search may ask for

// ---- kernels of the explicit-batch path -----------------------------------------------------

// Left-to-right layer sums for every stage composition: chain[n] = start + n blocks, where
// start is 0 or the embedding layer's entry.  One thread per (table, start, type, tp[, mbs]).
__global__ void chain_kernel(unsigned char* blob) {
    TabView v;
    v.bind(blob, blob);
    const TabHdr* h = v.h;
    const uint32_t gts = h->T * h->n_tp;
    const uint32_t n4 = 2 * gts * h->n_mbs;                  // [start][type][tp][mbs]
    const uint32_t n3 = 2 * gts;                             // [start][type][tp]
    const uint32_t x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x < 2 * n4) {
        const bool is_b = x >= n4;
        const uint32_t y = is_b ? x - n4 : x;
        const uint32_t mi = y % h->n_mbs, gt = (y / h->n_mbs) % gts, start = y / (h->n_mbs * gts);
        const double* tab = is_b ? v.bwd : v.fwd;
        double* out = reinterpret_cast<double*>(blob + (is_b ? h->off_chain_b : h->off_chain_f)) + (size_t)y * h->chain_len;
        const double e = tab[((size_t)KIND_EMBED * gts + gt) * h->n_mbs + mi];
        const double b = tab[((size_t)KIND_BLOCK * gts + gt) * h->n_mbs + mi];
        double acc = start ? add_rn(0.0, e) : 0.0;
        out[0] = acc;
        for (uint32_t n = 1; n < h->chain_len; ++n) { acc = add_rn(acc, b); out[n] = acc; }
    } else if (x < 2 * n4 + n3) {
        const uint32_t y = x - 2 * n4;
        const uint32_t gt = y % gts, start = y / gts;
        double* out = reinterpret_cast<double*>(blob + h->off_chain_u) + (size_t)y * h->chain_len;
        const double e = v.upd[(size_t)KIND_EMBED * gts + gt];
        const double b = v.upd[(size_t)KIND_BLOCK * gts + gt];
        double acc = start ? add_rn(0.0, e) : 0.0;
        out[0] = acc;
        for (uint32_t n = 1; n < h->chain_len; ++n) { acc = add_rn(acc, b); out[n] = acc; }
    }
}

// What a stage needs, per stage composition (embedding?, head?, number of blocks): parameters, gradient bytes per
// worker, memory without and per in-flight microbatch, f + b, update time.  Formed with the same functions and
// the same operation order as a stage-by-stage evaluation; one thread per (composition, type, tp, mbs, rc).
__global__ void compose_kernel(unsigned char* blob) {
    TabView v;
    v.bind(blob, blob);
    const TabHdr* h = v.h;
    const size_t n_comp = (size_t)4 * h->chain_len;
    const size_t total = n_comp * h->T * h->n_tp * h->n_mbs * 2;
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
        reinterpret_cast<double*>(blob + h->off_cmp_fb)[x] = add_rn(st.f, b);
        if (mi == 0 && rc == 0) reinterpret_cast<double*>(blob + h->off_cmp_upd)[(comp * h->T + g) * h->n_tp + tpi] = st.u;
        if (g == 0) {
            const StageMem one = stage_memory(v, tpi, mi, rc, nb, e, hd, 1);     // model + 1 * kept + work
            const StageMem zero = stage_memory(v, tpi, mi, rc, nb, e, hd, 0);    // model + work
            uint64_t* mm = reinterpret_cast<uint64_t*>(blob + h->off_cmp_mem) + (((comp * h->n_tp + tpi) * h->n_mbs + mi) * 2 + rc) * 2;
            mm[0] = zero.mem;
            mm[1] = one.mem - zero.mem;
            if (mi == 0 && rc == 0) {
                reinterpret_cast<double*>(blob + h->off_cmp_grad)[comp * h->n_tp + tpi] =
                    (double)(ceil_div64(one.params, h->tp_values[tpi]) * h->grad_bytes);
                if (tpi == 0) reinterpret_cast<uint64_t*>(blob + h->off_cmp_params)[comp] = one.params;
            }
        }
    }
}

// A warp per plan with mixed replicas (records `stride` bytes apart holding `max_stages` stages, read in place): all plans of up
// to 32 stages of a small batch (DEEP = false; see mixb_takes), or the deeper ones of any batch.  The launch for shallow plans,
// this or simulate_mixed_kernel, notes in `deep_seen` that there are deep ones; the DEEP launch that follows returns at once when
// there are none (three times the scratch per warp).
template <bool DEEP> constexpr uint32_t MIX_WARPS = DEEP ? 4 : 8;
template <bool DEEP> constexpr uint32_t MIX_STAGES = DEEP ? SAILOR_MIX_P_MAX : MIXB_P_MAX;

template <bool DEEP>
__global__ void __launch_bounds__(32 * MIX_WARPS<DEEP>, 4)
simulate_mixed_each_kernel(const __grid_constant__ MixbCall p) {
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ uint64_t mbar;
    if (DEEP && *reinterpret_cast<const volatile unsigned int*>(p.deep_seen) == 0) return;
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    constexpr uint32_t WARPS = MIX_WARPS<DEEP>;
    const uint32_t static_bytes = reinterpret_cast<const TabHdr*>(p.blob)->static_bytes;
    if (!bulk_load(dyn, p.blob, static_bytes, &mbar)) {
        if (tid == 0) atomicOr(p.error, SIM_ERR_DEVICE);
        for (uint32_t x = tid; x < static_bytes / 16; x += 32 * WARPS)
            reinterpret_cast<uint4*>(dyn)[x] = reinterpret_cast<const uint4*>(p.blob)[x];
        __syncthreads();
    }
    TabView v;
    v.bind(dyn, p.blob);
    auto& scratch = reinterpret_cast<MixScratch<MIX_STAGES<DEEP>>*>(dyn + static_bytes)[warp];
    for (uint64_t j = (uint64_t)blockIdx.x * WARPS + warp; j < p.n; j += (uint64_t)gridDim.x * WARPS) {
        const sailor_mixed_plan& r = *reinterpret_cast<const sailor_mixed_plan*>(p.plans + j * p.stride);
        const uint32_t P = r.P;
        SimOut o;
        if (DEEP && (P <= MIXB_P_MAX || P > p.max_stages)) continue;     // done by the first launch
        if (P > p.max_stages) {                                  // more stages than the record has room for
            o.t_iter = o.cost = make_nan();
            o.peak_mem = 0;
            o.status = SAILOR_ST_BAD_RECORD;
        } else if (!DEEP && P > MIXB_P_MAX) {
            if (lane == 0) *reinterpret_cast<volatile unsigned int*>(p.deep_seen) = 1u;
            continue;
        } else {
            o = simulate_mixed_warp(v, p.blob, p.avail, r, scratch, lane);
        }
        if (lane == 0) mixb_store(p, j, o);
        __syncwarp();
    }
}

template <bool DEEP>
size_t mixed_smem(const TabHdr& h) { return h.static_bytes + sizeof(MixScratch<MIX_STAGES<DEEP>>) * MIX_WARPS<DEEP>; }
template <bool DEEP>
size_t mixed_finish_smem(const TabHdr& h) { return h.static_bytes + sizeof(MixFinishWarp<DEEP>) * MIXF_WARPS<DEEP>; }

// ---- host state -----------------------------------------------------------------------------

struct MixedTables {
    sailor_mixed_space key;                    // the space the tables are of
    MixedSpaceDesc desc;
    std::vector<uint64_t> combs;
    std::vector<uint64_t> flat_base;           // [n_config + 1]
    uint32_t n_config = 0;
};

struct SpaceCache {
    bool valid = false;
    sailor_space key;
    SpaceDesc desc;
    uint32_t n_config = 0, n_chunks = 0, p_max = 0;
    uint64_t n_total = 0;
    std::vector<uint32_t> chunk_start;     // host copies, for range -> chunk lookup
    std::vector<uint64_t> flat_base;
    unsigned char* d_mem = nullptr;        // one piece of device memory that holds everything below
    uint32_t* d_chunk_start = nullptr;
    uint64_t* d_flat_base = nullptr;
    size_t smem = 0, smem_screen = 0;      // dynamic shared memory of a search block, without and with the binary32 tables
    // chunks of live prefixes only (see survey_kernel), for whole-space searches with pruning on
    uint32_t* d_live_start = nullptr;      // [n_config + 1]
    uint32_t live_chunks = 0;
    unsigned long long closed[3] = {0, 0, 0};   // candidates counted in closed form: total, invalid, oom
    // searches in degree order (spaces of at most WAVE_CONFIG_MAX configurations)
    unsigned long long* d_cfg_closed = nullptr;   // [n_config][3] the closed-form counts per configuration
    uint32_t* d_wave_start = nullptr;             // [n_config + 1] chunk offsets of the current wave
    unsigned long long* d_cfg_best = nullptr;     // [n_config] best feasible score per configuration
    GroupState* d_groups = nullptr;               // [n_config / n_d]
    // the per-configuration tables, built once per space (spaces whose records fit CFG_CACHE_MAX_BYTES)
    uint4* d_cfg_cache = nullptr;
    uint32_t cache_head16 = 0, cache_arr16 = 0;
};

// What a context keeps in pinned host memory the device can write.
constexpr size_t HOST_SMALL_BYTES = 192 * 1024;


struct HostBlock {
    PlanOut out;                           // results of a search
    SurveyOut survey;                      // what the survey of a space found
    uint16_t avail[R_MAX];                 // the availability snapshot last set
    unsigned int sim_error;                // error word of the explicit-batch kernels: read and cleared by the next host-side batch
    MixedOut mixed;                        // results of a search over plans with mixed replicas
    DpOut dp;                              // results of a search over per-stage GPU types
    alignas(256) unsigned char batch[HOST_SMALL_BYTES];     // a small host batch: records, results
};

constexpr size_t CFG_CACHE_MAX_BYTES = 512ull << 20;

constexpr uint64_t WAVE_CONFIG_MAX = 1u << 16;

}  // namespace

static_assert(offsetof(Ctrl, thr_bits) == offsetof(Ctrl, min_cost_bits) + 8, "cleared together");

struct sailor_ctx {
    int device = 0;
    cudaStream_t stream = nullptr;
    int last_cuda = 0;
    int sm_count = 0;
    TabHdr hdr;                            // host copy of the header
    unsigned char* d_mem = nullptr;        // one piece of device memory: the blob and the small buffers below
    unsigned char* d_blob = nullptr;
    uint16_t* d_avail = nullptr;           // device copy for the kernels that take a pointer (brought up to date lazily)
    HostBlock* host = nullptr;             // pinned, one of the process's few such blocks
    uint16_t* h_avail = nullptr;           // host->avail
    bool avail_dirty = false;              // d_avail is older than h_avail
    PlanOut* d_out_mapped = nullptr;       // device address of h_out (mapped pinned memory)
    Ctrl* d_ctrl = nullptr;
    unsigned int* d_sim_error = nullptr;   // device address of host->sim_error
    unsigned int* d_deep_seen = nullptr;   // mixed batches: "deep plans seen"
    PlanOut* h_out = nullptr;              // &host->out
    bool ctrl_dirty = true;                // the counters must be cleared from the host (first call, or after a failed one)
    uint64_t ticket = 0;                   // calls that ended with one (wait_ticket)
    uint64_t sync_epoch = 1;               // stream synchronisations by this context so far
    uint64_t avail_epoch = 0;              // sync_epoch when the pinned availability buffer was last handed to a copy
    bool h2d_fresh = false;                // an availability upload has been timed and not yet read
    float h2d_ms = 0.f;
    Hit* d_partial = nullptr;
    uint32_t* d_partial_n = nullptr;
    uint32_t max_grid = 0;                 // capacity of the partial-result buffers
    uint32_t grid_of[30] = {0};            // resident blocks per kernel variant, for the cached space
    SpaceCache space;
    cudaEvent_t ev0 = nullptr, ev1 = nullptr, ev2 = nullptr, evh0 = nullptr, evh1 = nullptr;
    cudaStream_t out_stream = nullptr;     // results of a host batch leave on it while the next chunk comes in
    cudaEvent_t ev_chunk = nullptr, ev_join = nullptr, ev_slot[3] = {nullptr, nullptr, nullptr};
    // explicit-batch staging (grow-only)
    unsigned char* d_stage = nullptr;
    size_t stage_bytes = 0;
    std::vector<unsigned char> h_static;   // host copy of the blob's static part
    // the search over plans with mixed replicas: tables of the space last searched, working memory (grow-only)
    MixedTables* mix = nullptr;
    unsigned char* d_mix = nullptr;
    size_t mix_bytes = 0;
    bool mix_dirty = true;                 // the counters must be cleared from the host (fresh memory, or a failed search)
    // tables of the dynamic-programming search (grow-only)
    unsigned char* d_dp = nullptr;
    size_t dp_bytes = 0;
    unsigned char* d_dp_up = nullptr;      // layouts, jobs and block lists of a batch
    size_t dp_up_bytes = 0;
};

namespace {

#define CU(ctx, call)                                  \
    do {                                               \
        cudaError_t e_ = (call);                       \
        if (e_ != cudaSuccess) {                       \
            (ctx)->last_cuda = (int)e_;                \
            return SAILOR_E_CUDA;                      \
        }                                              \
    } while (0)

// Synchronise the context's stream; everything enqueued before (the availability upload among it) is done after.
cudaError_t stream_sync(sailor_ctx* ctx) {
    const cudaError_t e = cudaStreamSynchronize(ctx->stream);
    if (e == cudaSuccess) ++ctx->sync_epoch;
    return e;
}

inline void cpu_relax() {
#if defined(__x86_64__)
    __builtin_ia32_pause();
#endif
}

// Waits until the kernel that ends a call has left its results, with `ticket` behind them, in the context's pinned memory:
// the host sees them some microseconds before the stream counts as idle (a search of one zone with new availability:
// 55.2 us by cudaStreamSynchronize, 52.5 this way).  Everything enqueued earlier on the stream is done by then.  Longer
// searches, of which those microseconds are a small part, wait in cudaStreamSynchronize after a millisecond, the way the
// application has chosen for the device (blocking, yielding); it also finds out a stream that fails.
constexpr std::chrono::microseconds TICKET_SPIN(1000);

cudaError_t wait_ticket(sailor_ctx* ctx, const uint64_t* slot, uint64_t ticket) {
    const volatile uint64_t* seen = slot;
    const auto until = std::chrono::steady_clock::now() + TICKET_SPIN;
    for (uint32_t spin = 1; *seen != ticket; ++spin) {
        if (spin % 256 == 0 && std::chrono::steady_clock::now() > until) {
            const cudaError_t e = cudaStreamSynchronize(ctx->stream);
            if (e != cudaSuccess) return e;
            break;                                             // (what is missing now never comes)
        }
        cpu_relax();
    }
    std::atomic_thread_fence(std::memory_order_acquire);
    ++ctx->sync_epoch;
    return *seen == ticket ? cudaSuccess : cudaErrorUnknown;
}

struct Bump {                       // carves 256-byte aligned pieces out of one device buffer
    unsigned char* base;
    size_t at = 0;
    template <typename T>
    T* take(size_t n) {
        T* p = reinterpret_cast<T*>(base + at);
        at += (n * sizeof(T) + 255) & ~(size_t)255;
        return p;
    }
};

size_t padded(size_t bytes) { return (bytes + 255) & ~(size_t)255; }

// Device memory comes from one memory pool per device that the library owns: a context's first buffers then cost
// microseconds where cudaMalloc and cudaFree of a megabyte cost 0.3 ms each (up to 12 ms seen).  The pool keeps at most
// POOL_KEEP bytes that no context uses; what is beyond goes back to the device at the synchronisation that ends a call, or
// one at the end of sailor_destroy.  Allocation and release are ordered on the context's stream; the pool itself is safe to
// use from any thread.
constexpr uint64_t POOL_KEEP = 256ull << 20;
constexpr int POOL_DEVICES_MAX = 64;

int device_pool(sailor_ctx* ctx, cudaMemPool_t* out) {
    static std::mutex lock;
    static cudaMemPool_t pools[POOL_DEVICES_MAX];
    if (ctx->device < 0 || ctx->device >= POOL_DEVICES_MAX) return SAILOR_E_RANGE;
    std::lock_guard<std::mutex> hold(lock);
    if (!pools[ctx->device]) {
        cudaMemPoolProps props;
        memset(&props, 0, sizeof(props));
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = ctx->device;
        cudaMemPool_t pool;
        CU(ctx, cudaMemPoolCreate(&pool, &props));
        uint64_t keep = POOL_KEEP;
        CU(ctx, cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep));
        pools[ctx->device] = pool;
    }
    *out = pools[ctx->device];
    return SAILOR_OK;
}

int device_alloc(sailor_ctx* ctx, unsigned char** p, size_t bytes) {
    cudaMemPool_t pool;
    const int rc = device_pool(ctx, &pool);
    if (rc) return rc;
    void* got = nullptr;
    const cudaError_t e = cudaMallocFromPoolAsync(&got, bytes, pool, ctx->stream);
    if (e != cudaSuccess) {
        ctx->last_cuda = (int)e;
        (void)cudaGetLastError();
        return e == cudaErrorMemoryAllocation ? SAILOR_E_NOMEM : SAILOR_E_CUDA;
    }
    *p = static_cast<unsigned char*>(got);
    return SAILOR_OK;
}

// The work that uses the memory is on the context's stream (or has been joined with it).
void device_free(sailor_ctx* ctx, unsigned char* p) {
    if (p) cudaFreeAsync(p, ctx->stream);
}

// A working buffer that only grows: at least `need` bytes after a successful call.
int device_grow(sailor_ctx* ctx, unsigned char** p, size_t* have, size_t need) {
    if (need <= *have) return SAILOR_OK;
    device_free(ctx, *p);
    *p = nullptr;
    *have = 0;
    const int rc = device_alloc(ctx, p, need);
    if (rc == SAILOR_OK) *have = need;
    return rc;
}

// Pinned host blocks (268 KB each): allocating one can cost a millisecond, so the process keeps a few that no context
// uses at the moment.
class HostBlocks {
  public:
    int take(sailor_ctx* ctx, HostBlock** out) {
        {
            std::lock_guard<std::mutex> hold(lock_);
            if (n_) { *out = kept_[--n_]; return SAILOR_OK; }
        }
        void* p = nullptr;
        const cudaError_t e = cudaHostAlloc(&p, sizeof(HostBlock), cudaHostAllocMapped | cudaHostAllocPortable);
        if (e != cudaSuccess) {
            ctx->last_cuda = (int)e;
            return e == cudaErrorMemoryAllocation ? SAILOR_E_NOMEM : SAILOR_E_CUDA;
        }
        *out = static_cast<HostBlock*>(p);
        return SAILOR_OK;
    }
    void give_back(HostBlock* b) {
        if (!b) return;
        {
            std::lock_guard<std::mutex> hold(lock_);
            if (n_ < KEEP) { kept_[n_++] = b; return; }
        }
        cudaFreeHost(b);
    }

  private:
    static constexpr int KEEP = 8;
    std::mutex lock_;
    HostBlock* kept_[KEEP] = {};
    int n_ = 0;
};
HostBlocks g_host_blocks;

struct DeviceGuard {
    int prev = -1;
    explicit DeviceGuard(int dev) {
        cudaGetDevice(&prev);
        if (prev != dev) cudaSetDevice(dev);
        else prev = -1;
    }
    ~DeviceGuard() {
        if (prev >= 0) cudaSetDevice(prev);
    }
};

float span_ms(const DeviceSpan& s) { return s.end > s.start ? (float)((double)(s.end - s.start) * 1e-6) : 0.f; }

bool finite_nonneg(const double* p, size_t n) {
    for (size_t i = 0; i < n; ++i)
        if (!(p[i] >= 0.0) || std::isinf(p[i])) return false;
    return true;
}

uint32_t align16(uint32_t x) { return (x + 15u) & ~15u; }

template <typename T>
uint32_t put(std::vector<unsigned char>& blob, const T* src, size_t n) {
    const uint32_t off = align16((uint32_t)blob.size());
    blob.resize(off + n * sizeof(T));
    if (src) memcpy(blob.data() + off, src, n * sizeof(T));
    return off;
}

int check_space(const sailor_ctx* ctx, const sailor_space* s) {
    if (!ctx || !s) return SAILOR_E_ARG;
    if (s->n_p == 0 || s->n_mbs == 0 || s->n_tp == 0 || s->n_rc == 0 || s->n_d == 0) return SAILOR_E_ARG;
    if (s->n_p > SAILOR_NP_MAX || s->n_mbs > SAILOR_MBS_MAX || s->n_tp > SAILOR_TP_MAX || s->n_rc > 2 ||
        s->n_d > SAILOR_ND_MAX || s->seg_max < 1 || s->seg_max > SAILOR_SEG_MAX)
        return SAILOR_E_RANGE;
    for (uint32_t i = 0; i < s->n_p; ++i)
        if (s->p_values[i] < 1 || s->p_values[i] > SAILOR_P_MAX) return SAILOR_E_RANGE;
    for (uint32_t i = 0; i < s->n_mbs; ++i)
        if (s->mbs_idx[i] >= ctx->hdr.n_mbs) return SAILOR_E_RANGE;
    for (uint32_t i = 0; i < s->n_tp; ++i)
        if (s->tp_idx[i] >= ctx->hdr.n_tp) return SAILOR_E_RANGE;
    for (uint32_t i = 0; i < s->n_rc; ++i)
        if (s->rc_values[i] > 1) return SAILOR_E_RANGE;
    for (uint32_t i = 0; i < s->n_d; ++i)
        if (s->d_values[i] < 1) return SAILOR_E_RANGE;
    return SAILOR_OK;
}

SpaceDesc to_desc(const sailor_space* s) {
    SpaceDesc d;
    memset(&d, 0, sizeof(d));
    d.n_p = s->n_p; d.n_mbs = s->n_mbs; d.n_tp = s->n_tp; d.n_rc = s->n_rc; d.n_d = s->n_d; d.seg_max = s->seg_max;
    memcpy(d.p_values, s->p_values, sizeof(d.p_values));
    memcpy(d.mbs_idx, s->mbs_idx, sizeof(d.mbs_idx));
    memcpy(d.tp_idx, s->tp_idx, sizeof(d.tp_idx));
    memcpy(d.rc_values, s->rc_values, sizeof(d.rc_values));
    memcpy(d.d_values, s->d_values, sizeof(d.d_values));
    return d;
}

// Candidate count with overflow check (limit 2^63).
int space_total(const sailor_ctx* ctx, const SpaceDesc& d, uint64_t* out) {
    const uint64_t R = ctx->hdr.R;
    const uint64_t base = (uint64_t)d.n_mbs * d.n_tp * d.n_rc * d.n_d;
    unsigned __int128 n = 0;
    for (uint32_t j = 0; j < d.n_p; ++j) {
        n += (unsigned __int128)base * ipow64(R, nseg_of(d.p_values[j], d.seg_max));
        if (n >> 63) return SAILOR_E_RANGE;
    }
    *out = (uint64_t)n;
    return SAILOR_OK;
}

bool same_space(const sailor_space& a, const sailor_space& b) {
    if (a.n_p != b.n_p || a.n_mbs != b.n_mbs || a.n_tp != b.n_tp || a.n_rc != b.n_rc || a.n_d != b.n_d ||
        a.seg_max != b.seg_max)
        return false;
    return !memcmp(a.p_values, b.p_values, a.n_p) && !memcmp(a.mbs_idx, b.mbs_idx, a.n_mbs) &&
           !memcmp(a.tp_idx, b.tp_idx, a.n_tp) && !memcmp(a.rc_values, b.rc_values, a.n_rc) &&
           !memcmp(a.d_values, b.d_values, a.n_d * sizeof(uint16_t));
}

// Per-configuration chunk and flat-index offsets; uploaded once per distinct space.
int prepare_space(sailor_ctx* ctx, const sailor_space* s) {
    SpaceCache& sc = ctx->space;
    if (sc.valid && same_space(sc.key, *s)) return SAILOR_OK;
    int rc = check_space(ctx, s);
    if (rc) return rc;
    SpaceDesc d = to_desc(s);
    uint64_t total = 0;
    rc = space_total(ctx, d, &total);
    if (rc) return rc;
    const uint64_t R = ctx->hdr.R;
    const uint32_t per_p = d.n_mbs * d.n_tp * d.n_rc * d.n_d;
    const uint64_t n_config = (uint64_t)per_p * d.n_p;
    if (n_config > (1u << 24)) return SAILOR_E_RANGE;
    std::vector<uint32_t> cs(n_config + 1);
    std::vector<uint64_t> fb(n_config);
    uint64_t chunks = 0, flat = 0;
    uint32_t p_max = 0;
    for (uint32_t j = 0; j < d.n_p; ++j) {
        const uint32_t nseg = nseg_of(d.p_values[j], d.seg_max);
        p_max = d.p_values[j] > p_max ? d.p_values[j] : p_max;
        const uint64_t items = ipow64(R, nseg - 1);
        const uint64_t per_cfg = (items + PLAN_THREADS - 1) / PLAN_THREADS;
        for (uint32_t c = 0; c < per_p; ++c) {
            cs[(size_t)j * per_p + c] = (uint32_t)chunks;
            fb[(size_t)j * per_p + c] = flat;
            chunks += per_cfg;
            flat += items * R;
            if (chunks >= 0xfff00000ull) return SAILOR_E_RANGE;
        }
    }
    cs[n_config] = (uint32_t)chunks;
    const size_t smem = plan_smem_bytes(ctx->hdr.static_bytes, p_max, ctx->hdr.T, ctx->hdr.Z, (uint32_t)n_config);
    if (smem > (size_t)PLAN_SMEM_CEILING) return SAILOR_E_RANGE;

    sc.valid = false;
    sc.cache_head16 = cache_head16();
    sc.cache_arr16 = cache_arr16(ctx->hdr.T, ctx->hdr.Z);
    const bool with_waves = n_config <= WAVE_CONFIG_MAX;
    // the tables of every configuration, built once: later searches copy them instead of building them
    const size_t cache_bytes = n_config * 16 * ((size_t)sc.cache_head16 + sc.cache_arr16);
    bool with_cache = cache_bytes <= CFG_CACHE_MAX_BYTES;
    unsigned long long* d_closed = nullptr;
    auto carve_space = [&](unsigned char* base) {
        Bump bump{base};
        d_closed = bump.take<unsigned long long>(3);
        sc.d_chunk_start = bump.take<uint32_t>(n_config + 1);
        sc.d_flat_base = bump.take<uint64_t>(n_config);
        sc.d_live_start = bump.take<uint32_t>(n_config + 1);
        sc.d_cfg_closed = with_waves ? bump.take<unsigned long long>(n_config * 3) : nullptr;
        sc.d_wave_start = with_waves ? bump.take<uint32_t>(n_config + 1) : nullptr;
        sc.d_cfg_best = with_waves ? bump.take<unsigned long long>(n_config) : nullptr;
        sc.d_groups = with_waves ? bump.take<GroupState>(n_config / d.n_d) : nullptr;
        sc.d_cfg_cache = with_cache ? bump.take<uint4>(cache_bytes / 16) : nullptr;
        return bump.at;
    };
    device_free(ctx, sc.d_mem);
    sc.d_mem = nullptr;
    if (device_alloc(ctx, &sc.d_mem, carve_space(nullptr)) != SAILOR_OK) {
        with_cache = false;                // no room for the tables: searches build them themselves
        rc = device_alloc(ctx, &sc.d_mem, carve_space(nullptr));
        if (rc) return rc;
    }
    carve_space(sc.d_mem);
    // survey the space: chunk and flat-index offsets, live chunks per configuration, the closed-form class counts
    CU(ctx, cudaMemsetAsync(d_closed, 0, 3 * sizeof(unsigned long long), ctx->stream));
    survey_kernel<<<(uint32_t)std::min<uint64_t>(n_config, 2048), SURVEY_THREADS, 0, ctx->stream>>>(
        ctx->d_blob, d, (uint32_t)n_config, sc.d_live_start, sc.d_chunk_start, sc.d_flat_base, d_closed, sc.d_cfg_closed);
    CU(ctx, cudaGetLastError());
    SurveyOut* d_survey = nullptr;
    CU(ctx, cudaHostGetDevicePointer(reinterpret_cast<void**>(&d_survey), &ctx->host->survey, 0));
    live_scan_kernel<<<1, SCAN_THREADS, 0, ctx->stream>>>(sc.d_live_start, (uint32_t)n_config, d_closed, d_survey);
    CU(ctx, cudaGetLastError());
    if (sc.d_cfg_cache) {
        // (setting the attribute twice from two threads is harmless: both set the same value)
        static std::atomic<bool> optin_done[64];
        const bool tracked = ctx->device >= 0 && ctx->device < 64;
        if (!tracked || !optin_done[ctx->device].load(std::memory_order_acquire)) {
            CU(ctx, cudaFuncSetAttribute(cfg_cache_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, PLAN_SMEM_CEILING));
            if (tracked) optin_done[ctx->device].store(true, std::memory_order_release);
        }
        PlanParams pp;
        memset(&pp, 0, sizeof(pp));
        pp.blob = ctx->d_blob;
        memcpy(pp.avail, ctx->h_avail, sizeof(pp.avail));
        pp.ctrl = ctx->d_ctrl;
        pp.cfg_flat_base = sc.d_flat_base;
        pp.sp = d;
        pp.n_config = (uint32_t)n_config;
        pp.p_max = p_max;
        pp.live_mode = 1;                  // the lists of usable digits are part of a record
        pp.min_tp_only = 1;                // and so are the masks of the smaller tensor-parallel degrees
        pp.cache_head16 = sc.cache_head16;
        pp.cache_arr16 = sc.cache_arr16;
        const uint32_t grid = (uint32_t)(n_config < (uint64_t)ctx->sm_count * 2 ? n_config : (uint64_t)ctx->sm_count * 2);
        cfg_cache_kernel<<<grid, PLAN_THREADS, smem, ctx->stream>>>(pp, sc.d_cfg_cache);
        CU(ctx, cudaGetLastError());
    }
    CU(ctx, stream_sync(ctx));             // the host needs the number of live chunks
    sc.live_chunks = ctx->host->survey.live_chunks;
    memcpy(sc.closed, ctx->host->survey.closed, sizeof(sc.closed));
    sc.key = *s;
    sc.desc = d;
    sc.n_config = (uint32_t)n_config;
    sc.n_chunks = (uint32_t)chunks;
    sc.n_total = total;
    sc.p_max = p_max;
    sc.chunk_start.swap(cs);
    sc.flat_base.swap(fb);
    sc.smem = smem;
    sc.smem_screen = plan_smem_bytes(ctx->hdr.static_bytes, p_max, ctx->hdr.T, ctx->hdr.Z, (uint32_t)n_config, true);
    sc.valid = true;
    for (uint32_t& g : ctx->grid_of) g = 0;
    return SAILOR_OK;
}

// Chunk that contains flat index f (f < n_total) of a configuration whose items are taken in flat order.
uint32_t chunk_of(const sailor_ctx* ctx, uint64_t f) {
    const SpaceCache& sc = ctx->space;
    uint32_t lo = 0, hi = sc.n_config;
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) / 2;
        if (sc.flat_base[mid] <= f) lo = mid; else hi = mid;
    }
    const uint64_t item = (f - sc.flat_base[lo]) / ctx->hdr.R;
    return sc.chunk_start[lo] + (uint32_t)(item / PLAN_THREADS);
}

constexpr int PLAN_VARIANTS = 30;      // (objective x constraint x fused, then the three screened kernels) x every candidate or not

uint32_t variant_of(uint32_t obj, bool constr, bool fused, bool eval_all, bool screen = false) {
    return (screen ? 12 + obj : (obj * 2 + (constr ? 1 : 0)) * 2 + (fused ? 1 : 0)) * 2 + (eval_all ? 1 : 0);
}

PlanKernel pick_kernel(uint32_t obj, bool constr, bool fused, bool eval_all, bool screen = false) {
    switch (obj) {
        case SAILOR_OBJ_MAX_THROUGHPUT: return plan_kernel_of<SAILOR_OBJ_MAX_THROUGHPUT>(constr, fused, screen, eval_all);
        case SAILOR_OBJ_MIN_COST: return plan_kernel_of<SAILOR_OBJ_MIN_COST>(constr, fused, screen, eval_all);
        default: return plan_kernel_of<SAILOR_OBJ_MAX_THROUGHPUT_PER_USD>(constr, fused, screen, eval_all);
    }
}

// Searches of up to this many chunks per resident block end their pass inside the search kernel; longer ones
// launch finish_kernel after it.
constexpr uint32_t FUSED_CHUNKS_PER_BLOCK = 256;

// The dynamic shared-memory opt-in belongs to the kernel (per device), not to a context: raise it
// once per (device, variant) to the ceiling every space is checked against, so that contexts
// with different table sizes cannot lower it under one another.
// The flags are atomic: contexts on different host threads may get here together, and setting the
// attribute twice to the same value is harmless.
std::atomic<bool> g_optin_done[64][PLAN_VARIANTS];

int smem_optin(sailor_ctx* ctx, PlanKernel kern, uint32_t variant) {
    const bool tracked = ctx->device >= 0 && ctx->device < 64;
    if (tracked && g_optin_done[ctx->device][variant].load(std::memory_order_acquire)) return SAILOR_OK;
    CU(ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, PLAN_SMEM_CEILING));
    if (tracked) g_optin_done[ctx->device][variant].store(true, std::memory_order_release);
    return SAILOR_OK;
}

// Enqueue one search pass on the context's stream: the search kernel, whose last block also merges the
// blocks' lists and writes the results (no separate merge launch, no clearing from the host).
//
// With SAILOR_FLAG_DEGREE_ORDER (whole space, live layout) the search runs as n_d waves: a one-block
// step kernel applies the H3/H4 rule to the previous wave's per-configuration bests and lays out the
// next wave's chunks, then the search kernel evaluates them; every block carries its list from wave
// to wave, and the last wave's launch ends the pass.
int enqueue_pass(sailor_ctx* ctx, uint32_t obj, double budget, bool budget_from_ctrl, double min_rate,
                 uint32_t flags, uint64_t lo, uint64_t hi, bool live, uint32_t k, double next_budget_factor,
                 uint32_t* n_launches, bool* launched) {
    SpaceCache& sc = ctx->space;
    const bool waves = (flags & SAILOR_FLAG_DEGREE_ORDER) != 0;
    // the counters start from the values the last finished pass (or the host, after a failure) left them at
    PlanParams pp;
    memset(&pp, 0, sizeof(pp));
    pp.blob = ctx->d_blob;
    memcpy(pp.avail, ctx->h_avail, sizeof(pp.avail));
    pp.cfg_chunk_start = sc.d_chunk_start;
    pp.cfg_flat_base = sc.d_flat_base;
    pp.ctrl = ctx->d_ctrl;
    pp.partial = ctx->d_partial;
    pp.partial_n = ctx->d_partial_n;
    pp.sp = sc.desc;
    pp.n_config = sc.n_config;
    pp.flat_lo = lo;
    pp.flat_hi = hi;
    pp.k = k;
    pp.min_tp_only = (flags & SAILOR_FLAG_MIN_TP_ONLY) ? 1u : 0u;
    pp.cfg_cache = sc.d_cfg_cache;
    pp.cache_head16 = sc.cache_head16;
    pp.cache_arr16 = sc.cache_arr16;
    pp.budget_from_ctrl = budget_from_ctrl ? 1u : 0u;
    pp.p_max = sc.p_max;
    pp.budget = budget;
    pp.min_rate = min_rate;
    pp.out = ctx->d_out_mapped;        // the block that ends the pass writes the results straight into pinned host memory
    pp.finish = 1;
    pp.ticket = ctx->ticket;
    pp.first = *n_launches == 0 && !waves ? 1u : 0u;
    pp.next_budget_factor = next_budget_factor;
    pp.cost_only = next_budget_factor > 0.0 ? 1u : 0u;
    uint32_t grid = 0;
    if (waves) {                   // the chunk table and the chunk count of each wave are written on the device
        pp.cfg_chunk_start = sc.d_wave_start;
        pp.live_mode = 1;
        pp.chunk_lo = 0;
        pp.chunk_hi = 1;                           // the waves always run: they also gather the class counts
        pp.chunk_hi_dev = &ctx->d_ctrl->wave_chunks;
        pp.cfg_best = sc.d_cfg_best;
    } else if (live) {                    // whole space, pruning on: only chunks of live prefixes exist
        pp.cfg_chunk_start = sc.d_live_start;
        pp.live_mode = 1;
        pp.chunk_lo = 0;
        pp.chunk_hi = sc.live_chunks;
    } else if (hi > lo) {                 // a configuration that a range holds a part of is taken in flat order (run_items)
        pp.chunk_lo = chunk_of(ctx, lo);
        pp.chunk_hi = chunk_of(ctx, hi - 1) + 1;
    }
    if (pp.chunk_hi > pp.chunk_lo) {
        const uint32_t n_chunks = waves ? sc.live_chunks : pp.chunk_hi - pp.chunk_lo;
        const bool constr = budget_from_ctrl || budget > 0.0 || min_rate > 0.0;
        const bool screen = (flags & SAILOR_FLAG_F32_SCREEN) != 0;
        const bool fused = !screen && n_chunks <= FUSED_CHUNKS_PER_BLOCK * 2u * (uint32_t)ctx->sm_count;
        const bool eval_all = (flags & SAILOR_FLAG_EVAL_ALL) != 0;
        PlanKernel kern = pick_kernel(obj, constr, fused, eval_all, screen);
        const uint32_t variant = variant_of(obj, constr, fused, eval_all, screen);
        const size_t smem_k = screen ? sc.smem_screen : sc.smem;
        if (smem_k > (size_t)PLAN_SMEM_CEILING) return SAILOR_E_RANGE;
        pp.screen = screen ? 1u : 0u;
        uint32_t& resident = ctx->grid_of[variant];
        if (resident == 0) {       // once per (space, kernel variant): size the grid
            int rc_opt = smem_optin(ctx, kern, variant);
            if (rc_opt) return rc_opt;
            int per_sm = 0;
            CU(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, PLAN_THREADS, smem_k));
            if (per_sm < 1) return SAILOR_E_RANGE;
            resident = (uint32_t)per_sm * (uint32_t)ctx->sm_count;
            if (resident > ctx->max_grid) resident = ctx->max_grid;
        }
        grid = n_chunks < resident ? (n_chunks ? n_chunks : 1u) : resident;
        const uint32_t batch = n_chunks / (grid * 32u);
        pp.batch = batch < 1 ? 1 : (batch > 16 ? 16 : batch);
        if (!waves) {
            kern<<<grid, PLAN_THREADS, smem_k, ctx->stream>>>(pp);
            CU(ctx, cudaGetLastError());
            ++*n_launches;
        } else {
            grid = resident < sc.live_chunks ? resident : (sc.live_chunks ? sc.live_chunks : 1u);   // the same blocks in every wave
            WaveParams wp;
            memset(&wp, 0, sizeof(wp));
            wp.live_start = sc.d_live_start;
            wp.cfg_closed = sc.d_cfg_closed;
            wp.wave_start = sc.d_wave_start;
            wp.cfg_best = sc.d_cfg_best;
            wp.groups = sc.d_groups;
            wp.ctrl = ctx->d_ctrl;
            wp.out = ctx->d_out_mapped;
            wp.n_config = sc.n_config;
            wp.n_d = sc.desc.n_d;
            // H3: largest degree first when throughput is maximised; H4: smallest first when cost is minimised
            const bool descending = obj == SAILOR_OBJ_MAX_THROUGHPUT;
            for (uint32_t j = 0; j < wp.n_d; ++j) wp.order[j] = (uint8_t)j;
            for (uint32_t a = 1; a < wp.n_d; ++a) {        // stable insertion sort by degree
                const uint8_t x = wp.order[a];
                uint32_t b = a;
                while (b > 0 && (descending ? sc.desc.d_values[wp.order[b - 1]] < sc.desc.d_values[x]
                                            : sc.desc.d_values[wp.order[b - 1]] > sc.desc.d_values[x])) {
                    wp.order[b] = wp.order[b - 1];
                    --b;
                }
                wp.order[b] = x;
            }
            for (uint32_t w = 0; w < wp.n_d; ++w) {
                wp.wave = w;
                wp.first = *n_launches == 0 ? 1u : 0u;
                wave_step_kernel<<<1, WAVE_THREADS, 0, ctx->stream>>>(wp);
                CU(ctx, cudaGetLastError());
                pp.carry_lists = w ? 1u : 0u;
                pp.finish = (w + 1 == wp.n_d) ? 1u : 0u;       // the last wave's launch ends the pass
                kern<<<grid, PLAN_THREADS, sc.smem, ctx->stream>>>(pp);
                CU(ctx, cudaGetLastError());
                *n_launches += 2;
            }
        }
        if (!fused) {              // the end of the pass as a launch of its own
            finish_kernel<<<1, PLAN_THREADS, ctx->hdr.static_bytes + sizeof(uint32_t) * SAILOR_K_MAX, ctx->stream>>>(pp, grid);
            CU(ctx, cudaGetLastError());
            ++*n_launches;
        }
    }
    *launched = grid != 0;
    return SAILOR_OK;
}

// End of a host-side batch call: wait, and report (and clear) what the batch kernels left in their error word.  The word
// is pinned host memory that they write on a fault only, so looking at it costs nothing.  Device-side batch calls only
// enqueue work; a fault in one of them is reported here as well, by the next host-side call of whatever size.
int finish_host_batch(sailor_ctx* ctx) {
    CU(ctx, stream_sync(ctx));
    volatile unsigned int* word = &ctx->host->sim_error;
    const unsigned int err = *word;
    *word = 0;
    return err == 0 ? SAILOR_OK : (err & SIM_ERR_DEVICE) ? SAILOR_E_DEVICE : SAILOR_E_RANGE;
}

// A host-side batch: records of `rec_bytes` in, four result arrays out (any may be NULL).  The batch goes through
// the device in chunks that take turns in HOST_SLOTS staging slots: a chunk's records are copied in and evaluated
// on the context's stream, its results leave on a second stream while the next chunk comes in, so that the two
// directions of the host link carry data at the same time; a slot is filled again only after its results have
// left.  The staging memory therefore does not grow with the batch beyond HOST_SLOTS chunks.  Records are checked
// by the kernel that reads them (`launch` passes the error word along, and a record outside its tables sets
// SIM_ERR_BAD_RECORD in it).  `launch(d_records, m, d_t, d_m, d_c, d_s, error)` enqueues the evaluation of m records on
// the context's stream.
constexpr uint64_t HOST_CHUNK_RECORDS = 1u << 19, HOST_CHUNK_BYTES = 1u << 26;
constexpr uint32_t HOST_SLOTS = 3;
int upload_availability(sailor_ctx* ctx);

// A host batch of up to HOST_SMALL_BYTES: its records go through the context's pinned block in one copy, the kernel writes
// the results straight back into that block.  1 000 records: 96 us with pageable copies each way (four of results,
// one of the error word), 61 with one copy back, 54 this way; a tenth of that is the host's own copying, which larger batches
// would pay instead of the driver's.
template <class Launch>
int host_batch_small(sailor_ctx* ctx, const unsigned char* recs, size_t rec_bytes, uint64_t n, double* t_iter, uint64_t* peak_mem,
                     double* cost, uint32_t* status, Launch launch) {
    int rc = device_grow(ctx, &ctx->d_stage, &ctx->stage_bytes, HOST_SMALL_BYTES);
    if (rc == SAILOR_OK) rc = upload_availability(ctx);
    if (rc != SAILOR_OK) return rc;
    unsigned char* const h_recs = ctx->host->batch;            // records, t_iter, cost, peak_mem, status
    unsigned char* const h_out = h_recs + (n * rec_bytes + 15) / 16 * 16;
    double* t = nullptr;
    CU(ctx, cudaHostGetDevicePointer(reinterpret_cast<void**>(&t), h_out, 0));
    memcpy(h_recs, recs, n * rec_bytes);
    CU(ctx, cudaMemcpyAsync(ctx->d_stage, h_recs, n * rec_bytes, cudaMemcpyHostToDevice, ctx->stream));
    rc = launch(ctx->d_stage, n, t_iter ? t : nullptr, peak_mem ? reinterpret_cast<uint64_t*>(t + 2 * n) : nullptr,
                cost ? t + n : nullptr, status ? reinterpret_cast<uint32_t*>(t + 3 * n) : nullptr, ctx->d_sim_error);
    const int rc_end = finish_host_batch(ctx);                 // the pinned block is free again, whatever happened
    if (rc != SAILOR_OK) return rc;
    if (rc_end == SAILOR_E_CUDA) return rc_end;
    if (t_iter) memcpy(t_iter, h_out, 8 * n);
    if (cost) memcpy(cost, h_out + 8 * n, 8 * n);
    if (peak_mem) memcpy(peak_mem, h_out + 16 * n, 8 * n);
    if (status) memcpy(status, h_out + 24 * n, 4 * n);
    return rc_end;
}

// A second stream of the context and the events around it, made when a call first needs them.
int side_stream(sailor_ctx* ctx) {
    if (ctx->out_stream) return SAILOR_OK;
    for (cudaEvent_t* e : {&ctx->ev_chunk, &ctx->ev_join, &ctx->ev_slot[0], &ctx->ev_slot[1], &ctx->ev_slot[2]})
        if (!*e) CU(ctx, cudaEventCreateWithFlags(e, cudaEventDisableTiming));
    CU(ctx, cudaStreamCreateWithFlags(&ctx->out_stream, cudaStreamNonBlocking));
    return SAILOR_OK;
}

template <class Launch>
int host_batch(sailor_ctx* ctx, const unsigned char* recs, size_t rec_bytes, uint64_t n, double* t_iter, uint64_t* peak_mem,
               double* cost, uint32_t* status, Launch launch) {
    if (n <= (HOST_SMALL_BYTES - 32) / (rec_bytes + 28))
        return host_batch_small(ctx, recs, rec_bytes, n, t_iter, peak_mem, cost, status, launch);
    uint64_t chunk = HOST_CHUNK_BYTES / rec_bytes;             // records per chunk: 64 MB of records, 2^19 at most
    chunk = chunk > HOST_CHUNK_RECORDS ? HOST_CHUNK_RECORDS : chunk;
    const bool split = n > chunk;
    const uint64_t slot_records = split ? chunk : n;
    const size_t slot_bytes = (slot_records * (rec_bytes + 32) + 255) / 256 * 256;
    const uint64_t n_chunks = (n + chunk - 1) / chunk;
    const size_t need = slot_bytes * (split ? (n_chunks < HOST_SLOTS ? n_chunks : HOST_SLOTS) : 1);
    {
        const int rc_mem = device_grow(ctx, &ctx->d_stage, &ctx->stage_bytes, need);
        if (rc_mem) return rc_mem;
    }
    if (split) {
        const int rc_side = side_stream(ctx);
        if (rc_side) return rc_side;
    }
    {
        const int rc_up = upload_availability(ctx);
        if (rc_up) return rc_up;
    }
    cudaStream_t out = split ? ctx->out_stream : ctx->stream;
    int rc = SAILOR_OK;
    cudaError_t ce = cudaSuccess;
    uint64_t c = 0;
    for (uint64_t off = 0; off < n && ce == cudaSuccess && rc == SAILOR_OK; off += chunk, ++c) {
        const uint64_t m = n - off < chunk ? n - off : chunk;
        const uint32_t slot = (uint32_t)(c % HOST_SLOTS);
        unsigned char* base = ctx->d_stage + (split ? slot * slot_bytes : 0);
        double* d_t = reinterpret_cast<double*>(base);
        double* d_c = reinterpret_cast<double*>(base + 8 * slot_records);
        uint64_t* d_m = reinterpret_cast<uint64_t*>(base + 16 * slot_records);
        uint32_t* d_s = reinterpret_cast<uint32_t*>(base + 24 * slot_records);
        unsigned char* d_recs = base + 32 * slot_records;
        if (split && c >= HOST_SLOTS)                          // the slot's earlier results have to be out first
            if ((ce = cudaStreamWaitEvent(ctx->stream, ctx->ev_slot[slot], 0)) != cudaSuccess) break;
        ce = cudaMemcpyAsync(d_recs, recs + off * rec_bytes, m * rec_bytes, cudaMemcpyHostToDevice, ctx->stream);
        if (ce != cudaSuccess) break;
        rc = launch(d_recs, m, d_t, d_m, d_c, d_s, ctx->d_sim_error);
        if (rc != SAILOR_OK) break;
        if (split) {
            if ((ce = cudaEventRecord(ctx->ev_chunk, ctx->stream)) != cudaSuccess) break;
            if ((ce = cudaStreamWaitEvent(out, ctx->ev_chunk, 0)) != cudaSuccess) break;
        }
        if (t_iter && ce == cudaSuccess) ce = cudaMemcpyAsync(t_iter + off, d_t, 8 * m, cudaMemcpyDeviceToHost, out);
        if (cost && ce == cudaSuccess) ce = cudaMemcpyAsync(cost + off, d_c, 8 * m, cudaMemcpyDeviceToHost, out);
        if (peak_mem && ce == cudaSuccess) ce = cudaMemcpyAsync(peak_mem + off, d_m, 8 * m, cudaMemcpyDeviceToHost, out);
        if (status && ce == cudaSuccess) ce = cudaMemcpyAsync(status + off, d_s, 4 * m, cudaMemcpyDeviceToHost, out);
        if (split && ce == cudaSuccess) ce = cudaEventRecord(ctx->ev_slot[slot], out);
    }
    if (split) {                   // whatever happened, the context's stream waits for what the second one was given
        cudaError_t cj = cudaEventRecord(ctx->ev_join, out);
        if (cj == cudaSuccess) cj = cudaStreamWaitEvent(ctx->stream, ctx->ev_join, 0);
        if (cj != cudaSuccess) { cudaStreamSynchronize(out); if (ce == cudaSuccess) ce = cj; }
    }
    const int rc_end = finish_host_batch(ctx);                 // waits for everything enqueued above
    if (ce != cudaSuccess) { ctx->last_cuda = (int)ce; return SAILOR_E_CUDA; }
    return rc != SAILOR_OK ? rc : rc_end;
}

// The device copy of the availability snapshot, for kernels that read it through a pointer.
int upload_availability(sailor_ctx* ctx) {
    if (!ctx->avail_dirty) return SAILOR_OK;
    CU(ctx, cudaEventRecord(ctx->evh0, ctx->stream));
    CU(ctx, cudaMemcpyAsync(ctx->d_avail, ctx->h_avail, ctx->hdr.R * sizeof(uint16_t), cudaMemcpyHostToDevice, ctx->stream));
    CU(ctx, cudaEventRecord(ctx->evh1, ctx->stream));
    ctx->avail_epoch = ctx->sync_epoch;
    ctx->h2d_fresh = true;
    ctx->avail_dirty = false;
    return SAILOR_OK;
}

}  // namespace

// ---- C ABI ------------------------------------------------------------------------------------

extern "C" {

const char* sailor_strerror(int code) {
    switch (code) {
        case SAILOR_OK: return "ok";
        case SAILOR_E_ARG: return "invalid argument";
        case SAILOR_E_RANGE: return "index or size out of range";
        case SAILOR_E_CUDA: return "CUDA call failed";
        case SAILOR_E_NOMEM: return "out of memory";
        case SAILOR_E_DEVICE: return "kernel reported an internal fault";
        default: return "unknown error";
    }
}

int sailor_last_cuda_error(const sailor_ctx* ctx) { return ctx ? ctx->last_cuda : 0; }

static int create_impl(const sailor_model* m, const sailor_profile* p, const sailor_cluster* c, int cuda_device,
                       void* cuda_stream, sailor_ctx** out) {
    if (!m || !p || !c || !out) return SAILOR_E_ARG;
    *out = nullptr;
    if (!p->fwd || !p->bwd || !p->upd || !p->params || !p->act_saved || !p->act_ckpt || !p->act_work ||
        !p->p2p_bytes || !c->capacity || !c->reserved || !c->gpus_per_node || !c->price_per_hour ||
        !c->intra_alpha || !c->intra_inv_bw || !c->inter_alpha || !c->inter_inv_bw || !c->zone_alpha ||
        !c->zone_inv_bw || !c->egress)
        return SAILOR_E_ARG;
    const uint32_t T = p->n_types, Z = c->n_zones, n_tp = p->n_tp, n_mbs = p->n_mbs;
    if (T == 0 || Z == 0 || n_tp == 0 || n_mbs == 0 || T != c->n_types || m->n_blocks == 0) return SAILOR_E_ARG;
    if (m->gbs == 0 || m->heads == 0 || m->mul_factor == 0 || m->dtype_size == 0 || m->grad_dtype_size == 0)
        return SAILOR_E_ARG;
    if (T > SAILOR_T_MAX || Z > SAILOR_Z_MAX || n_tp > SAILOR_TP_MAX || n_mbs > SAILOR_MBS_MAX ||
        m->n_blocks > 4096)
        return SAILOR_E_RANGE;
    for (uint32_t i = 0; i < n_tp; ++i)
        if (p->tp_values[i] == 0) return SAILOR_E_ARG;
    for (uint32_t i = 0; i < n_mbs; ++i)
        if (p->mbs_values[i] == 0) return SAILOR_E_ARG;
    for (uint32_t g = 0; g < T; ++g)
        if (c->gpus_per_node[g] == 0) return SAILOR_E_ARG;
    const size_t n4 = (size_t)SAILOR_KINDS * T * n_tp * n_mbs, n3 = (size_t)SAILOR_KINDS * T * n_tp;
    const size_t na = (size_t)SAILOR_KINDS * n_tp * n_mbs, R = (size_t)T * Z;
    if (!finite_nonneg(p->fwd, n4) || !finite_nonneg(p->bwd, n4) || !finite_nonneg(p->upd, n3) ||
        !finite_nonneg(c->price_per_hour, R) || !finite_nonneg(c->intra_alpha, R) ||
        !finite_nonneg(c->intra_inv_bw, R) || !finite_nonneg(c->inter_alpha, R) ||
        !finite_nonneg(c->inter_inv_bw, R) || !finite_nonneg(c->zone_alpha, (size_t)Z * Z) ||
        !finite_nonneg(c->zone_inv_bw, (size_t)Z * Z) || !finite_nonneg(c->egress, (size_t)Z * Z))
        return SAILOR_E_ARG;
    {   // bandwidth polynomials: coefficients finite and >= 0, constant term > 0 (bandwidth stays positive)
        const double* polys[3] = {c->intra_bw_poly, c->inter_bw_poly, c->zone_bw_poly};
        const size_t counts[3] = {R, R, (size_t)Z * Z};
        for (int q = 0; q < 3; ++q) {
            if (!polys[q]) continue;
            if (!finite_nonneg(polys[q], 4 * counts[q])) return SAILOR_E_ARG;
            for (size_t j = 0; j < counts[q]; ++j)
                if (!(polys[q][4 * j] > 0.0)) return SAILOR_E_ARG;
        }
    }

    sailor_ctx* ctx = new (std::nothrow) sailor_ctx();
    if (!ctx) return SAILOR_E_NOMEM;
    ctx->device = cuda_device;
    ctx->stream = (cudaStream_t)cuda_stream;
    DeviceGuard guard(cuda_device);

    // pack the blob: header, raw tables, cluster tables (static part), then the chains
    TabHdr& h = ctx->hdr;
    memset(&h, 0, sizeof(h));
    h.n_blocks = m->n_blocks; h.has_embed = m->has_embed ? 1 : 0; h.has_head = m->has_head ? 1 : 0;
    h.heads = m->heads; h.gbs = m->gbs;
    h.mul_bytes = (uint64_t)m->mul_factor * m->dtype_size;
    h.grad_bytes = m->grad_dtype_size;
    h.T = T; h.Z = Z; h.R = (uint32_t)R; h.n_tp = n_tp; h.n_mbs = n_mbs; h.chain_len = m->n_blocks + 1;
    memcpy(h.tp_values, p->tp_values, n_tp * sizeof(uint32_t));
    memcpy(h.mbs_values, p->mbs_values, n_mbs * sizeof(uint32_t));
    for (uint32_t g = 0; g < T; ++g) {
        h.gpn[g] = c->gpus_per_node[g];
        h.capacity[g] = c->capacity[g];
        h.reserved[g] = c->reserved[g];
    }
    for (int k = 0; k < SAILOR_KINDS; ++k) h.params[k] = p->params[k];
    for (uint32_t i = 0; i < n_tp; ++i)
        if (m->heads % p->tp_values[i] == 0) h.heads_ok |= 1u << i;

    std::vector<unsigned char> blob(sizeof(TabHdr));
    h.off_fwd = put(blob, p->fwd, n4);
    h.off_bwd = put(blob, p->bwd, n4);
    h.off_upd = put(blob, p->upd, n3);
    h.off_saved = put(blob, p->act_saved, na);
    h.off_ckpt = put(blob, p->act_ckpt, na);
    h.off_work = put(blob, p->act_work, na);
    h.off_p2p = put(blob, p->p2p_bytes, n_mbs);
    std::vector<double> price_s(R);
    for (size_t d = 0; d < R; ++d) price_s[d] = c->price_per_hour[d] / 3600.0;   // dollars per GPU-second
    h.off_price_s = put(blob, price_s.data(), R);
    h.off_intra_a = put(blob, c->intra_alpha, R);
    h.off_intra_i = put(blob, c->intra_inv_bw, R);
    h.off_inter_a = put(blob, c->inter_alpha, R);
    h.off_inter_i = put(blob, c->inter_inv_bw, R);
    h.off_zone_a = put(blob, c->zone_alpha, (size_t)Z * Z);
    h.off_zone_i = put(blob, c->zone_inv_bw, (size_t)Z * Z);
    h.off_egress = put(blob, c->egress, (size_t)Z * Z);
    h.off_intra_p = c->intra_bw_poly ? put(blob, c->intra_bw_poly, 4 * R) : 0;
    h.off_inter_p = c->inter_bw_poly ? put(blob, c->inter_bw_poly, 4 * R) : 0;
    h.off_zone_p = c->zone_bw_poly ? put(blob, c->zone_bw_poly, 4 * (size_t)Z * Z) : 0;
    h.static_bytes = align16((uint32_t)blob.size());
    blob.resize(h.static_bytes);
    const size_t c4 = (size_t)2 * T * n_tp * n_mbs * h.chain_len, c3 = (size_t)2 * T * n_tp * h.chain_len;
    const size_t n_comp = (size_t)4 * h.chain_len;
    const size_t cmp_fb = n_comp * T * n_tp * n_mbs * 2, cmp_upd = n_comp * T * n_tp, cmp_mem = n_comp * n_tp * n_mbs * 2 * 2,
                 cmp_grad = n_comp * n_tp;
    if (h.static_bytes + (2 * c4 + c3 + cmp_fb + cmp_upd + cmp_mem + cmp_grad + n_comp) * sizeof(double) +
                cmp_fb * sizeof(PieceRec) + (2 * R + (size_t)Z * Z) * n_mbs * sizeof(double) + 512 > (1ull << 30) ||
        h.static_bytes > 96 * 1024) {
        delete ctx;
        return SAILOR_E_RANGE;
    }
    // what the kernels below form from the static part lies behind it, on the device only
    size_t at = h.static_bytes;
    auto reserve = [&](size_t bytes, size_t align) {
        at = (at + align - 1) / align * align;
        const uint32_t off = (uint32_t)at;
        at += bytes;
        return off;
    };
    h.off_chain_f = reserve(c4 * 8, 16);
    h.off_chain_b = reserve(c4 * 8, 16);
    h.off_chain_u = reserve(c3 * 8, 16);
    h.off_cmp_params = reserve(n_comp * 8, 16);
    h.off_cmp_grad = reserve(cmp_grad * 8, 16);
    h.off_cmp_mem = reserve(cmp_mem * 8, 16);
    h.off_cmp_fb = reserve(cmp_fb * 8, 16);
    h.off_cmp_upd = reserve(cmp_upd * 8, 16);
    h.off_piece = reserve(cmp_fb * sizeof(PieceRec), 32);  // a table entry is one 32-byte sector
    h.off_lnk_intra2 = reserve(R * n_mbs * 8, 16);
    h.off_lnk_inter2 = reserve(R * n_mbs * 8, 16);
    h.off_lnk_zone2 = reserve((size_t)Z * Z * n_mbs * 8, 16);
    h.total_bytes = align16((uint32_t)at);
    memcpy(blob.data(), &h, sizeof(h));

    auto fail = [&](int code) { sailor_destroy(ctx); return code; };
#define CUF(call)                                                   \
    do {                                                            \
        cudaError_t e_ = (call);                                    \
        if (e_ != cudaSuccess) {                                    \
            ctx->last_cuda = (int)e_;                               \
            return fail(e_ == cudaErrorMemoryAllocation ? SAILOR_E_NOMEM : SAILOR_E_CUDA); \
        }                                                           \
    } while (0)
    CUF(cudaDeviceGetAttribute(&ctx->sm_count, cudaDevAttrMultiProcessorCount, cuda_device));
    ctx->max_grid = (uint32_t)ctx->sm_count * 8;
    int rc = g_host_blocks.take(ctx, &ctx->host);
    if (rc) return fail(rc);
    memset(static_cast<void*>(ctx->host), 0, offsetof(HostBlock, mixed));     // availability starts at zero on both sides
    ctx->h_avail = ctx->host->avail;
    ctx->h_out = &ctx->host->out;
    CUF(cudaHostGetDevicePointer(reinterpret_cast<void**>(&ctx->d_out_mapped), ctx->h_out, 0));
    CUF(cudaHostGetDevicePointer(reinterpret_cast<void**>(&ctx->d_sim_error), &ctx->host->sim_error, 0));
    auto carve_ctx = [&](unsigned char* base) {              // returns (bytes that start from zero, all bytes)
        Bump bump{base};
        ctx->d_avail = bump.take<uint16_t>(R_MAX);
        ctx->d_ctrl = bump.take<Ctrl>(1);
        ctx->d_deep_seen = bump.take<unsigned int>(1);
        const size_t zeroed = bump.at;
        ctx->d_blob = bump.take<unsigned char>(h.total_bytes);
        ctx->d_partial = bump.take<Hit>((size_t)SAILOR_K_MAX * ctx->max_grid);
        ctx->d_partial_n = bump.take<uint32_t>(ctx->max_grid);
        return std::make_pair(zeroed, bump.at);
    };
    rc = device_alloc(ctx, &ctx->d_mem, carve_ctx(nullptr).second);
    if (rc) return fail(rc);
    const size_t zeroed = carve_ctx(ctx->d_mem).first;
    CUF(cudaEventCreate(&ctx->ev0));
    CUF(cudaEventCreate(&ctx->ev1));
    CUF(cudaEventCreate(&ctx->ev2));
    CUF(cudaEventCreate(&ctx->evh0));
    CUF(cudaEventCreate(&ctx->evh1));
    CUF(cudaMemsetAsync(ctx->d_mem, 0, zeroed, ctx->stream));
    CUF(cudaMemcpyAsync(ctx->d_blob, blob.data(), h.static_bytes, cudaMemcpyHostToDevice, ctx->stream));   // returns when `blob` has been read
    ctx->h_static.swap(blob);
    {
        const uint32_t n_threads = 4 * T * n_tp * n_mbs + 2 * T * n_tp;
        chain_kernel<<<(n_threads + 127) / 128, 128, 0, ctx->stream>>>(ctx->d_blob);
        CUF(cudaGetLastError());
        const size_t n_cmp = cmp_fb;
        const uint32_t grid = (uint32_t)((n_cmp + 127) / 128 < 65536 ? (n_cmp + 127) / 128 : 65536);
        compose_kernel<<<grid, 128, 0, ctx->stream>>>(ctx->d_blob);
        CUF(cudaGetLastError());
        batch_tables_kernel<<<grid, 128, 0, ctx->stream>>>(ctx->d_blob);
        CUF(cudaGetLastError());
    }
    // both kernels stage the static tables in dynamic shared memory; the create-time limit is 96 KB
    CUF(cudaFuncSetAttribute(simulate_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024));
    CUF(cudaFuncSetAttribute(simulate_mixed_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(sizeof(MixbShared) + 2 * R_MAX * SAILOR_MBS_MAX * sizeof(double))));
    CUF(cudaFuncSetAttribute(simulate_mixed_each_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024 + (int)sizeof(MixScratch<MIX_STAGES<false>>) * MIX_WARPS<false>));
    CUF(cudaFuncSetAttribute(simulate_mixed_each_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024 + (int)sizeof(MixScratch<MIX_STAGES<true>>) * MIX_WARPS<true>));
    CUF(cudaFuncSetAttribute(finish_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (96 + 8) * 1024));
    CUF(cudaFuncSetAttribute(mixed_finish_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024 + (int)sizeof(MixFinishWarp<false>) * MIXF_WARPS<false>));
    CUF(cudaFuncSetAttribute(mixed_finish_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024 + (int)sizeof(MixFinishWarp<true>) * MIXF_WARPS<true>));
#undef CUF
    *out = ctx;
    return SAILOR_OK;
}

int sailor_destroy(sailor_ctx* ctx) {
    if (!ctx) return SAILOR_OK;
    DeviceGuard guard(ctx->device);
    if (ctx->d_mem) cudaStreamSynchronize(ctx->stream);
    for (unsigned char* p : {ctx->d_mem, ctx->space.d_mem, ctx->d_stage, ctx->d_mix, ctx->d_dp, ctx->d_dp_up}) device_free(ctx, p);
    // what the pool does not keep goes back to the device here, and not when some stream is next synchronised: another
    // allocator of the process may need it before
    cudaMemPool_t pool;
    uint64_t reserved = 0;
    if (ctx->d_mem && device_pool(ctx, &pool) == SAILOR_OK &&
        cudaMemPoolGetAttribute(pool, cudaMemPoolAttrReservedMemCurrent, &reserved) == cudaSuccess && reserved > POOL_KEEP)
        cudaStreamSynchronize(ctx->stream);
    g_host_blocks.give_back(ctx->host);
    delete ctx->mix;
    for (cudaEvent_t e : {ctx->ev0, ctx->ev1, ctx->ev2, ctx->evh0, ctx->evh1, ctx->ev_chunk, ctx->ev_join, ctx->ev_slot[0],
                          ctx->ev_slot[1], ctx->ev_slot[2]})
        if (e) cudaEventDestroy(e);
    if (ctx->out_stream) cudaStreamDestroy(ctx->out_stream);
    delete ctx;
    return SAILOR_OK;
}

int sailor_set_availability(sailor_ctx* ctx, const uint16_t* avail) {
    if (!ctx || !avail) return SAILOR_E_ARG;
    DeviceGuard guard(ctx->device);
    // A search takes the snapshot along in its launch parameters; the device copy that the other kernels read
    // through a pointer is brought up to date when one of them is next enqueued (upload_availability).  The pinned
    // buffer may still feed such a copy, unless the stream has been synchronised since.
    if (ctx->avail_epoch == ctx->sync_epoch) CU(ctx, stream_sync(ctx));
    memcpy(ctx->h_avail, avail, ctx->hdr.R * sizeof(uint16_t));
    ctx->avail_dirty = true;
    return SAILOR_OK;
}

int sailor_simulate(sailor_ctx* ctx, const sailor_plan_rec* plans, uint64_t n, int on_device, double* t_iter,
                    uint64_t* peak_mem, double* cost, uint32_t* status) {
    if (!ctx || (!plans && n)) return SAILOR_E_ARG;
    if (n == 0) return SAILOR_OK;
    if ((uintptr_t)plans % 8 != 0) return SAILOR_E_ARG;
    DeviceGuard guard(ctx->device);
    auto launch = [ctx](const sailor_plan_rec* d_plans, uint64_t m, double* d_t, uint64_t* d_m, double* d_c, uint32_t* d_s,
                        unsigned int* error, uint32_t report_bad) {
        // as many pools for every SM, and no larger ones than that takes
        const uint64_t turns = (m + (uint64_t)ctx->sm_count * BATCH_POOL - 1) / ((uint64_t)ctx->sm_count * BATCH_POOL);
        const uint64_t share = (m + ctx->sm_count * turns - 1) / (ctx->sm_count * turns);
        const uint32_t pool = (uint32_t)((share + 31) / 32 * 32);
        const uint64_t pools = (m + pool - 1) / pool;
        // groups of fewer lanes diverge less: as few as leave every group a warp of its own (1 000 records in groups of 32:
        // 32.3 us on the device, of 8: 30.9, of 4: 30.1; 45 000 records: no difference)
        uint32_t lanes = 4;
        while (lanes < 32 && pool > lanes * BATCH_WARPS) lanes *= 2;
        const uint32_t grid = (uint32_t)std::min<uint64_t>(pools, (uint64_t)ctx->sm_count);
        const BatchParams p = batch_params(ctx->hdr, ctx->d_blob);
        simulate_kernel<<<grid, BATCH_THREADS, p.smem, ctx->stream>>>(
            p, ctx->d_avail, d_plans, m, pool, lanes, d_t, d_m, d_c, d_s, error, report_bad);
        CU(ctx, cudaGetLastError());
        return (int)SAILOR_OK;
    };
    if (!on_device)                                               // records are checked by the kernel (SIM_ERR_BAD_RECORD)
        return host_batch(ctx, reinterpret_cast<const unsigned char*>(plans), sizeof(sailor_plan_rec), n, t_iter, peak_mem, cost,
                          status, [&](const unsigned char* d_recs, uint64_t m, double* d_t, uint64_t* d_m, double* d_c, uint32_t* d_s, unsigned int* error) {
                              return launch(reinterpret_cast<const sailor_plan_rec*>(d_recs), m, d_t, d_m, d_c, d_s, error, 1u);
                          });
    {
        const int rc_up = upload_availability(ctx);
        if (rc_up) return rc_up;
    }
    return launch(plans, n, t_iter, peak_mem, cost, status, ctx->d_sim_error, 0u);
}

int sailor_simulate_mixed(sailor_ctx* ctx, const sailor_mixed_plan* plans, uint64_t n, int on_device, double* t_iter,
                          uint64_t* peak_mem, double* cost, uint32_t* status) {
    return sailor_simulate_mixed_strided(ctx, plans, n, (uint32_t)sizeof(sailor_mixed_plan), on_device, t_iter, peak_mem,
                                         cost, status);
}

int sailor_simulate_mixed_strided(sailor_ctx* ctx, const void* plans_v, uint64_t n, uint32_t record_bytes, int on_device,
                                  double* t_iter, uint64_t* peak_mem, double* cost, uint32_t* status) {
    constexpr uint32_t HEAD = (uint32_t)offsetof(sailor_mixed_plan, stage);
    if (!ctx || (!plans_v && n)) return SAILOR_E_ARG;
    if (record_bytes % 8 != 0 || record_bytes < HEAD + sizeof(sailor_mixed_stage) || record_bytes > sizeof(sailor_mixed_plan))
        return SAILOR_E_ARG;
    if (n == 0) return SAILOR_OK;
    const unsigned char* plans = static_cast<const unsigned char*>(plans_v);
    if ((uintptr_t)plans % 8 != 0) return SAILOR_E_ARG;
    const uint32_t max_stages = (record_bytes - HEAD) / (uint32_t)sizeof(sailor_mixed_stage);
    DeviceGuard guard(ctx->device);
    auto launch = [ctx, record_bytes, max_stages](const unsigned char* d_plans, uint64_t m, double* d_t, uint64_t* d_m, double* d_c,
                                                  uint32_t* d_s, unsigned int* error, uint32_t report_bad) {
        MixbCall p = {};
        p.blob = ctx->d_blob; p.avail = ctx->d_avail;
        p.plans = d_plans; p.n = m; p.stride = record_bytes; p.max_stages = max_stages;
        p.t_iter = d_t; p.peak_mem = d_m; p.cost = d_c; p.status = d_s;
        p.error = error; p.deep_seen = ctx->d_deep_seen; p.report_bad = report_bad;
        if (max_stages > MIXB_P_MAX) CU(ctx, cudaMemsetAsync(ctx->d_deep_seen, 0, sizeof(unsigned int), ctx->stream));
        if (mixb_takes(ctx->hdr, max_stages, m)) {
            simulate_mixed_kernel<<<(uint32_t)std::min<uint64_t>(m, MIXB_BLOCKS * (uint64_t)ctx->sm_count), MIXB_THREADS, mixb_smem(ctx->hdr), ctx->stream>>>(mixb_params(p, ctx->hdr));
        } else {                                                 // (blocks take several plans per warp in larger batches)
            const uint64_t blocks = (m + MIX_WARPS<false> - 1) / MIX_WARPS<false>, cap = (uint64_t)ctx->sm_count * 32;
            simulate_mixed_each_kernel<false><<<(uint32_t)std::min(blocks, cap), 32 * MIX_WARPS<false>, mixed_smem<false>(ctx->hdr), ctx->stream>>>(p);
        }
        CU(ctx, cudaGetLastError());
        if (max_stages > MIXB_P_MAX) {                           // the plans of more than 32 stages, if the first launch saw any
            const uint64_t blocks = (m + MIX_WARPS<true> - 1) / MIX_WARPS<true>, cap = (uint64_t)ctx->sm_count * 16;
            simulate_mixed_each_kernel<true><<<(uint32_t)std::min(blocks, cap), 32 * MIX_WARPS<true>, mixed_smem<true>(ctx->hdr), ctx->stream>>>(p);
            CU(ctx, cudaGetLastError());
        }
        return (int)SAILOR_OK;
    };
    if (!on_device)                                               // records are checked by the kernel (SIM_ERR_BAD_RECORD)
        return host_batch(ctx, plans, record_bytes, n, t_iter, peak_mem, cost, status,
                          [&](const unsigned char* d_recs, uint64_t m, double* d_t, uint64_t* d_m, double* d_c, uint32_t* d_s, unsigned int* error) {
                              return launch(d_recs, m, d_t, d_m, d_c, d_s, error, 1u);
                          });
    {
        const int rc_up = upload_availability(ctx);
        if (rc_up) return rc_up;
    }
    return launch(plans, n, t_iter, peak_mem, cost, status, ctx->d_sim_error, 0u);
}

int sailor_space_size(const sailor_ctx* ctx, const sailor_space* s, uint64_t* n_out) {
    if (!n_out) return SAILOR_E_ARG;
    int rc = check_space(ctx, s);
    if (rc) return rc;
    return space_total(ctx, to_desc(s), n_out);
}

int sailor_decode(const sailor_ctx* ctx, const sailor_space* s, uint64_t flat, sailor_plan_rec* out) {
    if (!out) return SAILOR_E_ARG;
    int rc = check_space(ctx, s);
    if (rc) return rc;
    return decode_flat(to_desc(s), ctx->hdr.T, ctx->hdr.Z, flat, out) ? SAILOR_OK : SAILOR_E_RANGE;
}

static int plan_range_impl(sailor_ctx* ctx, const sailor_space* s, const sailor_objective* o, uint64_t flat_lo,
                           uint64_t flat_hi, uint32_t k, sailor_result* topk, uint32_t* n_found, sailor_stats* stats) {
    if (!ctx || !s || !o || !topk || !n_found || k == 0) return SAILOR_E_ARG;
    if (k > SAILOR_K_MAX || o->kind > SAILOR_OBJ_MAX_THROUGHPUT_PER_USD) return SAILOR_E_RANGE;
    if (std::isnan(o->budget_usd_per_iter) || std::isnan(o->min_iters_per_s) ||
        std::isnan(o->budget_factor_over_cheapest))
        return SAILOR_E_ARG;
    if (o->flags & ~(SAILOR_FLAG_EVAL_ALL | SAILOR_FLAG_DEGREE_ORDER | SAILOR_FLAG_MIN_TP_ONLY | SAILOR_FLAG_F32_SCREEN))
        return SAILOR_E_ARG;
    if ((o->flags & SAILOR_FLAG_F32_SCREEN) &&
        (o->budget_usd_per_iter > 0.0 || o->min_iters_per_s > 0.0 || o->budget_factor_over_cheapest > 0.0 ||
         (o->flags & SAILOR_FLAG_DEGREE_ORDER)))
        return SAILOR_E_ARG;                                   // the screen covers unconstrained searches
    DeviceGuard guard(ctx->device);
    int rc = prepare_space(ctx, s);
    if (rc) return rc;
    const uint64_t total = ctx->space.n_total;
    if (flat_hi > total) flat_hi = total;
    if (flat_lo > flat_hi) flat_lo = flat_hi;
    const bool waves = (o->flags & SAILOR_FLAG_DEGREE_ORDER) != 0;
    if (waves) {
        if (o->kind == SAILOR_OBJ_MAX_THROUGHPUT_PER_USD || (o->flags & SAILOR_FLAG_EVAL_ALL) || flat_lo != 0 ||
            flat_hi != total)
            return SAILOR_E_ARG;
        if (!ctx->space.d_cfg_closed) return SAILOR_E_RANGE;     // more configurations than the wave tables hold
    }

    uint32_t launches = 0;
    if (ctx->ctrl_dirty) {             // first search of the context, or the last one failed half-way
        CU(ctx, cudaMemsetAsync(ctx->d_ctrl, 0, sizeof(Ctrl), ctx->stream));
        CU(ctx, cudaMemsetAsync(&ctx->d_ctrl->min_cost_bits, 0x7f, 2 * sizeof(unsigned long long), ctx->stream));
    }
    ctx->ctrl_dirty = true;            // until this call has gone through
    ++ctx->ticket;
    const bool two_pass = o->budget_factor_over_cheapest > 0.0;
    // a whole-space search with pruning on walks only the prefixes the survey found live
    const bool live = !(o->flags & SAILOR_FLAG_EVAL_ALL) && flat_lo == 0 && flat_hi == total;
    bool launched = false;
    if (two_pass) {
        // cheapest feasible plan first; the block that ends that pass leaves factor * cost in ctrl->budget
        rc = enqueue_pass(ctx, SAILOR_OBJ_MIN_COST, 0.0, false, 0.0, o->flags, flat_lo, flat_hi, live, 1,
                          o->budget_factor_over_cheapest, &launches, &launched);
        if (rc) return rc;
    }
    rc = enqueue_pass(ctx, o->kind, o->budget_usd_per_iter, two_pass, o->min_iters_per_s, o->flags, flat_lo,
                      flat_hi, live, k, 0.0, &launches, &launched);
    if (rc) return rc;
    if (!launched) memset(&ctx->h_out->ctrl, 0, sizeof(Ctrl));    // an empty range: nothing ran, nothing was found
    if (launched) CU(ctx, wait_ticket(ctx, &ctx->h_out->ticket, ctx->ticket));
    else CU(ctx, stream_sync(ctx));
    ctx->ctrl_dirty = false;
    const Ctrl& cr = ctx->h_out->ctrl;
    if (cr.error) return SAILOR_E_DEVICE;
    if (cr.n_found > k) return SAILOR_E_DEVICE;               // cannot happen; never copy past the caller's k records
    *n_found = cr.n_found;
    memcpy(topk, ctx->h_out->results, sizeof(sailor_result) * cr.n_found);
    if (stats) {
        // in live mode the kernels count the evaluated candidates only; the rest is the survey's closed form
        // (in degree order: of the configurations the waves selected, summed on the device)
        const SpaceCache& sc = ctx->space;
        const bool closed_form = live && !waves;
        stats->n_total = closed_form ? sc.closed[0] : cr.stats[0];
        stats->n_invalid = closed_form ? sc.closed[1] : cr.stats[1];
        stats->n_oom = closed_form ? sc.closed[2] : cr.stats[2];
        stats->n_pruned_tp = cr.stats[6];
        stats->n_skipped = waves ? sc.closed[0] - cr.stats[0] : 0;
        stats->n_configs = sc.n_config;
        stats->n_configs_evaluated = waves ? cr.n_cfg_evaluated : sc.n_config;
        stats->n_over_avail = cr.stats[3];
        stats->n_over_constraint = cr.stats[4];
        stats->n_feasible = cr.stats[5];
        stats->budget_used = two_pass ? (launched ? cr.budget : 0.0) : o->budget_usd_per_iter;
        double mc;
        memcpy(&mc, &cr.min_cost_bits, sizeof(mc));
        stats->min_feasible_cost = cr.stats[5] ? mc : 0.0;
        stats->kernel_ms = launched ? span_ms(ctx->h_out->span) : 0.f;
        stats->n_launches = launches;
        stats->d2h_ms = 0.f;               // no copy of its own: the results were written in place
        if (ctx->h2d_fresh) {              // an upload for another entry point was enqueued before this search: complete by now
            CU(ctx, cudaEventElapsedTime(&ctx->h2d_ms, ctx->evh0, ctx->evh1));
            ctx->h2d_fresh = false;
        }
        stats->h2d_ms = ctx->h2d_ms;
    }
    return SAILOR_OK;
}

int sailor_plan(sailor_ctx* ctx, const sailor_space* s, const sailor_objective* o, uint32_t k,
                sailor_result* topk, uint32_t* n_found, sailor_stats* stats) {
    return sailor_plan_range(ctx, s, o, 0, ~0ull >> 1, k, topk, n_found, stats);
}

}  // extern "C"

// ---- search without device allocation ----------------------------------------------------------
//
// sailor_plan_range keeps its per-space index arrays in memory it allocates when a new space
// arrives.  The variant below takes every byte of working memory from one fixed array that is
// part of the library image instead, so it can serve callers that must not allocate.

namespace {

constexpr uint32_t NOALLOC_GRID_MAX = 1024;     // blocks whose partial lists fit the fixed scratch

struct NoAllocScratch {                         // layout of the fixed scratch array
    Ctrl ctrl;
    PlanOut out;
    uint32_t partial_n[NOALLOC_GRID_MAX];
    Hit partial[(size_t)NOALLOC_GRID_MAX * SAILOR_K_MAX];
    uint32_t cfg_chunk_start[SAILOR_NOALLOC_CONFIG_MAX + 1];
    uint64_t cfg_flat_base[SAILOR_NOALLOC_CONFIG_MAX];
};

// About 0.6 MB, held by every GPU that loads the library until the process exits.  In host code
// this name is only a handle for cudaGetSymbolAddress; it is never passed to a kernel.
static __device__ __align__(256) unsigned char g_noalloc_scratch[sizeof(NoAllocScratch)];
static_assert(offsetof(NoAllocScratch, partial) % 16 == 0, "the lists are read 16 bytes at a time");

constexpr int NOALLOC_DEVICES_MAX = 64;
// device address of the array, per device (atomic: two threads resolving it together store the same address)
std::atomic<NoAllocScratch*> g_noalloc_ptr[NOALLOC_DEVICES_MAX];
// resident blocks per SM of each kernel variant at a given shared-memory size, per device (0 = not asked yet)
struct OccupancyMemo { std::atomic<uint64_t> smem_and_blocks; };
OccupancyMemo g_noalloc_occ[NOALLOC_DEVICES_MAX][PLAN_VARIANTS];

// Device address of the scratch on the current device; resolved on first use per device.
int noalloc_scratch(sailor_ctx* ctx, NoAllocScratch** out) {
    if (ctx->device < 0 || ctx->device >= NOALLOC_DEVICES_MAX) return SAILOR_E_RANGE;
    NoAllocScratch* known = g_noalloc_ptr[ctx->device].load(std::memory_order_acquire);
    if (!known) {
        void* p = nullptr;
        CU(ctx, cudaGetSymbolAddress(&p, g_noalloc_scratch));
        known = static_cast<NoAllocScratch*>(p);
        g_noalloc_ptr[ctx->device].store(known, std::memory_order_release);
    }
    *out = known;
    return SAILOR_OK;
}

// One pass (clear, search with its merge) whose scratch all lies in `sc`.
int enqueue_pass_noalloc(sailor_ctx* ctx, NoAllocScratch* sc, const SpaceDesc& desc, uint32_t n_config,
                         uint32_t p_max, size_t smem, uint32_t chunk_lo, uint32_t chunk_hi, uint64_t total,
                         uint32_t obj, double budget, bool budget_from_ctrl, double min_rate, uint32_t flags,
                         uint32_t k, double next_budget_factor, uint32_t* n_launches) {
    // the array keeps the previous call's contents: counters and the work counter restart at zero
    CU(ctx, cudaMemsetAsync(&sc->ctrl, 0, offsetof(Ctrl, min_cost_bits), ctx->stream));
    CU(ctx, cudaMemsetAsync(&sc->ctrl.min_cost_bits, 0x7f, 2 * sizeof(unsigned long long), ctx->stream));
    PlanParams pp;
    memset(&pp, 0, sizeof(pp));
    pp.blob = ctx->d_blob;
    memcpy(pp.avail, ctx->h_avail, sizeof(pp.avail));
    pp.cfg_chunk_start = sc->cfg_chunk_start;
    pp.cfg_flat_base = sc->cfg_flat_base;
    pp.ctrl = &sc->ctrl;
    pp.partial = sc->partial;
    pp.partial_n = sc->partial_n;
    pp.sp = desc;
    pp.n_config = n_config;
    pp.flat_lo = 0;
    pp.flat_hi = total;
    pp.k = k;
    pp.min_tp_only = (flags & SAILOR_FLAG_MIN_TP_ONLY) ? 1u : 0u;
    pp.budget_from_ctrl = budget_from_ctrl ? 1u : 0u;
    pp.p_max = p_max;
    pp.budget = budget;
    pp.min_rate = min_rate;
    pp.chunk_lo = chunk_lo;
    pp.chunk_hi = chunk_hi;
    pp.out = &sc->out;
    pp.finish = 1;
    pp.next_budget_factor = next_budget_factor;
    pp.cost_only = next_budget_factor > 0.0 ? 1u : 0u;
    const uint32_t n_chunks = chunk_hi - chunk_lo;
    const bool constr = budget_from_ctrl || budget > 0.0 || min_rate > 0.0;
    const bool eval_all = (flags & SAILOR_FLAG_EVAL_ALL) != 0;
    PlanKernel kern = pick_kernel(obj, constr, true, eval_all);
    const uint32_t variant = variant_of(obj, constr, true, eval_all);
    {
        const int rc_opt = smem_optin(ctx, kern, variant);
        if (rc_opt) return rc_opt;
    }
    // the occupancy query costs host time on a path that exists for its latency: ask once per (device, variant, size)
    int per_sm = 0;
    std::atomic<uint64_t>& memo = g_noalloc_occ[ctx->device][variant].smem_and_blocks;
    const uint64_t seen = memo.load(std::memory_order_acquire);
    if (seen && (seen >> 8) == (uint64_t)smem) per_sm = (int)(seen & 0xff);
    else {
        CU(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, PLAN_THREADS, smem));
        if (per_sm >= 1 && per_sm < 256) memo.store(((uint64_t)smem << 8) | (uint64_t)per_sm, std::memory_order_release);
    }
    if (per_sm < 1) return SAILOR_E_RANGE;
    uint32_t grid = (uint32_t)per_sm * (uint32_t)ctx->sm_count;
    if (grid > NOALLOC_GRID_MAX) grid = NOALLOC_GRID_MAX;
    if (grid > n_chunks) grid = n_chunks;
    const uint32_t batch = n_chunks / (grid * 32u);
    pp.batch = batch < 1 ? 1 : (batch > 16 ? 16 : batch);
    kern<<<grid, PLAN_THREADS, smem, ctx->stream>>>(pp);
    CU(ctx, cudaGetLastError());
    ++*n_launches;
    return SAILOR_OK;
}

}  // namespace

extern "C" int sailor_plan_noalloc(sailor_ctx* ctx, const sailor_space* s, const sailor_objective* o, uint32_t k,
                                   sailor_result* topk, uint32_t* n_found, sailor_stats* stats) {
    if (!ctx || !s || !o || !topk || !n_found || k == 0) return SAILOR_E_ARG;
    if (k > SAILOR_K_MAX || o->kind > SAILOR_OBJ_MAX_THROUGHPUT_PER_USD) return SAILOR_E_RANGE;
    if (std::isnan(o->budget_usd_per_iter) || std::isnan(o->min_iters_per_s) ||
        std::isnan(o->budget_factor_over_cheapest))
        return SAILOR_E_ARG;
    if (o->flags & ~(SAILOR_FLAG_EVAL_ALL | SAILOR_FLAG_MIN_TP_ONLY)) return SAILOR_E_ARG;   // degree order needs tables this variant has no room for
    int rc = check_space(ctx, s);
    if (rc) return rc;
    const SpaceDesc d = to_desc(s);
    uint64_t total = 0;
    rc = space_total(ctx, d, &total);
    if (rc) return rc;
    const uint32_t per_p = d.n_mbs * d.n_tp * d.n_rc * d.n_d;
    const uint64_t n_config = (uint64_t)per_p * d.n_p;
    if (n_config > SAILOR_NOALLOC_CONFIG_MAX) return SAILOR_E_RANGE;       // beyond the fixed scratch

    // per-configuration offsets, built in fixed-size host arrays (thread-local: no heap, no device memory)
    static thread_local uint32_t h_chunk_start[SAILOR_NOALLOC_CONFIG_MAX + 1];
    static thread_local uint64_t h_flat_base[SAILOR_NOALLOC_CONFIG_MAX];
    const uint64_t R = ctx->hdr.R;
    uint64_t chunks = 0, flat = 0;
    uint32_t p_max = 0;
    for (uint32_t j = 0; j < d.n_p; ++j) {
        const uint32_t nseg = nseg_of(d.p_values[j], d.seg_max);
        p_max = d.p_values[j] > p_max ? d.p_values[j] : p_max;
        const uint64_t items = ipow64(R, nseg - 1);
        const uint64_t per_cfg = (items + PLAN_THREADS - 1) / PLAN_THREADS;
        for (uint32_t c = 0; c < per_p; ++c) {
            h_chunk_start[(size_t)j * per_p + c] = (uint32_t)chunks;
            h_flat_base[(size_t)j * per_p + c] = flat;
            chunks += per_cfg;
            flat += items * R;
            if (chunks >= 0xfff00000ull) return SAILOR_E_RANGE;
        }
    }
    h_chunk_start[n_config] = (uint32_t)chunks;
    const size_t smem = plan_smem_bytes(ctx->hdr.static_bytes, p_max, ctx->hdr.T, ctx->hdr.Z, (uint32_t)n_config);
    if (smem > 200 * 1024) return SAILOR_E_RANGE;

    DeviceGuard guard(ctx->device);
    NoAllocScratch* sc = nullptr;
    rc = noalloc_scratch(ctx, &sc);
    if (rc) return rc;
    // the host arrays are reused by the next call on this thread: once a copy from them is enqueued, no path
    // leaves this function without waiting for the stream
    cudaError_t ce = cudaMemcpyAsync(sc->cfg_chunk_start, h_chunk_start, (n_config + 1) * sizeof(uint32_t),
                                     cudaMemcpyHostToDevice, ctx->stream);
    if (ce == cudaSuccess)
        ce = cudaMemcpyAsync(sc->cfg_flat_base, h_flat_base, n_config * sizeof(uint64_t), cudaMemcpyHostToDevice, ctx->stream);
    if (ce == cudaSuccess) ce = cudaMemsetAsync(&sc->ctrl, 0, sizeof(Ctrl), ctx->stream);      // also the error word
    if (ce == cudaSuccess) ce = cudaMemsetAsync(&sc->out.ctrl, 0, sizeof(Ctrl), ctx->stream);  // read back even if nothing runs

    uint32_t launches = 0;
    if (ce == cudaSuccess) ce = cudaEventRecord(ctx->ev0, ctx->stream);
    const bool two_pass = o->budget_factor_over_cheapest > 0.0;
    rc = SAILOR_OK;
    if (ce == cudaSuccess && total > 0) {
        if (two_pass)
            rc = enqueue_pass_noalloc(ctx, sc, d, (uint32_t)n_config, p_max, smem, 0, (uint32_t)chunks, total,
                                      SAILOR_OBJ_MIN_COST, 0.0, false, 0.0, o->flags, 1,
                                      o->budget_factor_over_cheapest, &launches);
        if (rc == SAILOR_OK)
            rc = enqueue_pass_noalloc(ctx, sc, d, (uint32_t)n_config, p_max, smem, 0, (uint32_t)chunks, total, o->kind,
                                      o->budget_usd_per_iter, two_pass, o->min_iters_per_s, o->flags, k, 0.0, &launches);
    }
    if (ce == cudaSuccess && rc == SAILOR_OK) ce = cudaEventRecord(ctx->ev1, ctx->stream);
    if (ce == cudaSuccess && rc == SAILOR_OK)
        ce = cudaMemcpyAsync(ctx->h_out, &sc->out, offsetof(PlanOut, results) + sizeof(sailor_result) * k, cudaMemcpyDeviceToHost, ctx->stream);
    if (ce == cudaSuccess && rc == SAILOR_OK && stats) ce = cudaEventRecord(ctx->ev2, ctx->stream);
    {
        const cudaError_t se = stream_sync(ctx);               // on every path: the copies above read this thread's arrays
        if (ce == cudaSuccess) ce = se;
    }
    if (ce != cudaSuccess) { ctx->last_cuda = (int)ce; return SAILOR_E_CUDA; }
    if (rc) return rc;
    const Ctrl& cr = ctx->h_out->ctrl;
    if (cr.error) return SAILOR_E_DEVICE;
    // overlapping calls race on the shared array (documented): whatever they left, never copy past k records
    if (cr.n_found > k) return SAILOR_E_DEVICE;
    *n_found = cr.n_found;
    memcpy(topk, ctx->h_out->results, sizeof(sailor_result) * cr.n_found);
    if (stats) {
        stats->n_total = cr.stats[0];
        stats->n_invalid = cr.stats[1];
        stats->n_oom = cr.stats[2];
        stats->n_over_avail = cr.stats[3];
        stats->n_over_constraint = cr.stats[4];
        stats->n_feasible = cr.stats[5];
        stats->n_pruned_tp = cr.stats[6];
        stats->n_skipped = 0;
        stats->n_configs = stats->n_configs_evaluated = (uint32_t)n_config;
        stats->budget_used = two_pass ? cr.budget : o->budget_usd_per_iter;
        double mc;
        memcpy(&mc, &cr.min_cost_bits, sizeof(mc));
        stats->min_feasible_cost = cr.stats[5] ? mc : 0.0;
        float ms = 0.f;
        CU(ctx, cudaEventElapsedTime(&ms, ctx->ev0, ctx->ev1));
        stats->kernel_ms = ms;
        stats->n_launches = launches;
        stats->d2h_ms = 0.f;
        CU(ctx, cudaEventElapsedTime(&stats->d2h_ms, ctx->ev1, ctx->ev2));
        if (ctx->h2d_fresh) {
            CU(ctx, cudaEventElapsedTime(&ctx->h2d_ms, ctx->evh0, ctx->evh1));
            ctx->h2d_fresh = false;
        }
        stats->h2d_ms = ctx->h2d_ms;
    }
    return SAILOR_OK;
}

// ---- per-stage GPU types by dynamic programming ---------------------------------------------------

namespace {

// A layout as the host lays it down (see DpLayout), its positions' rank tables and its live rows.
struct LayoutInfo {
    DpLayout l;
    std::vector<uint32_t> w;           // rank tables, position after position
    std::vector<uint32_t> live;        // [P][dp_live_words(nz)]
    uint64_t total_live = 0;           // live vectors of all stages (a byte of successors per type each)
    uint32_t max_live = 0;
    int batch = -1;                    // the last batch it was put into, and its place there
    uint32_t place = 0;
};

// The layout of pipelines of P stages of `need` GPUs each over the zones of `order`, with the types of `usable`.
// Returns SAILOR_E_RANGE when a position has more than 2^31 vectors; a stage without live vectors leaves max_live at 0.
int build_layout(const sailor_ctx* ctx, uint32_t P, uint64_t need, const sailor_zone_order& order, uint32_t usable,
                 std::vector<uint64_t>& W, LayoutInfo& info) {
    const uint32_t T = ctx->hdr.T, w = P + 1;
    DpLayout& l = info.l;
    memset(&l, 0, sizeof(l));
    memset(l.first_later, DP_NONE, sizeof(l.first_later));
    l.P = P;
    uint64_t lo = 0, mx = 0;               // stages before a position: at least, at most
    uint64_t lo_of[SAILOR_Z_MAX], mx_of[SAILOR_Z_MAX], n_vec = 0;
    bool uncounted_of[SAILOR_Z_MAX], hosts[SAILOR_Z_MAX];
    W.resize((size_t)(T + 1) * w);         // (scratch)
    info.w.reserve((size_t)order.n * (T + 1) * w);
    for (uint32_t zp = 0; zp < order.n && lo < P; ++zp) {
        l.nz = zp + 1;
        l.zone[zp] = order.zone[zp];
        uint32_t types[SAILOR_T_MAX], m = 0;
        uint64_t least = ~0ull, all = 0;
        uncounted_of[zp] = hosts[zp] = false;
        for (uint32_t g = 0; g < T; ++g) {
            if (!((usable >> g) & 1u)) continue;
            const uint64_t cap = ctx->h_avail[order.zone[zp] * T + g] / need;
            l.cap[zp][g] = (uint8_t)(cap > 255 ? 255 : cap);
            least = cap < least ? cap : least;
            all += cap;
            hosts[zp] = hosts[zp] || cap > 0;
            if (cap >= P) uncounted_of[zp] = true;
            else if (cap > 0) { types[m++] = g; l.counted[zp] |= (uint8_t)(1u << g); }
        }
        l.n_counted[zp] = (uint8_t)m;
        lo_of[zp] = lo;
        mx_of[zp] = mx;
        const uint32_t most = P - (uint32_t)lo;              // largest sum a stage here can have behind it
        l.sum_max[zp] = most;
        // W[j][s]: vectors of the counted types from the j-th on, within the caps, that add up to at most s
        for (uint32_t s = 0; s < w; ++s) W[(size_t)m * w + s] = 1;
        for (uint32_t j = m; j-- > 0;) {
            const uint64_t cj = l.cap[zp][types[j]];
            const uint64_t* below = &W[(size_t)(j + 1) * w];
            uint64_t* row = &W[(size_t)j * w];
            // exact counts N[j][s] = sum over x <= cj of N[j + 1][s - x] = W[j + 1][s] - W[j + 1][s - cj - 1]
            uint64_t run = 0;
            for (uint32_t s = 0; s < w; ++s) {
                run += below[s] - (s > cj ? below[s - cj - 1] : 0);
                row[s] = run < (1ull << 40) ? run : (1ull << 40);        // (beyond the limit below: only kept from running over)
            }
        }
        if (W[most] > (1ull << 31)) return SAILOR_E_RANGE;
        l.w_off[zp] = (uint32_t)info.w.size();
        info.w.resize(info.w.size() + (size_t)(m + 1) * w);
        uint32_t* out = info.w.data() + l.w_off[zp];
        for (size_t x = 0; x < (size_t)(m + 1) * w; ++x) out[x] = (uint32_t)(W[x] < 0xffffffffull ? W[x] : 0xffffffffull);
        l.vec_base[zp] = (uint32_t)n_vec;
        for (uint32_t j = 0; j < m; ++j)
            l.first_vec[zp][types[j]] = (uint32_t)(n_vec + W[0] + (P >= 1 ? W[(size_t)(j + 1) * w + 1] - W[(size_t)(j + 1) * w] : 0));
        for (uint32_t g = 0; g < T; ++g)
            if (l.cap[zp][g] && !((l.counted[zp] >> g) & 1u)) l.first_vec[zp][g] = (uint32_t)n_vec;
        n_vec += W[most];
        if (n_vec > (1ull << 31)) return SAILOR_E_RANGE;
        lo += least == ~0ull ? P : least;
        mx = uncounted_of[zp] ? (uint64_t)1 << 32 : mx + all;
    }
    l.vec_base[l.nz] = (uint32_t)n_vec;
    for (uint32_t zp = 0; zp < l.nz; ++zp)
        for (uint32_t g = 0; g < T; ++g)
            for (uint32_t q = zp + 1; q < l.nz; ++q)
                if (l.cap[q][g] >= 1) { l.first_later[zp][g] = (uint8_t)q; break; }
    const uint32_t words = dp_live_words(l.nz);
    info.live.assign((size_t)P * words, 0);
    for (uint32_t i = 0; i < P; ++i) {
        uint32_t* row = &info.live[(size_t)i * words];
        row[1] = (uint32_t)info.total_live;
        row[2] = (uint32_t)(info.total_live >> 32);
        uint64_t slots = 0;
        for (uint32_t zp = 0; zp < l.nz; ++zp) {
            const uint32_t* W0 = &info.w[l.w_off[zp]];
            uint64_t first = 0, count = 0;
            if (hosts[zp] && i + 1 > lo_of[zp]) {
                const uint64_t top = i + 1 - lo_of[zp];
                uint64_t bottom = uncounted_of[zp] ? 0 : 1;
                if (!uncounted_of[zp] && i + 1 > mx_of[zp] && i + 1 - mx_of[zp] > bottom) bottom = i + 1 - mx_of[zp];
                if (bottom <= top) {
                    first = bottom ? W0[bottom - 1] : 0;
                    count = W0[top] - first;
                }
            }
            row[3 + 2 * zp] = (uint32_t)(l.vec_base[zp] + first);
            row[4 + 2 * zp] = (uint32_t)slots;
            slots += count;
        }
        row[0] = (uint32_t)slots;
        info.total_live += slots;
        if (slots == 0 || (slots + 1) * ctx->hdr.T >= 0xffffffffull) {
            const bool none = slots == 0;
            info.max_live = 0;
            return none ? SAILOR_OK : SAILOR_E_RANGE;
        }
        info.max_live = std::max(info.max_live, (uint32_t)slots);
    }
    return SAILOR_OK;
}

// The stretches of stages of one make-up in a pipeline, with what a stage of each needs of the memory: bytes without a
// microbatch in flight, bytes per microbatch.  The same for every data-parallel degree.
struct Stretches {
    uint32_t n = 0, first[4], last[4];
    uint64_t fixed[4], kept[4];
    Stretches(const TabHdr& h, const TabView& v, const Config& k) {
        const uint32_t P = k.P, base = h.n_blocks / P, extra = h.n_blocks % P;
        for (uint32_t i = 0; i < P;) {
            uint32_t end = P;
            if (i == 0 && h.has_embed) end = 1;
            else {
                if (i < extra && extra < end) end = extra;
                if (h.has_head && i < P - 1 && P - 1 < end) end = P - 1;
            }
            const bool e = (i == 0) && h.has_embed, hd = (i == P - 1) && h.has_head;
            const uint32_t nb = base + (i < extra ? 1u : 0u);
            first[n] = i;
            last[n] = end - 1;
            fixed[n] = stage_memory(v, k.tpi, k.mi, k.rc, nb, e, hd, 0).mem;
            kept[n] = stage_memory(v, k.tpi, k.mi, k.rc, nb, e, hd, 1).mem - fixed[n];
            ++n;
            i = end;
        }
    }
};

// The GPU types that fit the memory of some stage of a configuration; 0 when a stage fits none.  Inside a stretch the first
// stage keeps the most microbatches and the last the fewest.
uint32_t usable_types(const TabHdr& h, const Stretches& st, const Config& k, uint64_t n_b) {
    const uint32_t tp = h.tp_values[k.tpi];
    auto fits = [&](uint32_t q, uint32_t i) {
        const uint64_t inflight = (uint64_t)(k.P - i) < n_b ? (uint64_t)(k.P - i) : n_b, mem = st.fixed[q] + inflight * st.kept[q];
        uint32_t mask = 0;
        for (uint32_t g = 0; g < h.T; ++g)
            if (mem + h.reserved[g] <= h.capacity[g] && tp <= h.gpn[g]) mask |= 1u << g;
        return mask;
    };
    uint32_t all = 0;
    for (uint32_t q = 0; q < st.n; ++q) {
        if (!fits(q, st.first[q])) return 0;
        all |= fits(q, st.last[q]);
    }
    return all;
}

// SAILOR_DP_FLAG_INDEX_DENSE: the size the tables of a problem would have in mixed radix over all its scarce types.
int dense_fits(const sailor_ctx* ctx, uint32_t P, uint64_t need, const sailor_zone_order& order, uint64_t workspace_bytes) {
    const uint32_t T = ctx->hdr.T;
    uint64_t entries = 0;
    for (uint32_t zp = 0; zp < order.n; ++zp) {
        uint64_t box = T;
        for (uint32_t g = 0; g < T; ++g) {
            const uint64_t cap = ctx->h_avail[order.zone[zp] * T + g] / need;
            if (cap >= 1 && cap < P) box *= cap + 1;
            if (box > (1ull << 31)) return SAILOR_E_RANGE;
        }
        entries += box;
    }
    return entries > (1ull << 31) || entries * (2 * sizeof(DpVal) + P) > workspace_bytes ? SAILOR_E_RANGE : SAILOR_OK;
}

}  // namespace

// The recursion steered by the budget (Sec. 4.2.3): a warp per problem and type of its first stage, or of its first two, depth first.
static int plan_dp_budget_impl(sailor_ctx* ctx, const SpaceDesc& d, const sailor_zone_order* orders, uint32_t n_orders,
                               const sailor_objective* o, uint64_t workspace_bytes, uint32_t k, sailor_dp_result* topk,
                               uint32_t* n_found, sailor_dp_stats* stats) {
    const TabHdr& h = ctx->hdr;
    const uint32_t T = h.T;
    const uint64_t n_config = (uint64_t)d.n_p * d.n_mbs * d.n_tp * d.n_rc * d.n_d, n_problems = n_config * n_orders;
    uint32_t p_max = 0;
    for (uint32_t j = 0; j < d.n_p; ++j) p_max = d.p_values[j] > p_max ? d.p_values[j] : p_max;
    DeviceGuard guard(ctx->device);
    DpTabLayout lay;
    lay.p_max = p_max; lay.T = T; lay.R = h.R;
    const size_t tab_bytes = (size_t)n_config * lay.stride() * sizeof(double);
    const size_t others = padded(tab_bytes) + padded(n_problems * sizeof(DpResult)) + padded(n_problems * sizeof(DpProblem)) +
                          padded(n_problems * sizeof(double)) + padded(40) + std::max<size_t>(padded(n_orders * sizeof(sailor_zone_order)), 4096);
    DpBudgetParams bp;
    memset(&bp, 0, sizeof(bp));
    bp.T = T; bp.p_max = p_max;
    const uint64_t per_length = n_problems / d.n_p, per_first = per_length * T;
    // A length has a walk per pair of first types where that is worth it and the workspace holds them all.
    uint8_t order[SAILOR_NP_MAX];
    for (uint32_t j = 0; j < d.n_p; ++j) order[j] = (uint8_t)j;
    std::sort(order, order + d.n_p, [&](uint8_t a, uint8_t b) { return d.p_values[a] != d.p_values[b] ? d.p_values[a] > d.p_values[b] : a < b; });
    uint64_t extra = 0;
    for (uint32_t x = 0; x < d.n_p; ++x) {
        uint64_t calls = 1;                                  // that a walk from one type of stage 0 can make without charging again
        for (uint32_t i = 1; i < d.p_values[order[x]] && calls < (1u << 20); ++i) calls = calls * T + 1;
        if (T < 2 || calls < DPB_SPLIT_CALLS || extra + per_first * (T - 1) > DPB_SPLIT_WORTH * calls) continue;
        extra += per_first * (T - 1);
        bp.split |= 1u << order[x];
    }
    uint64_t n_walks = n_problems * T + extra;
    if (n_walks > DPB_SPLIT_WALKS || others + padded(n_walks * sizeof(DpbRoot)) > workspace_bytes) {
        bp.split = 0;
        n_walks = n_problems * T;
    }
    if (!bp.split)
        for (uint32_t j = 0; j < d.n_p; ++j) order[j] = (uint8_t)j;
    const size_t total = others + padded(n_walks * sizeof(DpbRoot));
    if (total > workspace_bytes) return SAILOR_E_RANGE;
    bp.n_walks = (uint32_t)n_walks;
    bp.per_length = (uint32_t)per_length;
    for (uint32_t x = 1; x < d.n_p; ++x)
        bp.first[order[x]] = bp.first[order[x - 1]] + (uint32_t)per_first * bp.walks_of_type(order[x - 1]);
    {
        const int rc_mem = device_grow(ctx, &ctx->d_dp, &ctx->dp_bytes, total);
        if (rc_mem) return rc_mem;
    }
    Bump bump{ctx->d_dp};
    double* d_tabs = bump.take<double>(tab_bytes / sizeof(double));
    DpResult* d_results = bump.take<DpResult>(n_problems);
    DpProblem* d_problems = bump.take<DpProblem>(n_problems);
    DpbRoot* d_roots = bump.take<DpbRoot>(n_walks);
    double* d_value = bump.take<double>(n_problems);
    unsigned long long* d_counters = bump.take<unsigned long long>(5);
    sailor_zone_order* d_orders = bump.take<sailor_zone_order>(n_orders);
    DpOut* d_out = nullptr;
    CU(ctx, cudaHostGetDevicePointer(reinterpret_cast<void**>(&d_out), &ctx->host->dp, 0));

    uint32_t launches = 0;
    {
        const int rc_up = upload_availability(ctx);
        if (rc_up) return rc_up;
    }
    CU(ctx, cudaMemcpyAsync(d_orders, orders, n_orders * sizeof(sailor_zone_order), cudaMemcpyHostToDevice, ctx->stream));
    {
        const uint32_t grid = (uint32_t)(n_config < 4096 ? n_config : 4096);
        dp_tables_kernel<<<grid, DP_THREADS, 0, ctx->stream>>>(ctx->d_blob, d, (uint32_t)n_config, n_orders, lay, nullptr, d_tabs, d_value, &d_out->span);
        CU(ctx, cudaGetLastError());
        ++launches;
    }
    dp_budget_problems_kernel<<<(uint32_t)((n_problems + 127) / 128), 128, 0, ctx->stream>>>(
        ctx->d_blob, ctx->d_avail, d, d_orders, n_orders, (uint32_t)n_problems, d_problems, d_counters);
    CU(ctx, cudaGetLastError());
    ++launches;
    bp.blob = ctx->d_blob; bp.avail = ctx->d_avail; bp.sp = d; bp.problems = d_problems; bp.tabs = d_tabs;
    bp.value = d_value; bp.results = d_results; bp.roots = d_roots; bp.counters = d_counters; bp.lay = lay;
    bp.n_problems = (uint32_t)n_problems;
    bp.limit = o->budget_usd_per_iter;
    bp.node_limit = 1ull << 24;
    auto launch = [&](auto kernel, uint32_t warps) {
        kernel<<<(bp.n_walks + warps - 1) / warps, 32 * warps, dpb_smem(p_max, warps), ctx->stream>>>(bp);
    };
    if (bp.split) launch(dp_budget_kernel<true>, DPB_WARPS<true>);
    else launch(dp_budget_kernel<false>, DPB_WARPS<false>);
    CU(ctx, cudaGetLastError());
    dp_budget_finish_kernel<<<(uint32_t)((n_problems + DP_FINISH_WARPS - 1) / DP_FINISH_WARPS), DP_FINISH_THREADS, 0, ctx->stream>>>(bp);
    CU(ctx, cudaGetLastError());
    launches += 2;
    DpSelectParams sel;
    memset(&sel, 0, sizeof(sel));
    sel.value = d_value; sel.results = d_results; sel.out = d_out; sel.counters = d_counters;
    sel.sp = d; sel.n_problems = (uint32_t)n_problems; sel.n_orders = n_orders; sel.k = k;
    sel.budget = o->budget_usd_per_iter; sel.min_rate = o->min_iters_per_s;
    dp_select_kernel<<<1, DP_SELECT_THREADS, 0, ctx->stream>>>(sel);
    CU(ctx, cudaGetLastError());
    ++launches;
    CU(ctx, stream_sync(ctx));
    const unsigned long long* counters = ctx->host->dp.counters;
    if (counters[1] > k) return SAILOR_E_DEVICE;
    *n_found = (uint32_t)counters[1];
    memcpy(topk, ctx->host->dp.results, sizeof(sailor_dp_result) * counters[1]);
    if (stats) {
        stats->n_problems = n_problems;
        stats->n_solved = counters[0];
        stats->n_over_constraint = counters[2];
        stats->n_states = counters[4];
        stats->workspace_used = total;
        stats->kernel_ms = span_ms(ctx->host->dp.span);
        stats->n_launches = launches;
        stats->n_batches = 1;
        stats->n_unfinished = (uint32_t)counters[3];
    }
    return SAILOR_OK;
}

static int plan_dp_impl(sailor_ctx* ctx, const sailor_space* s, const sailor_zone_order* orders,
                        uint32_t n_orders, const sailor_objective* o, uint64_t workspace_bytes, uint32_t k,
                        sailor_dp_result* topk, uint32_t* n_found, sailor_dp_stats* stats) {
    if (!ctx || !s || !orders || !o || !topk || !n_found || k == 0 || n_orders == 0) return SAILOR_E_ARG;
    if (k > SAILOR_K_MAX) return SAILOR_E_RANGE;
    // the recursion minimises iteration time; a constraint is checked on the plan it returns per problem
    constexpr uint32_t dp_flags = SAILOR_DP_FLAG_INDEX_DENSE | SAILOR_DP_FLAG_INDEX_COMPACT | SAILOR_DP_FLAG_ENUM_BY_TYPE |
                                  SAILOR_DP_FLAG_ENUM_BY_ENTRY | SAILOR_DP_FLAG_BUDGET_LOOP;
    if (o->kind != SAILOR_OBJ_MAX_THROUGHPUT || (o->flags & ~dp_flags) != 0 ||
        ((o->flags & SAILOR_DP_FLAG_INDEX_DENSE) && (o->flags & SAILOR_DP_FLAG_INDEX_COMPACT)) ||
        ((o->flags & SAILOR_DP_FLAG_ENUM_BY_TYPE) && (o->flags & SAILOR_DP_FLAG_ENUM_BY_ENTRY)) ||
        o->budget_factor_over_cheapest > 0.0 ||
        std::isnan(o->budget_usd_per_iter) || std::isnan(o->min_iters_per_s) || std::isnan(o->budget_factor_over_cheapest))
        return SAILOR_E_ARG;
    int rc = check_space(ctx, s);
    if (rc) return rc;
    const TabHdr& h = ctx->hdr;
    const uint32_t T = h.T, Z = h.Z;
    for (uint32_t q = 0; q < n_orders; ++q) {
        if (orders[q].n < 1 || orders[q].n > Z) return SAILOR_E_ARG;
        uint32_t seen = 0;
        for (uint32_t j = 0; j < orders[q].n; ++j) {
            if (orders[q].zone[j] >= Z || ((seen >> orders[q].zone[j]) & 1u)) return SAILOR_E_ARG;
            seen |= 1u << orders[q].zone[j];
        }
    }
    const SpaceDesc d = to_desc(s);
    const uint64_t n_config = (uint64_t)d.n_p * d.n_mbs * d.n_tp * d.n_rc * d.n_d;
    if (n_config * n_orders > (1u << 22)) return SAILOR_E_RANGE;
    if (workspace_bytes == 0) workspace_bytes = 8ull << 30;
    uint32_t p_max = 0;
    for (uint32_t j = 0; j < d.n_p; ++j) p_max = d.p_values[j] > p_max ? d.p_values[j] : p_max;
    if (o->flags & SAILOR_DP_FLAG_BUDGET_LOOP) {
        if (!(o->budget_usd_per_iter > 0.0)) return SAILOR_E_ARG;
        if (p_max > DP_BUDGET_P_MAX) return SAILOR_E_RANGE;
        return plan_dp_budget_impl(ctx, d, orders, n_orders, o, workspace_bytes, k, topk, n_found, stats);
    }

    // problems that can have a plan, and the layouts they share
    const uint64_t n_problems = n_config * n_orders;
    TabView hv;
    hv.bind(ctx->h_static.data(), ctx->h_static.data());
    std::vector<LayoutInfo> layouts;
    std::map<std::pair<uint64_t, uint64_t>, uint32_t> layout_of;
    struct Problem { uint32_t config, index, layout, place; };   // place: of the layout among its batch's
    std::vector<Problem> by_depth[SAILOR_P_MAX + 1];         // deepest first, so that a stage's launch covers a prefix
    std::vector<uint8_t> wanted(n_config, 0);                // configurations whose per-configuration tables are needed
    uint64_t n_states = 0;
    std::unique_ptr<Stretches> stretches;
    uint64_t stretches_end = 0;
    std::vector<uint64_t> scratch;
    layouts.reserve(512);
    for (uint64_t c = 0; c < n_config; ++c) {
        const Config cf = config_of(d, (uint32_t)c);
        const uint32_t tp = h.tp_values[cf.tpi];
        const uint64_t dm = (uint64_t)cf.D * h.mbs_values[cf.mi];
        const uint64_t need = (uint64_t)cf.D * tp;
        if (h.gbs % dm != 0 || h.heads % tp != 0) continue;  // no valid plan
        if (o->flags & SAILOR_DP_FLAG_INDEX_DENSE)
            for (uint32_t q = 0; q < n_orders; ++q)
                if (dense_fits(ctx, cf.P, need, orders[q], workspace_bytes) != SAILOR_OK) return SAILOR_E_RANGE;
        if (!stretches || c >= stretches_end) {              // the degree varies fastest
            stretches.reset(new Stretches(h, hv, cf));
            stretches_end = c - c % d.n_d + d.n_d;
        }
        const uint32_t usable = usable_types(h, *stretches, cf, h.gbs / dm);
        if (!usable) continue;                               // some stage fits no type
        for (uint32_t q = 0; q < n_orders; ++q) {
            const std::pair<uint64_t, uint64_t> key((uint64_t)q << 8 | cf.P, need << SAILOR_T_MAX | usable);
            const auto seen = layout_of.emplace(key, (uint32_t)layouts.size());
            if (seen.second) {
                layouts.emplace_back();
                const int rc_lay = build_layout(ctx, cf.P, need, orders[q], usable, scratch, layouts.back());
                if (rc_lay) return rc_lay;
            }
            const LayoutInfo& info = layouts[seen.first->second];
            if (info.max_live == 0) continue;                // some stage has nowhere to go
            by_depth[cf.P].push_back({(uint32_t)c, (uint32_t)(c * n_orders + q), seen.first->second, 0});
            wanted[c] = 1;
            n_states += info.total_live * T;
        }
    }
    std::vector<Problem> todo;
    for (uint32_t P = SAILOR_P_MAX; P > 0; --P) todo.insert(todo.end(), by_depth[P].begin(), by_depth[P].end());

    // cut into batches that fit the workspace: per problem two level buffers and its successors, per layout its moves.  What
    // bounds a problem alone is its own tables, (64 + stages) bytes a state at most; its moves may then come on top.
    const uint32_t TM = T <= 4 ? 4 : SAILOR_T_MAX;
    struct Batch {
        size_t first, count;
        uint64_t val_entries, succ_bytes, nxt_rows;
        std::vector<std::pair<uint32_t, uint32_t>> layouts;  // layout, its first row of moves in this batch
    };
    std::vector<Batch> batches;
    size_t largest = 0;
    auto pad8 = [](uint64_t x) { return (x + 7) / 8 * 8; };
    auto pad64 = [](uint64_t x) { return (x + 63) / 64 * 64; };
    for (size_t j = 0; j < todo.size();) {
        Batch b = {j, 0, 0, 0, 0, {}};
        uint64_t bytes = 0;
        for (; j < todo.size(); ++j) {
            LayoutInfo& info = layouts[todo[j].layout];
            const uint64_t val = pad8((uint64_t)info.max_live * T), succ = pad64(info.total_live * T);
            const uint64_t rows = info.batch == (int)batches.size() ? 0 : info.l.vec_base[info.l.nz];
            const uint64_t tables = val * 2 * sizeof(DpVal) + succ, moves = rows * TM * 4;
            if (b.count && (bytes + tables + moves > workspace_bytes || b.nxt_rows + rows >= (1ull << 32))) break;
            if (tables > workspace_bytes) return SAILOR_E_RANGE;     // one problem alone does not fit
            if (rows) {
                info.batch = (int)batches.size();
                info.place = (uint32_t)b.layouts.size();
                b.layouts.emplace_back(todo[j].layout, (uint32_t)b.nxt_rows);
                b.nxt_rows += rows;
            }
            todo[j].place = info.place;
            bytes += tables + moves;
            b.val_entries += val;
            b.succ_bytes += succ;
            ++b.count;
        }
        largest = std::max(largest, 2 * padded(b.val_entries * sizeof(DpVal)) + padded(b.succ_bytes) + padded(b.nxt_rows * TM * 4));
        batches.push_back(std::move(b));
    }

    DeviceGuard guard(ctx->device);
    {
        const int rc_up = upload_availability(ctx);
        if (rc_up) return rc_up;
    }
    DpTabLayout lay;
    lay.p_max = p_max; lay.T = T; lay.R = h.R;
    const size_t tab_bytes = (size_t)n_config * lay.stride() * sizeof(double);
    DpOut* d_out = nullptr;
    CU(ctx, cudaHostGetDevicePointer(reinterpret_cast<void**>(&d_out), &ctx->host->dp, 0));
    const size_t total = padded(tab_bytes) + padded(n_problems * sizeof(DpResult)) + padded(n_problems * sizeof(double)) + largest;
    {
        const int rc_mem = device_grow(ctx, &ctx->d_dp, &ctx->dp_bytes, total);
        if (rc_mem) return rc_mem;
    }
    Bump bump{ctx->d_dp};
    double* d_tabs = bump.take<double>(tab_bytes / sizeof(double));
    DpResult* d_results = bump.take<DpResult>(n_problems);
    double* d_value = bump.take<double>(n_problems);
    DpLevelParams lp;
    memset(&lp, 0, sizeof(lp));
    const size_t arena = bump.at;                            // the batches take turns in what follows
    lp.tabs = d_tabs; lp.lay = lay; lp.T = T;

    uint32_t launches = 0;
    std::vector<unsigned char> up;                           // what a batch uploads, in one copy
    auto add = [&](const void* p, size_t bytes) {
        const size_t off = padded(up.size());
        up.resize(off + bytes);
        if (bytes) memcpy(up.data() + off, p, bytes);
        return off;
    };
    const size_t off_wanted = add(wanted.data(), wanted.size());         // with the first batch
    for (size_t bi = 0; bi < std::max<size_t>(batches.size(), 1); ++bi) {
        const Batch* b = batches.empty() ? nullptr : &batches[bi];       // none: no problem has a plan
        std::vector<DpLayout> lays;
        std::vector<DpJob> jobs;
        std::vector<uint32_t> lay_blk(1, 0), wtab, live, prefix;
        std::vector<size_t> dist_off;
        uint32_t n_big = 0;
        if (b) {
            for (const auto& used : b->layouts) {            // layouts, with offsets into the joint tables
                const LayoutInfo& info = layouts[used.first];
                lays.push_back(info.l);
                lays.back().nxt_off = used.second;
                for (uint32_t zp = 0; zp < info.l.nz; ++zp) lays.back().w_off[zp] += (uint32_t)wtab.size();
                lays.back().live_off = (uint32_t)live.size();
                wtab.insert(wtab.end(), info.w.begin(), info.w.end());
                live.insert(live.end(), info.live.begin(), info.live.end());
                lay_blk.push_back(lay_blk.back() + (info.l.vec_base[info.l.nz] + DP_THREADS - 1) / DP_THREADS);
            }
            // jobs: those that go stage by stage first (deepest first), then the small ones
            jobs.resize(b->count);
            for (size_t j = 0; j < b->count; ++j) n_big += layouts[todo[b->first + j].layout].max_live > DP_SMALL ? 1u : 0u;
            uint32_t at_big = 0, at_small = n_big;
            uint64_t val_off = 0, succ_off = 0;
            for (size_t j = 0; j < b->count; ++j) {
                const Problem& pr = todo[b->first + j];
                const LayoutInfo& info = layouts[pr.layout];
                DpJob& job = jobs[info.max_live > DP_SMALL ? at_big++ : at_small++];
                job.val_off = val_off;
                job.succ_off = succ_off;
                job.config = pr.config; job.index = pr.index; job.layout = pr.place; job.P = info.l.P;
                job.slots = info.max_live;
                job._pad = 0;
                val_off += pad8((uint64_t)info.max_live * T);
                succ_off += pad64(info.total_live * T);
            }
            for (uint32_t dist = 0; n_big && dist < jobs[0].P; ++dist) {     // per distance from the last stage: blocks before each job
                dist_off.push_back(prefix.size());
                uint32_t blocks = 0;
                for (uint32_t j = 0; j < n_big && jobs[j].P > dist; ++j) {
                    prefix.push_back(blocks);
                    const DpLayout& l = lays[jobs[j].layout];
                    blocks += (live[l.live_off + (size_t)(jobs[j].P - 1 - dist) * dp_live_words(l.nz)] + DP_THREADS - 1) / DP_THREADS;
                }
                prefix.push_back(blocks);
            }
            dist_off.push_back(prefix.size());
        }
        const size_t off_lay = add(lays.data(), lays.size() * sizeof(DpLayout)), off_blk = add(lay_blk.data(), lay_blk.size() * 4),
                     off_w = add(wtab.data(), wtab.size() * 4), off_live = add(live.data(), live.size() * 4),
                     off_jobs = add(jobs.data(), jobs.size() * sizeof(DpJob)), off_prefix = add(prefix.data(), prefix.size() * 4);
        {
            const int rc_mem = device_grow(ctx, &ctx->d_dp_up, &ctx->dp_up_bytes, padded(up.size()));
            if (rc_mem) return rc_mem;
        }
        CU(ctx, cudaMemcpyAsync(ctx->d_dp_up, up.data(), up.size(), cudaMemcpyHostToDevice, ctx->stream));   // returns when `up` has been read
        if (bi == 0) {
            dp_tables_kernel<<<(uint32_t)std::min<uint64_t>(n_config, 4096), DP_THREADS, 0, ctx->stream>>>(
                ctx->d_blob, d, (uint32_t)n_config, n_orders, lay, ctx->d_dp_up + off_wanted, d_tabs, d_value, &d_out->span);
            CU(ctx, cudaGetLastError());
            ++launches;
        }
        if (!b) break;
        bump.at = arena;
        uint32_t* d_nxt = bump.take<uint32_t>(b->nxt_rows * TM);
        lp.nxt = d_nxt;
        lp.val[0] = bump.take<DpVal>(b->val_entries);
        lp.val[1] = bump.take<DpVal>(b->val_entries);
        lp.succ = bump.take<uint8_t>(b->succ_bytes);
        lp.layouts = reinterpret_cast<const DpLayout*>(ctx->d_dp_up + off_lay);
        lp.live = reinterpret_cast<const uint32_t*>(ctx->d_dp_up + off_live);
        lp.jobs = reinterpret_cast<const DpJob*>(ctx->d_dp_up + off_jobs);
        const uint32_t* d_prefix = reinterpret_cast<const uint32_t*>(ctx->d_dp_up + off_prefix);
        DpLayoutParams yp;
        memset(&yp, 0, sizeof(yp));
        yp.layouts = lp.layouts;
        yp.blk_prefix = reinterpret_cast<const uint32_t*>(ctx->d_dp_up + off_blk);
        yp.wtab = reinterpret_cast<const uint32_t*>(ctx->d_dp_up + off_w);
        yp.nxt = d_nxt; yp.n_layouts = (uint32_t)lays.size(); yp.T = T;
        if (TM == 4) dp_layout_kernel<4><<<lay_blk.back(), DP_THREADS, 0, ctx->stream>>>(yp);
        else dp_layout_kernel<SAILOR_T_MAX><<<lay_blk.back(), DP_THREADS, 0, ctx->stream>>>(yp);
        CU(ctx, cudaGetLastError());
        ++launches;
        // The small problems' blocks take each a problem through all its stages and mostly wait for one another: they run beside
        // the levels of the large ones, on a second stream (five zones, 48 stages: 300 us of a search's 2 315; joining in only
        // when levels have become small, as late as they hide, 1 984 instead of 1 809).
        const uint32_t n_small = (uint32_t)jobs.size() - n_big;
        const bool fork = n_small && n_big;
        auto joined = [&](cudaError_t e) {                       // nothing is left running there after a failure
            if (e != cudaSuccess && fork) cudaStreamSynchronize(ctx->out_stream);
            return e;
        };
        if (fork) {
            const int rc_side = side_stream(ctx);
            if (rc_side) return rc_side;
            CU(ctx, cudaEventRecord(ctx->ev_chunk, ctx->stream));
            CU(ctx, cudaStreamWaitEvent(ctx->out_stream, ctx->ev_chunk, 0));
        }
        if (n_small) {
            DpLevelParams sp = lp;
            sp.jobs = lp.jobs + n_big;
            cudaStream_t stream = fork ? ctx->out_stream : ctx->stream;
            if (TM == 4) dp_problem_kernel<4><<<n_small, DP_THREADS, 0, stream>>>(sp);
            else dp_problem_kernel<SAILOR_T_MAX><<<n_small, DP_THREADS, 0, stream>>>(sp);
            CU(ctx, joined(cudaGetLastError()));
            ++launches;
            if (fork) CU(ctx, joined(cudaEventRecord(ctx->ev_join, ctx->out_stream)));
        }
        for (uint32_t dist = 0; dist + 1 < dist_off.size(); ++dist) {
            lp.dist = dist;
            lp.blk_prefix = d_prefix + dist_off[dist];
            lp.n_active = (uint32_t)(dist_off[dist + 1] - dist_off[dist] - 1);
            const uint32_t n_blk = prefix[dist_off[dist + 1] - 1];
            // a level's blocks may start (and find their job and its tables) while the level before it ends
            cudaLaunchConfig_t cfg = {};
            cudaLaunchAttribute attr = {};
            attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
            attr.val.programmaticStreamSerializationAllowed = dist ? 1 : 0;
            cfg.gridDim = dim3(n_blk); cfg.blockDim = dim3(DP_THREADS); cfg.stream = ctx->stream;
            cfg.attrs = &attr; cfg.numAttrs = 1;
            CU(ctx, joined(TM == 4 ? cudaLaunchKernelEx(&cfg, dp_level_kernel<4>, (const DpLevelParams)lp)
                                   : cudaLaunchKernelEx(&cfg, dp_level_kernel<SAILOR_T_MAX>, (const DpLevelParams)lp)));
            ++launches;
        }
        if (fork) CU(ctx, joined(cudaStreamWaitEvent(ctx->stream, ctx->ev_join, 0)));
        DpFinishParams fp;
        memset(&fp, 0, sizeof(fp));
        fp.blob = ctx->d_blob; fp.avail = ctx->d_avail; fp.sp = d; fp.layouts = lp.layouts; fp.jobs = lp.jobs; fp.live = lp.live;
        fp.tabs = d_tabs; fp.val[0] = lp.val[0]; fp.val[1] = lp.val[1]; fp.succ = lp.succ; fp.nxt = d_nxt; fp.value = d_value;
        fp.results = d_results; fp.lay = lay; fp.n_jobs = (uint32_t)jobs.size(); fp.T = T; fp.TM = TM;
        dp_finish_kernel<<<(fp.n_jobs + DP_FINISH_WARPS - 1) / DP_FINISH_WARPS, DP_FINISH_THREADS, 0, ctx->stream>>>(fp);
        CU(ctx, cudaGetLastError());
        ++launches;
        up.clear();
    }
    DpSelectParams sel;
    memset(&sel, 0, sizeof(sel));
    sel.value = d_value; sel.results = d_results; sel.out = d_out;
    sel.sp = d; sel.n_problems = (uint32_t)n_problems; sel.n_orders = n_orders; sel.k = k;
    sel.budget = o->budget_usd_per_iter; sel.min_rate = o->min_iters_per_s;
    dp_select_kernel<<<1, DP_SELECT_THREADS, 0, ctx->stream>>>(sel);
    CU(ctx, cudaGetLastError());
    ++launches;
    CU(ctx, stream_sync(ctx));
    const unsigned long long* counters = ctx->host->dp.counters;
    if (counters[1] > k) return SAILOR_E_DEVICE;               // cannot happen; never copy past the caller's k records
    *n_found = (uint32_t)counters[1];
    memcpy(topk, ctx->host->dp.results, sizeof(sailor_dp_result) * counters[1]);
    if (stats) {
        stats->n_problems = n_problems;
        stats->n_solved = counters[0];
        stats->n_over_constraint = counters[2];
        stats->n_states = n_states;
        stats->workspace_used = largest;
        stats->kernel_ms = span_ms(ctx->host->dp.span);
        stats->n_launches = launches;
        stats->n_batches = (uint32_t)std::max<size_t>(batches.size(), 1);
        stats->n_unfinished = 0;
    }
    return SAILOR_OK;
}

// ---- search over plans with mixed replicas -------------------------------------------------------------

namespace {

// The combinations of `units` over T types with at most SAILOR_MIX_GROUPS_MAX non-empty types, in descending
// lexicographic order, one 64-bit word each (byte g = units on type g).
void list_combinations(uint32_t T, uint32_t units, std::vector<uint64_t>& out) {
    struct Rec {
        static void go(uint32_t T, uint32_t t, uint32_t left, uint32_t nonzero, uint64_t word, std::vector<uint64_t>& out) {
            if (t + 1 == T) {                                  // the last type takes what is left
                if (nonzero + (left ? 1u : 0u) <= SAILOR_MIX_GROUPS_MAX) out.push_back(word | ((uint64_t)left << (8 * t)));
                return;
            }
            for (uint32_t u = left + 1; u-- > 0;) {            // most units first
                const uint32_t nz = nonzero + (u ? 1u : 0u);
                if (nz > SAILOR_MIX_GROUPS_MAX) continue;
                go(T, t + 1, left - u, nz, word | ((uint64_t)u << (8 * t)), out);
            }
        }
    };
    Rec::go(T, 0, units, 0, 0, out);
}

int build_mixed_tables(const sailor_ctx* ctx, const sailor_mixed_space* s, MixedTables& mt) {
    if (!ctx || !s) return SAILOR_E_ARG;
    if (s->n_p == 0 || s->n_mbs == 0 || s->n_rc == 0 || s->n_d == 0 || s->granularity == 0) return SAILOR_E_ARG;
    if (s->n_p > SAILOR_NP_MAX || s->n_mbs > SAILOR_MBS_MAX || s->n_rc > 2 || s->n_d > SAILOR_ND_MAX || s->seg_max < 1 ||
        s->seg_max > SAILOR_SEG_MAX)
        return SAILOR_E_RANGE;
    const TabHdr& h = ctx->hdr;
    for (uint32_t i = 0; i < s->n_p; ++i)
        if (s->p_values[i] < 1 || s->p_values[i] > SAILOR_MIX_P_MAX) return SAILOR_E_RANGE;
    for (uint32_t i = 0; i < s->n_mbs; ++i)
        if (s->mbs_idx[i] >= h.n_mbs) return SAILOR_E_RANGE;
    for (uint32_t i = 0; i < s->n_rc; ++i)
        if (s->rc_values[i] > 1) return SAILOR_E_RANGE;
    for (uint32_t g = 0; g < h.T; ++g)
        if (s->tp_idx_of_type[g] >= h.n_tp) return SAILOR_E_RANGE;
    MixedSpaceDesc& d = mt.desc;
    memset(&d, 0, sizeof(d));
    d.n_p = s->n_p; d.n_mbs = s->n_mbs; d.n_rc = s->n_rc; d.n_d = s->n_d; d.seg_max = s->seg_max; d.granularity = s->granularity;
    memcpy(d.p_values, s->p_values, sizeof(d.p_values));
    memcpy(d.mbs_idx, s->mbs_idx, sizeof(d.mbs_idx));
    memcpy(d.rc_values, s->rc_values, sizeof(d.rc_values));
    memcpy(d.tp_idx_of_type, s->tp_idx_of_type, sizeof(d.tp_idx_of_type));
    memcpy(d.d_values, s->d_values, sizeof(d.d_values));
    std::map<uint32_t, std::pair<uint32_t, uint32_t>> by_units;        // units -> (offset, count): degrees often share them
    for (uint32_t j = 0; j < s->n_d; ++j) {
        const uint32_t D = s->d_values[j];
        if (D < 1) return SAILOR_E_RANGE;
        const uint32_t units = mixed_units(s->granularity, D);
        if (units > SAILOR_MIX_UNITS_MAX) return SAILOR_E_RANGE;
        auto it = by_units.find(units);
        if (it == by_units.end()) {
            const uint32_t off = (uint32_t)mt.combs.size();
            list_combinations(h.T, units, mt.combs);
            it = by_units.emplace(units, std::make_pair(off, (uint32_t)mt.combs.size() - off)).first;
        }
        d.comb_off[j] = it->second.first;
        d.n_comb[j] = it->second.second;
    }
    const uint64_t n_config = (uint64_t)s->n_p * s->n_mbs * s->n_rc * s->n_d;
    if (n_config > (1u << 16)) return SAILOR_E_RANGE;
    mt.n_config = (uint32_t)n_config;
    mt.flat_base.assign(n_config + 1, 0);
    unsigned __int128 run = 0;
    for (uint32_t c = 0; c < n_config; ++c) {
        mt.flat_base[c] = (uint64_t)run;
        const MixedConfig k = mixed_config_of(d, c);
        const unsigned __int128 radix = (unsigned __int128)h.Z * d.n_comb[k.di];
        unsigned __int128 block = 1;
        for (uint32_t q = 0; q < k.nseg; ++q) {
            block *= radix;
            if (block >> 63) return SAILOR_E_RANGE;
        }
        run += block;
        if (run >> 63) return SAILOR_E_RANGE;
    }
    mt.flat_base[n_config] = (uint64_t)run;
    return SAILOR_OK;
}

bool same_mixed_space(const sailor_mixed_space& a, const sailor_mixed_space& b, uint32_t n_types) {
    if (a.n_p != b.n_p || a.n_mbs != b.n_mbs || a.n_rc != b.n_rc || a.n_d != b.n_d || a.seg_max != b.seg_max ||
        a.granularity != b.granularity)
        return false;
    return !memcmp(a.p_values, b.p_values, a.n_p) && !memcmp(a.mbs_idx, b.mbs_idx, a.n_mbs) &&
           !memcmp(a.rc_values, b.rc_values, a.n_rc) && !memcmp(a.tp_idx_of_type, b.tp_idx_of_type, n_types) &&
           !memcmp(a.d_values, b.d_values, a.n_d * sizeof(uint16_t));
}

// The device pointers of a mixed search inside the context's working memory; returns the bytes it takes.
size_t mixed_carve(const sailor_ctx* ctx, const MixedTables& mt, MixedSearchParams& mp) {
    Bump bump{ctx->d_mix};
    mp.counters = bump.take<unsigned long long>(MIXC_N);
    mp.combs = bump.take<uint64_t>(mt.combs.size());
    mp.cfg_flat_base = bump.take<uint64_t>(mt.flat_base.size());
    mp.partial = bump.take<Hit>((size_t)SAILOR_K_MAX * ctx->sm_count * 4);
    mp.queue = bump.take<uint32_t>(std::min<uint64_t>(mt.flat_base[mt.n_config], MIXED_RANGE));
    return bump.at;
}

// Working memory for a mixed space and its tables on the device.
int mixed_workspace(sailor_ctx* ctx, const MixedTables& mt) {
    MixedSearchParams mp;
    const size_t need = mixed_carve(ctx, mt, mp);
    if (need > ctx->mix_bytes) {
        ctx->mix_dirty = true;
        const int rc = device_grow(ctx, &ctx->d_mix, &ctx->mix_bytes, need);
        if (rc) return rc;
        mixed_carve(ctx, mt, mp);
    }
    CU(ctx, cudaMemcpyAsync(const_cast<uint64_t*>(mp.combs), mt.combs.data(), mt.combs.size() * 8, cudaMemcpyHostToDevice, ctx->stream));
    CU(ctx, cudaMemcpyAsync(const_cast<uint64_t*>(mp.cfg_flat_base), mt.flat_base.data(), mt.flat_base.size() * 8,
                            cudaMemcpyHostToDevice, ctx->stream));
    CU(ctx, stream_sync(ctx));         // the tables are pageable host memory
    return SAILOR_OK;
}

}  // namespace

static int plan_mixed_impl(sailor_ctx* ctx, const sailor_mixed_space* s, const sailor_objective* o, uint32_t k,
                           sailor_mixed_result* topk, uint32_t* n_found, sailor_stats* stats) {
    if (!ctx || !s || !o || !topk || !n_found || k == 0) return SAILOR_E_ARG;
    if (k > SAILOR_K_MAX || o->kind > SAILOR_OBJ_MAX_THROUGHPUT_PER_USD) return SAILOR_E_RANGE;
    if (o->flags != 0 || o->budget_factor_over_cheapest > 0.0 || std::isnan(o->budget_usd_per_iter) ||
        std::isnan(o->min_iters_per_s) || std::isnan(o->budget_factor_over_cheapest))
        return SAILOR_E_ARG;
    DeviceGuard guard(ctx->device);
    const bool known = ctx->mix && same_mixed_space(ctx->mix->key, *s, ctx->hdr.T);
    if (!known) {                      // a space not searched last: its tables, laid out once
        std::unique_ptr<MixedTables> fresh(new MixedTables());
        const int rc = build_mixed_tables(ctx, s, *fresh);
        if (rc) return rc;
        fresh->key = *s;
        delete ctx->mix;               // nothing of it is in flight: every search ends synchronised
        ctx->mix = nullptr;
        const int rc_up = mixed_workspace(ctx, *fresh);
        if (rc_up) return rc_up;
        ctx->mix = fresh.release();
    }
    const MixedTables& mt = *ctx->mix;
    const uint64_t n_total = mt.flat_base[mt.n_config];
    const uint32_t grid = (uint32_t)ctx->sm_count * 4;
    MixedSearchParams mp;
    memset(&mp, 0, sizeof(mp));
    mixed_carve(ctx, mt, mp);
    if (ctx->mix_dirty) {              // afterwards every search leaves the counters at their starting values
        CU(ctx, cudaMemsetAsync(mp.counters, 0, MIXC_N * 8, ctx->stream));
        CU(ctx, cudaMemsetAsync(mp.counters + MIXC_MIN_COST, 0x7f, 8, ctx->stream));
    }
    ctx->mix_dirty = true;             // until this call has gone through
    CU(ctx, cudaHostGetDevicePointer(reinterpret_cast<void**>(&mp.out), &ctx->host->mixed, 0));
    mp.blob = ctx->d_blob; mp.sp = mt.desc; mp.n_config = mt.n_config; mp.k = k; mp.obj = o->kind;
    memcpy(mp.avail, ctx->h_avail, sizeof(mp.avail));
    mp.n_partial = grid; mp.n_total = n_total; mp.budget = o->budget_usd_per_iter; mp.min_rate = o->min_iters_per_s;
    bool deep = false;                                           // pipelines of more than 32 stages in the space
    for (uint32_t i = 0; i < s->n_p; ++i) deep = deep || s->p_values[i] > 32;
    uint32_t launches = 0;
    for (uint64_t lo = 0; lo < n_total; lo += MIXED_RANGE) {
        mp.range_lo = lo;
        mp.range_hi = std::min(n_total, lo + MIXED_RANGE);
        mp.carry_lists = lo ? 1u : 0u;
        if (lo) CU(ctx, cudaMemsetAsync(mp.counters + MIXC_QUEUED, 0, 8, ctx->stream));
        // a block takes at least a few rounds of candidates, since it sets its configuration up first
        const uint64_t stretches = (mp.range_hi - lo + 2 * MIXS_THREADS - 1) / (2 * MIXS_THREADS);
        const uint32_t class_grid = (uint32_t)std::min<uint64_t>(stretches, (uint64_t)ctx->sm_count * 8);
        mixed_class_kernel<<<class_grid, MIXS_THREADS, 0, ctx->stream>>>(mp);
        CU(ctx, cudaGetLastError());
        plan_mixed_kernel<<<grid, MIXS_THREADS, 0, ctx->stream>>>(mp);
        CU(ctx, cudaGetLastError());
        launches += 2;
    }
    if (deep) mixed_finish_kernel<true><<<1, 32 * MIXF_WARPS<true>, mixed_finish_smem<true>(ctx->hdr), ctx->stream>>>(mp);
    else mixed_finish_kernel<false><<<1, 32 * MIXF_WARPS<false>, mixed_finish_smem<false>(ctx->hdr), ctx->stream>>>(mp);
    CU(ctx, cudaGetLastError());
    ++launches;
    CU(ctx, stream_sync(ctx));
    const unsigned long long* counters = ctx->host->mixed.counters;
    if (counters[MIXC_ERROR]) return SAILOR_E_DEVICE;
    if (counters[MIXC_FOUND] > k) return SAILOR_E_DEVICE;
    ctx->mix_dirty = false;
    *n_found = (uint32_t)counters[MIXC_FOUND];
    memcpy(topk, ctx->host->mixed.results, sizeof(sailor_mixed_result) * counters[MIXC_FOUND]);
    if (stats) {
        memset(stats, 0, sizeof(*stats));
        stats->n_total = counters[0];
        stats->n_invalid = counters[1];
        stats->n_oom = counters[2];
        stats->n_over_avail = counters[3];
        stats->n_over_constraint = counters[4];
        stats->n_feasible = counters[5];
        stats->budget_used = o->budget_usd_per_iter;
        double mc;
        memcpy(&mc, &counters[MIXC_MIN_COST], sizeof(mc));
        stats->min_feasible_cost = counters[5] ? mc : 0.0;
        stats->kernel_ms = span_ms(ctx->host->mixed.span);
        stats->n_launches = launches;
        stats->n_configs = stats->n_configs_evaluated = mt.n_config;
    }
    return SAILOR_OK;
}

extern "C" int sailor_mixed_space_size(const sailor_ctx* ctx, const sailor_mixed_space* s, uint64_t* n_out) {
    if (!n_out) return SAILOR_E_ARG;
    try {
        MixedTables mt;
        const int rc = build_mixed_tables(ctx, s, mt);
        if (rc) return rc;
        *n_out = mt.flat_base[mt.n_config];
        return SAILOR_OK;
    } catch (const std::bad_alloc&) { return SAILOR_E_NOMEM; } catch (...) { return SAILOR_E_ARG; }
}

extern "C" int sailor_mixed_decode(const sailor_ctx* ctx, const sailor_mixed_space* s, uint64_t flat, sailor_mixed_plan* out) {
    if (!out) return SAILOR_E_ARG;
    try {
        MixedTables mt;
        const int rc = build_mixed_tables(ctx, s, mt);
        if (rc) return rc;
        if (flat >= mt.flat_base[mt.n_config]) return SAILOR_E_RANGE;
        const uint32_t c = (uint32_t)(std::upper_bound(mt.flat_base.begin(), mt.flat_base.end(), flat) - mt.flat_base.begin()) - 1;
        const MixedConfig k = mixed_config_of(mt.desc, c);
        const uint64_t radix = (uint64_t)ctx->hdr.Z * mt.desc.n_comb[k.di];
        uint64_t rem = flat - mt.flat_base[c];
        uint32_t digit[SAILOR_SEG_MAX] = {0, 0, 0, 0};
        for (uint32_t q = k.nseg; q-- > 0;) { digit[q] = (uint32_t)(rem % radix); rem /= radix; }
        memset(out, 0, sizeof(*out));
        out->P = (uint8_t)k.P; out->mbs_idx = (uint8_t)k.mi; out->rc = (uint8_t)k.rc; out->D = (uint16_t)k.D;
        for (uint32_t i = 0; i < k.P; ++i) mixed_build_stage(mt.desc, k, ctx->hdr.T, mt.combs.data(), digit, i, &out->stage[i]);
        return SAILOR_OK;
    } catch (const std::bad_alloc&) { return SAILOR_E_NOMEM; } catch (...) { return SAILOR_E_ARG; }
}

extern "C" int sailor_plan_mixed(sailor_ctx* ctx, const sailor_mixed_space* s, const sailor_objective* o, uint32_t k,
                                 sailor_mixed_result* topk, uint32_t* n_found, sailor_stats* stats) {
    try {
        return plan_mixed_impl(ctx, s, o, k, topk, n_found, stats);
    } catch (const std::bad_alloc&) { return SAILOR_E_NOMEM; } catch (...) { return SAILOR_E_ARG; }
}

// What a device-side batch leaves behind when a bounded wait in it ran out.  No input makes one run out, so tests of how
// the fault is reported put it there from the host; not part of the interface.
extern "C" int sailor_internal_post_batch_fault(sailor_ctx* ctx) {
    if (!ctx) return SAILOR_E_ARG;
    *const_cast<volatile unsigned int*>(&ctx->host->sim_error) = SIM_ERR_DEVICE;
    return SAILOR_OK;
}

// ---- sustained issue rates (measurement) ---------------------------------------------------------------

extern "C" int sailor_measure_issue_rates(int cuda_device, void* cuda_stream, uint32_t repeats, sailor_issue_rates* out) {
    if (!out || repeats == 0) return SAILOR_E_ARG;
    memset(out, 0, sizeof(*out));
    DeviceGuard guard(cuda_device);
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    cudaDeviceProp prop;
    if (cudaGetDeviceProperties(&prop, cuda_device) != cudaSuccess) return SAILOR_E_CUDA;
    double* sink = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (cudaMalloc(&sink, sizeof(double)) != cudaSuccess) return SAILOR_E_CUDA;
    int rc = SAILOR_OK;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) rc = SAILOR_E_CUDA;
    const uint32_t grid = (uint32_t)prop.multiProcessorCount * 4, iters = 2048;
    const uint64_t per_run = (uint64_t)grid * (PEAK_THREADS / 32) * iters * PEAK_CHAINS * PEAK_ROUNDS;
    float best[3] = {0.f, 0.f, 0.f};
    for (int kind = 0; kind < 3 && rc == SAILOR_OK; ++kind) {
        for (uint32_t r = 0; r <= repeats && rc == SAILOR_OK; ++r) {        // run 0 warms up
            cudaEventRecord(e0, stream);
            // multipliers just below one and small addends keep every chain finite for any run length
            if (kind == PEAK_FFMA) issue_stream_kernel<PEAK_FFMA><<<grid, PEAK_THREADS, 0, stream>>>(iters, 0.999f, 0.5f, 0, 0, 0.0, sink);
            else if (kind == PEAK_IMAD) issue_stream_kernel<PEAK_IMAD><<<grid, PEAK_THREADS, 0, stream>>>(iters, 0.f, 0.f, 2654435761u, 12345u, 0.0, sink);
            else issue_stream_kernel<PEAK_DADD><<<grid, PEAK_THREADS, 0, stream>>>(iters, 0.f, 0.f, 0, 0, 0.25, sink);
            cudaEventRecord(e1, stream);
            float ms = 0.f;
            if (cudaGetLastError() != cudaSuccess || cudaEventSynchronize(e1) != cudaSuccess ||
                cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess)
                rc = SAILOR_E_CUDA;
            else if (r > 0 && ms > 0.f && (best[kind] == 0.f || ms < best[kind])) best[kind] = ms;
        }
    }
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    cudaFree(sink);
    if (rc) return rc;
    out->ffma_ms = best[0]; out->imad_ms = best[1]; out->dadd_ms = best[2];
    out->ffma_warp_inst_per_s = best[0] > 0.f ? (double)per_run / (best[0] * 1e-3) : 0.0;
    out->imad_warp_inst_per_s = best[1] > 0.f ? (double)per_run / (best[1] * 1e-3) : 0.0;
    out->dadd_warp_inst_per_s = best[2] > 0.f ? (double)per_run / (best[2] * 1e-3) : 0.0;
    out->sm_count = (uint32_t)prop.multiProcessorCount;
    out->warp_inst_per_run = per_run;
    return SAILOR_OK;
}

// ---- entry points that build host-side tables: no exception may cross the C boundary -------------------

#define SAILOR_NO_THROW(call)                              \
    try {                                                  \
        return call;                                       \
    } catch (const std::bad_alloc&) {                      \
        return SAILOR_E_NOMEM;                             \
    } catch (...) {                                        \
        return SAILOR_E_ARG;                               \
    }

extern "C" {

int sailor_create(const sailor_model* m, const sailor_profile* p, const sailor_cluster* c, int cuda_device,
                  void* cuda_stream, sailor_ctx** out) {
    SAILOR_NO_THROW(create_impl(m, p, c, cuda_device, cuda_stream, out))
}

int sailor_plan_range(sailor_ctx* ctx, const sailor_space* s, const sailor_objective* o, uint64_t flat_lo,
                      uint64_t flat_hi, uint32_t k, sailor_result* topk, uint32_t* n_found, sailor_stats* stats) {
    SAILOR_NO_THROW(plan_range_impl(ctx, s, o, flat_lo, flat_hi, k, topk, n_found, stats))
}

int sailor_plan_dp(sailor_ctx* ctx, const sailor_space* s, const sailor_zone_order* orders, uint32_t n_orders,
                   const sailor_objective* o, uint64_t workspace_bytes, uint32_t k, sailor_dp_result* topk,
                   uint32_t* n_found, sailor_dp_stats* stats) {
    SAILOR_NO_THROW(plan_dp_impl(ctx, s, orders, n_orders, o, workspace_bytes, k, topk, n_found, stats))
}

}  // extern "C"
