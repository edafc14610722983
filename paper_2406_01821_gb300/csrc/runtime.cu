// Runtime: errors, contexts, dataset registration (feature-major, label-grouped, on device).
#include <cstdarg>
#include <cstring>
#include <cudaTypedefs.h>

#include "rs_internal.cuh"
#include "block_scan.cuh"
#include "dataset_lru.h"
#include "tma.cuh"

namespace rs {

// ------------------------------------------------------------------------------ errors

static thread_local std::string g_last_error;

void set_error(const char *fmt, ...)
{
    char buf[1024];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    g_last_error = buf;
}

const char *last_error() { return g_last_error.c_str(); }

static std::mutex g_inject_mu;
static int32_t g_inject_skip = 0, g_inject_fail = 0;
static std::atomic<bool> g_inject_armed{false};

void set_injected_alloc_failures(int32_t skip, int32_t count)
{
    std::lock_guard<std::mutex> lk(g_inject_mu);
    g_inject_skip = skip;
    g_inject_fail = count;
    g_inject_armed.store(count > 0);
}

bool take_injected_alloc_failure()
{
    if (!g_inject_armed.load(std::memory_order_relaxed)) return false;
    std::lock_guard<std::mutex> lk(g_inject_mu);
    if (g_inject_skip > 0) { --g_inject_skip; return false; }
    if (g_inject_fail > 0) {
        if (--g_inject_fail == 0) g_inject_armed.store(false);
        return true;
    }
    return false;
}

// A bounded wait on an mbarrier that nothing completes: the wait must give up within limit_ns.
__global__ void k_bounded_wait_selftest(uint64_t limit_ns, uint32_t *status)
{
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    const bool landed = mbar_wait_bounded(&bar, 0, limit_ns);
    if (!__syncthreads_and(landed) && threadIdx.x == 0) atomicOr(status, ST_WAIT_TIMEOUT);
}

rs_status selftest_bounded_wait(Ctx *ctx, int64_t limit_ns, cudaStream_t stream)
{
    const uint64_t lim = (uint64_t)std::min<int64_t>(std::max<int64_t>(limit_ns, 1000000), 2000000000);
    uint32_t *d = nullptr;
    RS_CUDA(cudaMallocAsync(&d, sizeof(uint32_t), stream));
    RS_CUDA(cudaMemsetAsync(d, 0, sizeof(uint32_t), stream));
    k_bounded_wait_selftest<<<1, 32, 0, stream>>>(lim, d);
    count_launch(ctx);
    uint32_t h = 0;
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, d, sizeof(uint32_t), cudaMemcpyDeviceToHost, stream);
    cudaFreeAsync(d, stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    if (e != cudaSuccess) return cuda_fail(e, "bounded-wait self-test");
    if (h & ST_WAIT_TIMEOUT) {
        set_error("device wait gave up after %.1f ms (self-test)", (double)lim / 1e6);
        return RS_ERR_TIMEOUT;
    }
    return RS_OK;
}

rs_status cuda_fail(cudaError_t e, const char *what)
{
    set_error("CUDA error %d (%s) in %s", (int)e, cudaGetErrorString(e), what);
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        return RS_ERR_OOM;
    }
    return RS_ERR_DEVICE;
}

std::string status_text(uint32_t st)
{
    std::string s;
    auto add = [&](uint32_t bit, const char *t) {
        if (st & bit) { if (!s.empty()) s += ", "; s += t; }
    };
    add(ST_BAD_OFFSETS, "malformed offset arrays");
    add(ST_BAD_CLASS, "class id out of range");
    add(ST_BAD_FEATURE, "feature index out of range");
    add(ST_BAD_OP, "comparison op not 0 ('>') or 1 ('<')");
    add(ST_BAD_LABEL, "label out of range");
    add(ST_TOO_LARGE, "a set exceeds the soft path's rule or condition limit");
    add(ST_WAIT_TIMEOUT, "device wait limit reached");
    add(ST_QUEUE_TIMEOUT, "work queue wait limit reached");
    return s;
}

uint32_t *host_status_slot()
{
    // one pinned word per host thread, allocated on first use and kept for the thread's life
    struct Slot {
        uint32_t *p = nullptr;
        ~Slot() { if (p) cudaFreeHost(p); }
    };
    static thread_local Slot slot;
    if (!slot.p) {
        if (cudaHostAlloc(&slot.p, 64, cudaHostAllocDefault) != cudaSuccess) {
            cudaGetLastError();
            slot.p = nullptr;
        }
    }
    return slot.p;
}

rs_status device_guard(Ctx *ctx)
{
    int cur = -1;
    RS_CUDA(cudaGetDevice(&cur));
    if (cur != ctx->device) RS_CUDA(cudaSetDevice(ctx->device));
    return RS_OK;
}

std::shared_ptr<Dataset> find_dataset(Ctx *ctx, uint64_t ds)
{
    std::lock_guard<std::mutex> lk(ctx->mu);
    auto it = ctx->datasets.find(ds);
    if (it == ctx->datasets.end()) return nullptr;
    return it->second;
}

// ------------------------------------------------------------------------------ profiling

static cudaEvent_t take_event(Profiler &p)
{
    if (!p.pool.empty()) { cudaEvent_t e = p.pool.back(); p.pool.pop_back(); return e; }
    cudaEvent_t e = nullptr;
    if (cudaEventCreate(&e) != cudaSuccess) { cudaGetLastError(); return nullptr; }
    return e;
}

TimedLaunch::TimedLaunch(Ctx *c, int k, cudaStream_t s) : ctx(c), kind(k), stream(s)
{
    if (!(ctx->flags & RS_CTX_PROFILE)) return;
    std::lock_guard<std::mutex> lk(ctx->prof.mu);
    e0 = take_event(ctx->prof);
    e1 = take_event(ctx->prof);
    if (e0) cudaEventRecord(e0, stream);
}

TimedLaunch::~TimedLaunch()
{
    if (!e0 || !e1) return;
    cudaEventRecord(e1, stream);
    std::lock_guard<std::mutex> lk(ctx->prof.mu);
    ctx->prof.pending.push_back({e0, e1, kind});
}

rs_status profile_read(Ctx *ctx, rs_profile *out, int reset)
{
    std::lock_guard<std::mutex> lk(ctx->prof.mu);
    for (auto &p : ctx->prof.pending) {
        RS_CUDA(cudaEventSynchronize(p.e1));
        float ms = 0.f;
        RS_CUDA(cudaEventElapsedTime(&ms, p.e0, p.e1));
        ctx->prof.n[p.kind] += 1;
        ctx->prof.ms[p.kind] += ms;
        ctx->prof.pool.push_back(p.e0);
        ctx->prof.pool.push_back(p.e1);
    }
    ctx->prof.pending.clear();
    unsigned long long w[4] = {0, 0, 0, 0};
    const bool walked = ctx->d_walked && (ctx->flags & RS_CTX_COUNT_WORK);
    if (walked) {
        RS_CUDA(cudaDeviceSynchronize());
        RS_CUDA(cudaMemcpy(w, ctx->d_walked, sizeof(w), cudaMemcpyDeviceToHost));
    }
    if (out) {
        out->launches = ctx->prof.launches.load();
        out->hard_launches = ctx->prof.n[TK_HARD];
        out->hard_ms = ctx->prof.ms[TK_HARD];
        out->soft_launches = ctx->prof.n[TK_SOFT];
        out->soft_ms = ctx->prof.ms[TK_SOFT];
        out->hard_records_walked = (int64_t)w[0];
        out->hard_rows_walked = (int64_t)w[1];
        out->hard_rule_ends_walked = (int64_t)w[2];
        out->hard_set_tiles = (int64_t)w[3];
    }
    if (reset) {
        ctx->prof.launches = 0;
        ctx->prof.n[0] = ctx->prof.n[1] = 0;
        ctx->prof.ms[0] = ctx->prof.ms[1] = 0;
        if (walked) RS_CUDA(cudaMemset(ctx->d_walked, 0, sizeof(w)));
    }
    return RS_OK;
}

// ------------------------------------------------------------------------------ registration

namespace {

constexpr int REG_BLOCK = 1024;

// Per block of REG_BLOCK samples: label histogram and each sample's rank among earlier samples
// of the same label in the block (a stable order within the block). The lanes of a warp that share a
// label find each other with one match; the warps add to the block's counts in turn. (A loop over
// the earlier samples of the block, as before, took 25 us on 300,000 samples; this takes 5.)
__global__ void k_label_rank(const int32_t *y, int64_t N, int K, int32_t *blk_count,
                             int32_t *rank, uint32_t *status)
{
    extern __shared__ int32_t hist[];  // [K]
    const int64_t n = (int64_t)blockIdx.x * REG_BLOCK + threadIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int k = threadIdx.x; k < K; k += blockDim.x) hist[k] = 0;
    int lab = -1;
    if (n < N) {
        lab = y[n];
        if (lab < 0 || lab >= K) { atomicOr(status, ST_BAD_LABEL); lab = -1; }
    }
    const uint32_t same = __match_any_sync(0xFFFFFFFFu, lab);
    const int within = __popc(same & ((1u << lane) - 1u));
    int base = 0;
    for (int w = 0; w < REG_BLOCK / 32; ++w) {
        __syncthreads();
        if (w != warp) continue;
        if (lab >= 0) base = hist[lab];
        __syncwarp();
        if (lab >= 0 && within == 0) hist[lab] = base + __popc(same);
    }
    __syncthreads();
    if (n < N) rank[n] = base + within;
    for (int k = threadIdx.x; k < K; k += blockDim.x)
        blk_count[(int64_t)blockIdx.x * K + k] = hist[k];
}

// One CTA per label: exclusive offsets of every block within the label-grouped order.
__global__ void k_label_offsets(int32_t *blk_count, int64_t nblk, int K, int64_t *class_total)
{
    const int k = blockIdx.x;
    int run = 0;
    for (int64_t b0 = 0; b0 < nblk; b0 += blockDim.x) {
        const int64_t b = b0 + threadIdx.x;
        const int c = b < nblk ? blk_count[b * K + k] : 0;
        int total;
        const int before = block_exclusive_scan(c, &total);
        if (b < nblk) blk_count[b * K + k] = run + before;
        run += total;
    }
    if (threadIdx.x == 0) class_total[k] = run;
}

__global__ void k_class_start(const int64_t *class_total, int K, int64_t *class_start)
{
    int run = 0;
    for (int k0 = 0; k0 < K; k0 += blockDim.x) {
        const int k = k0 + threadIdx.x;
        int total;
        const int before = block_exclusive_scan(k < K ? (int)class_total[k] : 0, &total);
        if (k < K) class_start[k] = run + before;
        run += total;
    }
}

__global__ void k_label_scatter(const int32_t *y, int64_t N, int64_t n_pad, int K, const int32_t *blk_off,
                                const int64_t *class_start, const int32_t *rank, int32_t *perm,
                                int32_t *inv, int32_t *y_sorted, const uint32_t *status)
{
    const int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= n_pad || *status) return;
    if (n >= N) { y_sorted[n] = -1; return; }
    const int lab = y[n];
    const int64_t blk = n / REG_BLOCK;
    const int64_t pos = class_start[lab] + blk_off[blk * K + lab] + rank[n];
    perm[pos] = (int32_t)n;
    inv[n] = (int32_t)pos;
    y_sorted[pos] = lab;
}

// Positions of a warp's 128 keys (lane l: the keys of samples l + 32 v) in ascending order, equal keys
// in sample order. The keys alone are sorted, by a bitonic network with lane l holding places 4 l ..
// 4 l + 3, and each key is then looked up in the sorted column: seven search steps cost less than
// carrying the sample number through the network as 64-bit keys (28 stages of two shuffles and a
// 64-bit compare-exchange). Equal keys find the same place and are told apart by a match.
// sorted: the warp's 128 words.
__device__ __forceinline__ void rank_column(const uint32_t (&key)[4], uint32_t *sorted, int lane, uint32_t (&pos)[4])
{
    uint32_t a[4] = {key[0], key[1], key[2], key[3]};
#pragma unroll
    for (int k = 2; k <= RANK_TILE; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            if (j >= 4) {                            // partners in lane ^ (j / 4), same slot
                const bool low = ((4 * lane & j) == 0) == ((4 * lane & k) == 0);
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    const uint32_t o = __shfl_xor_sync(0xFFFFFFFFu, a[v], j >> 2);
                    a[v] = low ? min(a[v], o) : max(a[v], o);
                }
            } else {                                 // partners within the lane
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    if (v & j) continue;
                    const bool asc = ((4 * lane + v) & k) == 0;
                    const uint32_t lo = min(a[v], a[v | j]), hi = max(a[v], a[v | j]);
                    a[v] = asc ? lo : hi;
                    a[v | j] = asc ? hi : lo;
                }
            }
        }
    }
    reinterpret_cast<uint4 *>(sorted)[lane] = make_uint4(a[0], a[1], a[2], a[3]);
    const uint32_t next = __shfl_down_sync(0xFFFFFFFFu, a[0], 1);
    const bool ties = __any_sync(0xFFFFFFFFu, a[0] == a[1] || a[1] == a[2] || a[2] == a[3] || (lane < 31 && a[3] == next));
    __syncwarp();
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        uint32_t p = 0;
#pragma unroll
        for (uint32_t step = RANK_TILE / 2; step >= 1; step >>= 1)
            if (sorted[p + step - 1] < key[v]) p += step;
        pos[v] = p;
    }
    if (!ties) return;
    __syncwarp();
    reinterpret_cast<uint4 *>(sorted)[lane] = make_uint4(0u, 0u, 0u, 0u);      // now: keys seen per place
    __syncwarp();
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        const uint32_t same = __match_any_sync(0xFFFFFFFFu, pos[v]);
        const uint32_t seen = sorted[pos[v]], within = __popc(same & ((1u << lane) - 1u));
        __syncwarp();
        if (within == 0) sorted[pos[v]] = seen + __popc(same);
        __syncwarp();
        pos[v] += seen + within;
    }
}

// One 128-sample tile of 32 features: Xt[f][m] = X[perm[m]][f] (0 for the padding), the tile's rank
// table (with Rk; finite data), and per feature whether it holds a non-finite value (bit 0) or one
// that is no category code 0..63 (bit 1). The rows are gathered into shared memory, so that the
// transpose, the rank sort and the tests read X once and Xt not at all: 300,007 x 96 in one pass where
// a transpose (83 us), a test (21 us) and a sort (338 us) took three: 173 us. Bound by instruction
// issue and shared-memory latency in the sort (260 MB of traffic are 38 us).
constexpr int REG_WARPS = 8;
__global__ void __launch_bounds__(REG_WARPS * 32) k_register_tile(const float *X, int64_t N, int F, int64_t n_pad,
                                                                  const int32_t *perm, float *Xt, uint8_t *Rk,
                                                                  uint32_t *flags, const uint32_t *status)
{
    __shared__ float tile[RANK_TILE][33];
    __shared__ __align__(16) uint32_t sorted[REG_WARPS][RANK_TILE];
    __shared__ __align__(4) uint8_t place[REG_WARPS][RANK_TILE];
    if (*status) return;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t m0 = (int64_t)blockIdx.x * RANK_TILE;
    const int f0 = blockIdx.y * 32;
    constexpr int ROWS = RANK_TILE / REG_WARPS;
    {
        const int64_t m = m0 + w * ROWS + (lane % ROWS);
        const int src = m < N ? perm[m] : -1;
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            const int s = __shfl_sync(0xFFFFFFFFu, src, r);
            tile[w * ROWS + r][lane] = (s >= 0 && f0 + lane < F) ? X[(int64_t)s * F + f0 + lane] : 0.f;
        }
    }
    __syncthreads();
    for (int c = w; c < 32 && f0 + c < F; c += REG_WARPS) {
        const int f = f0 + c;
        float *out = Xt + (int64_t)f * n_pad + m0 + lane;
        uint32_t key[4], pos[4];
        bool odd = false, plain = false;
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const float x = tile[lane + 32 * v][c];
            out[32 * v] = x;
            odd |= !isfinite(x);
            plain |= !(x >= 0.f && x <= 63.f && x == truncf(x));
            const uint32_t u = __float_as_uint(x);
            key[v] = (u & 0x80000000u) ? ~u : (u | 0x80000000u);               // float order
        }
        const uint32_t fl = (__any_sync(0xFFFFFFFFu, odd) ? 1u : 0u) | (__any_sync(0xFFFFFFFFu, plain) ? 2u : 0u);
        if (lane == 0 && (fl & ~__ldcg(flags + f))) atomicOr(flags + f, fl);
        if (!Rk) continue;
        rank_column(key, sorted[w], lane, pos);
        __syncwarp();
#pragma unroll
        for (int v = 0; v < 4; ++v) place[w][lane + 32 * v] = (uint8_t)pos[v];
        __syncwarp();
        reinterpret_cast<uint32_t *>(Rk + (int64_t)f * n_pad + m0)[lane] = reinterpret_cast<const uint32_t *>(place[w])[lane];
    }
}

// status[1]: some value is not finite; status[2]: features that hold category codes only.
__global__ void k_register_summary(const uint32_t *flags, int F, uint32_t *status)
{
    int odd = 0, codes = 0;
    for (int f = threadIdx.x; f < F; f += blockDim.x) {
        odd |= flags[f] & 1u;
        codes += flags[f] == 0u;
    }
    odd = __syncthreads_or(odd);
    int total;
    block_exclusive_scan(codes, &total);
    if (threadIdx.x == 0) {
        status[1] = odd;
        status[2] = total;
    }
}

}  // namespace

static PFN_cuTensorMapEncodeTiled_v12000 get_encode()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        cudaDriverEntryPointQueryResult q;
        void *p = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                             &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
        cudaGetLastError();
    });
    return fn;
}

const CUtensorMap *dataset_rank_tmap(Dataset *ds)
{
    std::lock_guard<std::mutex> lk(ds->mu);
    if (ds->rmap_ok) return &ds->rmap;
    if (!ds->Rk) { set_error("dataset has no rank tables"); return nullptr; }
    auto enc = get_encode();
    if (!enc) { set_error("cuTensorMapEncodeTiled not available"); return nullptr; }
    cuuint64_t dims[2] = {(cuuint64_t)ds->n_pad, (cuuint64_t)ds->F};
    cuuint64_t strides[1] = {(cuuint64_t)ds->n_pad};
    cuuint32_t box[2] = {(cuuint32_t)RANK_TILE, (cuuint32_t)(ds->F < 256 ? ds->F : 256)};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = enc(&ds->rmap, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, ds->Rk, dims, strides, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        set_error("cuTensorMapEncodeTiled failed (%d) for the rank table, F=%d", (int)r, ds->F);
        return nullptr;
    }
    ds->rmap_ok = true;
    return &ds->rmap;
}

const CUtensorMap *dataset_tmap(Dataset *ds, int S)
{
    std::lock_guard<std::mutex> lk(ds->mu);
    auto it = ds->tmaps.find(S);
    if (it != ds->tmaps.end()) return &it->second;
    auto enc = get_encode();
    if (!enc) { set_error("cuTensorMapEncodeTiled not available"); return nullptr; }
    CUtensorMap m;
    cuuint64_t dims[2] = {(cuuint64_t)ds->n_pad, (cuuint64_t)ds->F};
    cuuint64_t strides[1] = {(cuuint64_t)ds->n_pad * sizeof(float)};
    cuuint32_t box[2] = {(cuuint32_t)S, (cuuint32_t)(ds->F < 256 ? ds->F : 256)};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = enc(&m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, ds->Xt, dims, strides, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        set_error("cuTensorMapEncodeTiled failed (%d) for S=%d F=%d", (int)r, S, ds->F);
        return nullptr;
    }
    auto res = ds->tmaps.emplace(S, m);
    return &res.first->second;
}

rs_status dataset_pool_create(Ctx *ctx)
{
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = ctx->device;
    RS_CUDA(cudaMemPoolCreate(&ctx->ds_pool, &props));
    uint64_t keep = DATASET_POOL_KEEP;
    RS_CUDA(cudaMemPoolSetAttribute(ctx->ds_pool, cudaMemPoolAttrReleaseThreshold, &keep));
    RS_CUDA(cudaStreamCreateWithFlags(&ctx->ds_stream, cudaStreamNonBlocking));
    return RS_OK;
}

void dataset_pool_destroy(Ctx *ctx)
{
    if (ctx->ds_stream) {
        cudaStreamSynchronize(ctx->ds_stream);
        cudaStreamDestroy(ctx->ds_stream);
    }
    if (ctx->ds_pool) cudaMemPoolDestroy(ctx->ds_pool);
    ctx->ds_stream = nullptr;
    ctx->ds_pool = nullptr;
}

template <class T>
static cudaError_t ds_alloc(Ctx *ctx, T **p, size_t bytes)
{
    const cudaError_t e = dev_alloc_pool_async(p, bytes, ctx->ds_pool, ctx->ds_stream);
    if (e != cudaSuccess) { *p = nullptr; return e; }
    return cudaStreamSynchronize(ctx->ds_stream);
}

// The caller has seen to it that no device work uses p any more. The pool gives memory beyond
// DATASET_POOL_KEEP back to the driver when its stream is next waited for: ds_settle, after the last
// free of an operation, so that a dropped dataset's memory is there for any other allocator.
static void ds_free(Ctx *ctx, void *p)
{
    if (p) cudaFreeAsync(p, ctx->ds_stream);
}

static void ds_settle(Ctx *ctx) { cudaStreamSynchronize(ctx->ds_stream); }

// Build the device copy of dataset d (N, F, K and n_pad set) from X and y (host or device per
// `mem`): feature-major Xt grouped by label, labels, permutation and inverse, class counts, the
// finite flag and, for finite data of at most RANK_MAX_F features, the rank table. The dataset is one
// allocation (and one for the rank table), the temporary arrays another; the host waits once, at the
// end: every kernel after the label check does nothing when a label was out of range.
static rs_status build_device(Ctx *ctx, Dataset &d, const float *X, const int32_t *y, int32_t mem, cudaStream_t stream)
{
    const int64_t N = d.N;
    const int32_t F = d.F, K = d.K;
    const int64_t nblk = (N + REG_BLOCK - 1) / REG_BLOCK;
    const bool rank_tables = F <= RANK_MAX_F;

    char *own = nullptr, *tmp = nullptr;
    rs_status rc = RS_OK;
    auto fail = [&] {                 // everything taken so far
        cudaStreamSynchronize(stream);
        ds_free(ctx, own); ds_free(ctx, tmp); ds_free(ctx, d.Rk);
        ds_settle(ctx);
        d.Xt = nullptr; d.y = nullptr; d.perm = nullptr; d.inv = nullptr; d.flags = nullptr; d.Rk = nullptr;
    };
#define REG_CUDA(call)                                      \
    do {                                                    \
        cudaError_t e_ = (call);                            \
        if (e_ != cudaSuccess) {                            \
            rc = cuda_fail(e_, #call);                      \
            fail();                                         \
            return rc;                                      \
        }                                                   \
    } while (0)

    const auto up = [](size_t b) { return (b + 255) / 256 * 256; };
    size_t at = 0;
    const auto take = [&](size_t bytes) { const size_t o = at; at += up(bytes); return o; };
    const size_t o_x = take(sizeof(float) * (size_t)d.n_pad * F), o_y = take(sizeof(int32_t) * (size_t)d.n_pad),
                 o_perm = take(sizeof(int32_t) * (size_t)N), o_inv = take(sizeof(int32_t) * (size_t)N),
                 o_flags = take(sizeof(uint32_t) * (size_t)F);
    REG_CUDA(ds_alloc(ctx, &own, at));
    d.Xt = reinterpret_cast<float *>(own + o_x);
    d.y = reinterpret_cast<int32_t *>(own + o_y);
    d.perm = reinterpret_cast<int32_t *>(own + o_perm);
    d.inv = reinterpret_cast<int32_t *>(own + o_inv);
    d.flags = reinterpret_cast<uint32_t *>(own + o_flags);
    at = 0;
    // the status words and the class counts, read back together
    const size_t o_st = take(16 + sizeof(int64_t) * (size_t)K), o_start = take(sizeof(int64_t) * (size_t)K),
                 o_blk = take(sizeof(int32_t) * (size_t)nblk * K), o_rank = take(sizeof(int32_t) * (size_t)N);
    const size_t o_xd = mem == RS_MEM_HOST ? take(sizeof(float) * (size_t)N * F) : 0,
                 o_yd = mem == RS_MEM_HOST ? take(sizeof(int32_t) * (size_t)N) : 0;
    REG_CUDA(ds_alloc(ctx, &tmp, at));
    // The rank table comes last and is not insisted on before the data is known to be finite: data that
    // turns out not to be needs no memory for it.
    cudaError_t rank_alloc = cudaSuccess;
    if (rank_tables && (rank_alloc = ds_alloc(ctx, &d.Rk, (size_t)d.n_pad * F)) != cudaSuccess) {
        if (rank_alloc != cudaErrorMemoryAllocation) REG_CUDA(rank_alloc);
        cudaGetLastError();
    }
    uint32_t *st = reinterpret_cast<uint32_t *>(tmp + o_st);
    int64_t *ctot = reinterpret_cast<int64_t *>(tmp + o_st + 16), *cstart = reinterpret_cast<int64_t *>(tmp + o_start);
    int32_t *blk = reinterpret_cast<int32_t *>(tmp + o_blk), *rank = reinterpret_cast<int32_t *>(tmp + o_rank);
    const float *Xd = X;
    const int32_t *yd = y;
    if (mem == RS_MEM_HOST) {
        REG_CUDA(cudaMemcpyAsync(tmp + o_xd, X, sizeof(float) * (size_t)N * F, cudaMemcpyHostToDevice, stream));
        REG_CUDA(cudaMemcpyAsync(tmp + o_yd, y, sizeof(int32_t) * (size_t)N, cudaMemcpyHostToDevice, stream));
        Xd = reinterpret_cast<const float *>(tmp + o_xd);
        yd = reinterpret_cast<const int32_t *>(tmp + o_yd);
    }
    REG_CUDA(cudaMemsetAsync(st, 0, 16, stream));
    REG_CUDA(cudaMemsetAsync(d.flags, 0, sizeof(uint32_t) * (size_t)F, stream));
    k_label_rank<<<(unsigned)nblk, REG_BLOCK, sizeof(int32_t) * K, stream>>>(yd, N, K, blk, rank, st);
    k_label_offsets<<<K, 1024, 0, stream>>>(blk, nblk, K, ctot);
    k_class_start<<<1, 1024, 0, stream>>>(ctot, K, cstart);
    k_label_scatter<<<(unsigned)((d.n_pad + 255) / 256), 256, 0, stream>>>(yd, N, d.n_pad, K, blk, cstart, rank, d.perm,
                                                                           d.inv, d.y, st);
    const dim3 tg((unsigned)(d.n_pad / RANK_TILE), (unsigned)((F + 31) / 32));
    k_register_tile<<<tg, REG_WARPS * 32, 0, stream>>>(Xd, N, F, d.n_pad, d.perm, d.Xt, d.Rk, d.flags, st);
    k_register_summary<<<1, 1024, 0, stream>>>(d.flags, F, st);
    REG_CUDA(cudaGetLastError());
    std::vector<char> back(16 + sizeof(int64_t) * (size_t)K);
    REG_CUDA(cudaMemcpyAsync(back.data(), st, back.size(), cudaMemcpyDeviceToHost, stream));
    REG_CUDA(cudaStreamSynchronize(stream));
    uint32_t hst[4];
    std::memcpy(hst, back.data(), sizeof(hst));
    if (hst[0]) {
        set_error("dataset rejected: %s", status_text(hst[0]).c_str());
        fail();
        return RS_ERR_INVALID;
    }
    d.class_count.resize(K);
    std::memcpy(d.class_count.data(), back.data() + 16, sizeof(int64_t) * (size_t)K);
    d.finite = hst[1] == 0;
    d.ncode = (int32_t)hst[2];
    if (d.finite) REG_CUDA(rank_alloc);
    d.ranked = d.finite && rank_tables;
    if (!d.ranked && d.Rk) { ds_free(ctx, d.Rk); d.Rk = nullptr; }
    ds_free(ctx, tmp);
    ds_settle(ctx);
#undef REG_CUDA
    return RS_OK;
}

// Device bytes of a dataset: features, labels, order and its inverse, flags, rank table.
static size_t dataset_device_bytes(int64_t N, int64_t n_pad, int32_t F, bool rank_table)
{
    return sizeof(float) * (size_t)n_pad * F + sizeof(int32_t) * ((size_t)n_pad + 2 * (size_t)N + (size_t)F) +
           (rank_table ? (size_t)n_pad * F : 0);
}

static void free_device(Ctx *ctx, Dataset &d)
{
    ds_free(ctx, d.Xt);              // the start of the dataset's own allocation
    ds_free(ctx, d.Rk);
    ds_settle(ctx);
    d.Xt = nullptr; d.y = nullptr; d.perm = nullptr; d.inv = nullptr; d.flags = nullptr; d.Rk = nullptr;
    std::lock_guard<std::mutex> lk(d.mu);
    d.tmaps.clear();                 // tensor maps hold the device addresses
    d.rmap_ok = false;
}

// With ctx->mu held: drop the cached graphs that reference dataset h.
static void drop_graphs(Ctx *ctx, uint64_t h)
{
    const std::string key = "ds" + std::to_string(h) + "|";
    for (auto g = ctx->graphs.begin(); g != ctx->graphs.end();) {
        if (g->first.rfind(key, 0) == 0) g = ctx->graphs.erase(g);
        else ++g;
    }
}

// With ctx->mu held: return the dataset's completed in-flight marks to the spare events; true if
// none is left (no call's device work on it is pending, as far as the marks tell).
static bool reap_marks(Ctx *ctx, Dataset &d)
{
    auto &v = d.inflight;
    for (size_t i = 0; i < v.size();) {
        const cudaError_t q = cudaEventQuery(v[i]);
        if (q == cudaErrorNotReady) { ++i; continue; }
        cudaGetLastError();
        ctx->ds_events.push_back(v[i]);
        v[i] = v.back();
        v.pop_back();
    }
    return v.empty();
}

void mark_dataset_use(Ctx *ctx, Dataset *ds, cudaStream_t stream, bool may_create)
{
    std::lock_guard<std::mutex> lk(ctx->mu);
    // without a host copy it is never evicted; with one it is marked under no budget too: a budget set
    // while the call's work is still queued must not take its memory
    if (!ctx->ds_budget && ds->hy.empty()) return;
    reap_marks(ctx, *ds);
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(stream, &cap) != cudaSuccess) { cudaGetLastError(); cap = cudaStreamCaptureStatusActive; }
    cudaEvent_t ev = nullptr;
    if (cap == cudaStreamCaptureStatusNone) {
        if (!ctx->ds_events.empty()) {
            ev = ctx->ds_events.back();
            ctx->ds_events.pop_back();
        } else if (!may_create || cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess) {
            cudaGetLastError();
            ev = nullptr;
        }
    }
    if (ev && cudaEventRecord(ev, stream) == cudaSuccess) {
        ds->inflight.push_back(ev);
        return;
    }
    cudaGetLastError();
    if (ev) ctx->ds_events.push_back(ev);
    ds->unmarked_use = true;         // its eviction waits for the whole device
}

void release_dataset_events(Ctx *ctx)
{
    std::lock_guard<std::mutex> lk(ctx->mu);
    for (auto &kv : ctx->datasets) {
        for (cudaEvent_t e : kv.second->inflight) cudaEventDestroy(e);
        kv.second->inflight.clear();
    }
    for (cudaEvent_t e : ctx->ds_events) cudaEventDestroy(e);
    ctx->ds_events.clear();
}

// With ctx->mu held: evict least recently used datasets so that `need` more device bytes fit the
// budget (dataset_lru.h), `keep` excepted.
static void make_room(Ctx *ctx, size_t need, uint64_t keep)
{
    if (!ctx->ds_budget) return;
    std::vector<lru::Entry> entries;
    for (auto &kv : ctx->datasets) {
        Dataset &d = *kv.second;
        // the registry's own reference is the only one (no call or request holds the dataset), and
        // the device work of the calls that used it has completed, or is unknown (then waited for)
        const bool idle = kv.second.use_count() == 1 && (!d.resident || reap_marks(ctx, d));
        entries.push_back({kv.first, d.dev_bytes, d.last_use, d.resident, !d.hy.empty() && idle});
    }
    const std::vector<uint64_t> v = lru::victims(entries, ctx->ds_resident, need, ctx->ds_budget, keep);
    if (v.empty()) return;
    bool unmarked = false;
    for (uint64_t h : v) unmarked |= ctx->datasets[h]->unmarked_use;
    if (unmarked) cudaDeviceSynchronize();   // work that no mark covers finishes first
    for (uint64_t h : v) {
        Dataset &d = *ctx->datasets[h];
        drop_graphs(ctx, h);
        free_device(ctx, d);
        d.resident = false;
        d.unmarked_use = false;
        ctx->ds_resident -= std::min(ctx->ds_resident, d.dev_bytes);
        ++ctx->ds_evictions;
    }
}

rs_status dataset_create(Ctx *ctx, const float *X, const int32_t *y, int64_t N, int32_t F,
                         int32_t K, int32_t mem, cudaStream_t stream, uint64_t *out)
{
    if (!X || !y || !out) { set_error("null pointer"); return RS_ERR_INVALID; }
    if (N < 1 || N > (int64_t)INT32_MAX - 1024 || F < 1 || F > RS_MAX_FEATURES || K < 1 ||
        K > RS_MAX_CLASSES) {
        set_error("dataset shape out of range (N=%lld F=%d K=%d)", (long long)N, F, K);
        return RS_ERR_INVALID;
    }
    if (mem != RS_MEM_HOST && mem != RS_MEM_DEVICE) { set_error("bad mem kind"); return RS_ERR_INVALID; }
    auto ds = std::make_shared<Dataset>();
    ds->N = N;
    ds->F = F;
    ds->K = K;
    ds->n_pad = (N + 255) / 256 * 256;
    bool budget = false;
    {
        std::lock_guard<std::mutex> lk(ctx->mu);
        budget = ctx->ds_budget != 0;
        if (budget)                   // room for the largest form it can take (with a rank table)
            make_room(ctx, dataset_device_bytes(N, ds->n_pad, F, F <= RANK_MAX_F), 0);
    }
    if (budget) {                     // the host copy an eviction rebuilds from
        ds->hX.resize((size_t)N * F);
        ds->hy.resize((size_t)N);
        const cudaMemcpyKind kind = mem == RS_MEM_HOST ? cudaMemcpyHostToHost : cudaMemcpyDeviceToHost;
        cudaError_t e = cudaMemcpy(ds->hX.data(), X, sizeof(float) * (size_t)N * F, kind);
        if (e == cudaSuccess) e = cudaMemcpy(ds->hy.data(), y, sizeof(int32_t) * (size_t)N, kind);
        if (e != cudaSuccess) return cuda_fail(e, "dataset host copy");
    }
    const rs_status rc = build_device(ctx, *ds, X, y, mem, stream);
    if (rc) return rc;
    ds->dev_bytes = dataset_device_bytes(N, ds->n_pad, F, ds->Rk != nullptr);
    std::lock_guard<std::mutex> lk(ctx->mu);
    const uint64_t h = ctx->next_ds++;
    ds->last_use = ++ctx->ds_tick;
    ctx->ds_resident += ds->dev_bytes;
    ctx->datasets[h] = ds;
    *out = h;
    return RS_OK;
}

rs_status use_dataset(Ctx *ctx, uint64_t h, std::shared_ptr<Dataset> *out)
{
    std::lock_guard<std::mutex> lk(ctx->mu);
    auto it = ctx->datasets.find(h);
    if (it == ctx->datasets.end()) {
        set_error("unknown dataset %llu", (unsigned long long)h);
        return RS_ERR_NOT_FOUND;
    }
    Dataset &d = *it->second;
    d.last_use = ++ctx->ds_tick;
    if (!d.resident) {                // evicted: rebuild it from the host copy
        rs_status rc = device_guard(ctx);
        if (rc) return rc;
        make_room(ctx, d.dev_bytes, h);
        if ((rc = build_device(ctx, d, d.hX.data(), d.hy.data(), RS_MEM_HOST, nullptr))) return rc;
        d.resident = true;
        ctx->ds_resident += d.dev_bytes;
        ++ctx->ds_rebuilds;
    }
    *out = it->second;
    return RS_OK;
}

rs_status set_dataset_budget(Ctx *ctx, uint64_t bytes)
{
    std::lock_guard<std::mutex> lk(ctx->mu);
    ctx->ds_budget = bytes;
    // the pool keeps no more mapped than a budget allows
    uint64_t keep = bytes ? std::min<uint64_t>(bytes, DATASET_POOL_KEEP) : DATASET_POOL_KEEP;
    RS_CUDA(cudaMemPoolSetAttribute(ctx->ds_pool, cudaMemPoolAttrReleaseThreshold, &keep));
    // spare marks, so that calls that may not create one (the allocation-free entry) find one
    while (bytes && ctx->ds_events.size() < 32) {
        cudaEvent_t e = nullptr;
        if (cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess) { cudaGetLastError(); break; }
        ctx->ds_events.push_back(e);
    }
    make_room(ctx, 0, 0);
    if (bytes) RS_CUDA(cudaMemPoolTrimTo(ctx->ds_pool, keep));
    return RS_OK;
}

rs_status dataset_destroy(Ctx *ctx, uint64_t h, bool force)
{
    std::shared_ptr<Dataset> ds;
    {
        std::lock_guard<std::mutex> lk(ctx->mu);
        auto it = ctx->datasets.find(h);
        if (it == ctx->datasets.end()) { set_error("unknown dataset %llu", (unsigned long long)h); return RS_ERR_NOT_FOUND; }
        // another reference than the registry's: a call running on the dataset, or a serving
        // request on it (queued, running or not yet polled) whose kernels would read the freed copy
        if (!force && it->second.use_count() > 1) {
            set_error("dataset %llu is in use: a call on it is running, or a serving request on it has not "
                      "been polled", (unsigned long long)h);
            return RS_ERR_INVALID;
        }
        ds = it->second;
        ctx->datasets.erase(it);
        drop_graphs(ctx, h);          // cached graphs that reference this dataset
        if (ds->resident) ctx->ds_resident -= std::min(ctx->ds_resident, ds->dev_bytes);
        for (cudaEvent_t e : ds->inflight) ctx->ds_events.push_back(e);   // the device wait below covers them
        ds->inflight.clear();
    }
    RS_CUDA(cudaDeviceSynchronize());
    free_device(ctx, *ds);
    return RS_OK;
}

// Load the kernels of this file now (CUDA loads a kernel lazily at its first launch, which would
// otherwise land on the first request that needs it).
void preload_dataset_kernels()
{
    cudaFuncAttributes fa;
    cudaFuncGetAttributes(&fa, k_label_rank);
    cudaFuncGetAttributes(&fa, k_label_offsets);
    cudaFuncGetAttributes(&fa, k_class_start);
    cudaFuncGetAttributes(&fa, k_label_scatter);
    cudaFuncGetAttributes(&fa, k_register_tile);
    cudaFuncGetAttributes(&fa, k_register_summary);
}

}  // namespace rs
