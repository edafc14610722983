// Rank-coded batch evaluator and direct walk (record format v5); the method and the device code are described in
// eval_rank.cuh.
#include <algorithm>

#include "rs_internal.cuh"
#include "eval_core.cuh"
#include "eval_rank.cuh"
#include "tma.cuh"

namespace rs {

namespace {

using namespace rank;
constexpr uint64_t TMA_WAIT_LIMIT_NS = 2000000000ull;

// PRED: every sample's prediction is written (class counts up to 256), in the caller's sample order:
// four scattered 4-byte stores a lane, which L2 gathers (the store adds 10 to 20 us to 200 sets on
// 100,000 samples). The predicted classes of a lane's samples are the bytes of one word; the walk has
// no class-tail stop, and hits are the bytes equal to the label's.
// DIRECT: the direct walk on datasets without rank tables (tmr unused).
template <int W, bool CAT, bool PRED, bool DIRECT>
__global__ void __launch_bounds__(W * 32, 32 / W) k_hard5(const __grid_constant__ CUtensorMap tmx,
                                                  const __grid_constant__ CUtensorMap tmr, HardArgs a)
{
    extern __shared__ __align__(512) unsigned char smem[];
    const int F = a.F;
    const int Fb = F < 256 ? F : 256;
    const int nbox = (F + Fb - 1) / Fb;
    const int Frows = nbox * Fb;
    unsigned char *xs = smem;                                         // float [Frows][T]
    float *ones = reinterpret_cast<float *>(xs + (size_t)Frows * T * 4);  // [T] of 1.0 (products)
    unsigned char *rs = reinterpret_cast<unsigned char *>(ones + T);  // u8 [Frows][T], then reversed
    uint4 *stage_all = reinterpret_cast<uint4 *>(rs + (DIRECT ? 0 : (size_t)Frows * T * 2));
    constexpr int VS = CAT ? VSLOTS_CAT : VSLOTS;
    uint32_t *vrows = reinterpret_cast<uint32_t *>(stage_all + W * 32);     // [W][VS][32]
    uint64_t *bar = reinterpret_cast<uint64_t *>(vrows + W * VS * 32);
    int *next = reinterpret_cast<int *>(bar + 1);
    uint32_t *walked = reinterpret_cast<uint32_t *>(bar + 2);        // [W][4] work counters (counting)
    int32_t *place = reinterpret_cast<int32_t *>(walked + 4 * W);    // [T] the caller's sample, or -1 (PRED)
    // CAT: the code rows [a.code_rows][32] and each feature's row
    uint2 *codes = reinterpret_cast<uint2 *>(place + T);       // (rank-coded form)
    unsigned char *code_of = reinterpret_cast<unsigned char *>(codes + (CAT ? a.code_rows * 32 : 0));
    float *us = reinterpret_cast<float *>(code_of + (CAT ? (F + 3) / 4 * 4 : 0));   // float [F][US] sorted (built here)
    const uint4 *recs = reinterpret_cast<const uint4 *>(a.recs);

    const TileTask task(a);
    const int tile = task.tile, group = task.group, G = task.groups;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;

    if (threadIdx.x == 0) {
        mbar_init(bar, 1);
        *next = 0;
        fence_mbar_init();
    }
    if (threadIdx.x < 4 * W) walked[threadIdx.x] = 0;
    __syncthreads();
    if (threadIdx.x == 0) {
        mbar_arrive_expect_tx(bar, (uint32_t)Frows * T * (DIRECT ? 4u : 5u));
        for (int b = 0; b < nbox; ++b) {
            tma_load_2d(xs + (size_t)b * Fb * T * 4, &tmx, tile * T, b * Fb, bar);
            if (!DIRECT) tma_load_2d(rs + (size_t)b * Fb * T, &tmr, tile * T, b * Fb, bar);
        }
    }
    if (CAT && !DIRECT && warp == W - 1) {         // number the features that hold category codes only
        int n = 0;
        for (int f0 = 0; f0 < F; f0 += 32) {
            const bool code = f0 + lane < F && a.flags[f0 + lane] == 0u;
            const uint32_t b = __ballot_sync(FULL, code);
            const int row = n + __popc(b & ((1u << lane) - 1u));
            if (f0 + lane < F) code_of[f0 + lane] = code && row < a.code_rows ? (unsigned char)row : (unsigned char)CODE_NONE;
            n += __popc(b);
        }
    }
    const int32_t *yl = a.y + (int64_t)tile * T + lane * 4;   // n_pad is a multiple of T
    const int64_t t_last = min((int64_t)tile * T + T, a.N) - 1;
    const int kmin = a.y[(int64_t)tile * T], kmax = a.y[t_last];
    const bool uniform = kmin == kmax;
    const uint32_t claimed0 = class_bytes(yl, -1);                 // padding samples

    const bool landed = mbar_wait_bounded(bar, 0, TMA_WAIT_LIMIT_NS);
    if (!__syncthreads_and(landed)) {
        if (threadIdx.x == 0) atomicOr(a.status, ST_WAIT_TIMEOUT);
        mbar_wait_bounded(bar, 0, TMA_WAIT_LIMIT_NS);   // copies still in flight land first
        return;
    }
    const uint32_t rev_off = (uint32_t)Frows * T;
    if (DIRECT) {
        core::permute_rows<4>(reinterpret_cast<float *>(xs), F);
    } else if (CAT) {
        build_tile_tables(reinterpret_cast<float *>(xs), rs, rev_off, us, F, code_of, codes);
    } else {
        build_tile_tables(reinterpret_cast<float *>(xs), rs, rev_off, us, F);
    }
    if (threadIdx.x < T) {
        ones[threadIdx.x] = 1.f;
        const int64_t n = (int64_t)tile * T + threadIdx.x;
        if (PRED) place[threadIdx.x] = n < a.N ? a.perm[n] : -1;
    }
    __syncthreads();

    const unsigned char *rl = rs + lane * 4;       // this lane's four rank bytes of row 0
    const uint32_t ones_off = (uint32_t)Frows * T * 4;
    const int count = (a.P - group + G - 1) / G;
    uint4 *st = stage_all + warp * 32;
    uint32_t label4 = 0;                           // the labels of the lane's samples, a byte each
    if (PRED) {
        const int4 y = *reinterpret_cast<const int4 *>(yl);
        label4 = (uint32_t)(y.x & 0xFF) | (uint32_t)(y.y & 0xFF) << 8 | (uint32_t)(y.z & 0xFF) << 16 | (uint32_t)(y.w & 0xFF) << 24;
    }

    while (true) {
        int m = 0;
        if (lane == 0) m = atomicAdd(next, 1);
        m = __shfl_sync(FULL, m, 0);
        if (m >= count) break;
        const int p = a.order[group + m * G];
        const SetInfo si = a.sets[p];
        const int rb = si.rec_begin;
        // one label k in the tile: records after the set's last rule of class k (default of another
        // class) or of any other class (default k) cannot change its count
        const int nrec = (!PRED && uniform && a.last_end)
                             ? min(a.last_end[(int64_t)p * a.K + kmin], si.rec_end - si.rec_begin)
                             : si.rec_end - si.rec_begin;

        uint32_t *vr = vrows + warp * VS * 32;
        const uint32_t vr_off = (uint32_t)(reinterpret_cast<unsigned char *>(vr) - (DIRECT ? xs : rs));
        WalkCount wc;
        int more;
        uint32_t hit;
        if (PRED) {
            const uint32_t pred = walk_set<false, VS, CAT, true, DIRECT>(st, vr, vr_off, lane, recs, rb, nrec, us, rev_off, F, -2, rl,
                                                                 xs, ones_off, yl, claimed0, si.deflt, wc, more, CAT && !DIRECT ? code_of : nullptr, codes);
            const int4 to = *reinterpret_cast<const int4 *>(place + 4 * lane);
            int32_t *out = a.preds + (int64_t)p * a.N;
            if (to.x >= 0) out[to.x] = (int32_t)(pred & 0xFFu);
            if (to.y >= 0) out[to.y] = (int32_t)(pred >> 8 & 0xFFu);
            if (to.z >= 0) out[to.z] = (int32_t)(pred >> 16 & 0xFFu);
            if (to.w >= 0) out[to.w] = (int32_t)(pred >> 24);
            const uint32_t d = pred ^ label4;      // a byte of 0: a hit
            hit = ~(((d & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | d) & HIGH & ~claimed0;
        } else if (uniform) {
            hit = walk_set<true, VS, CAT, false, DIRECT>(st, vr, vr_off, lane, recs, rb, nrec, us, rev_off, F, kmin, rl, xs, ones_off, yl,
                                          claimed0, si.deflt, wc, more, CAT && !DIRECT ? code_of : nullptr, codes);
        } else {
            hit = walk_set<false, VS, CAT, false, DIRECT>(st, vr, vr_off, lane, recs, rb, nrec, us, rev_off, F, -2, rl, xs, ones_off, yl,
                                           claimed0, si.deflt, wc, more, CAT && !DIRECT ? code_of : nullptr, codes);
        }
        if (a.walked && lane == 0) {           // the warp's own slots: no atomics
            uint32_t *wk = walked + 4 * warp;
            wk[0] += wc.records;
            wk[1] += wc.rows;
            wk[2] += wc.ends;
            wk[3] += 1;
        }
        const int hits = __reduce_add_sync(FULL, __popc(hit) + more);
        if (lane == 0 && hits) atomicAdd(&a.correct[p], hits);
        if (a.per_class) {
            if (uniform) {
                if (lane == 0 && hits) atomicAdd(&a.per_class[(int64_t)p * a.K + kmin], hits);
            } else {
                for (int k = kmin; k <= kmax; ++k) {
                    const int ckc = __reduce_add_sync(FULL, __popc(hit & class_bytes(yl, k)));
                    if (lane == 0 && ckc) atomicAdd(&a.per_class[(int64_t)p * a.K + k], ckc);
                }
            }
        }
    }
    if (a.walked && lane < 4) atomicAdd(&a.walked[lane], (unsigned long long)walked[4 * warp + lane]);
}

}  // namespace

// Shared memory but for the tables: stages, pass rows, the ones row, the barrier, counters and places.
static size_t hard5_fixed_bytes(int W)
{
    return (size_t)W * 32 * 16 + (size_t)W * VSLOTS * 32 * 4 + T * 4 + 16 + (size_t)W * 16 + T * 4;
}

static size_t tma_rows(int F)
{
    const int Fb = F < 256 ? F : 256;
    return (size_t)((F + Fb - 1) / Fb) * Fb;
}

size_t hard5_smem_bytes(int F, int W)
{
    return tma_rows(F) * T * (4 + 2) + (size_t)F * US * 4 + hard5_fixed_bytes(W);
}

size_t direct_smem_bytes(int F, int W) { return tma_rows(F) * T * 4 + hard5_fixed_bytes(W); }

template <int W, bool CAT, bool PRED, bool DIRECT>
static rs_status launch5_t(Ctx *ctx, Dataset *ds, HardArgs a, cudaStream_t stream)
{
    size_t smem = DIRECT ? direct_smem_bytes(a.F, W) : hard5_smem_bytes(a.F, W);
    if (smem > ctx->smem_optin || !(DIRECT ? ds->finite : ds->ranked)) return RS_ERR_TOO_LARGE;
    if (CAT && !DIRECT) {
        // fewer pass-row slots make room for the code rows: all of them, or as many as keep the CTAs
        // per SM that the kernel has without them (features beyond them are tested on their floats)
        const size_t most = W == 16 && 2 * (smem + SMEM_RESERVED) <= SMEM_SM ? SMEM_SM / 2 - SMEM_RESERVED : SMEM_CTA;
        smem -= (size_t)W * (VSLOTS - VSLOTS_CAT) * 128;
        smem += (size_t)(a.F + 3) / 4 * 4;
        a.code_rows = (int32_t)std::min<size_t>({(size_t)ds->ncode, (size_t)CODE_NONE, (most - smem) / 256});
        smem += (size_t)a.code_rows * 256;
    }
    static std::once_flag once;
    static cudaError_t attr_err = cudaSuccess;
    std::call_once(once, [&] {
        attr_err = cudaFuncSetAttribute(k_hard5<W, CAT, PRED, DIRECT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)ctx->smem_optin);
    });
    if (attr_err != cudaSuccess) return cuda_fail(attr_err, "cudaFuncSetAttribute(k_hard5)");
    const CUtensorMap *tmx = dataset_tmap(ds, T);
    const CUtensorMap *tmr = DIRECT ? tmx : dataset_rank_tmap(ds);
    if (!tmx || !tmr) return RS_ERR_DEVICE;
    static std::atomic<uint64_t> asked{0};
    const int resident = resident_ctas(asked, k_hard5<W, CAT, PRED, DIRECT>, W * 32, smem);
    const int grid = split_tiles(ctx, a.N, a.F, a.P, T, W, resident, a);
    {
        TimedLaunch tl(ctx, TK_HARD, stream);
        k_hard5<W, CAT, PRED, DIRECT><<<grid, W * 32, smem, stream>>>(*tmx, *tmr, a);
    }
    RS_CUDA(cudaGetLastError());
    count_launch(ctx);
    return RS_OK;
}

template <int W, bool DIRECT>
static rs_status launch5_w(Ctx *ctx, Dataset *ds, const HardArgs &a, cudaStream_t stream)
{
    if (a.preds) return a.cat ? launch5_t<W, true, true, DIRECT>(ctx, ds, a, stream)
                              : launch5_t<W, false, true, DIRECT>(ctx, ds, a, stream);
    return a.cat ? launch5_t<W, true, false, DIRECT>(ctx, ds, a, stream)
                 : launch5_t<W, false, false, DIRECT>(ctx, ds, a, stream);
}

rs_status launch_hard5(Ctx *ctx, Dataset *ds, int W, bool direct, const HardArgs &a, cudaStream_t stream)
{
    if (a.P == 0) return RS_OK;
    if (W == 16) return direct ? launch5_w<16, true>(ctx, ds, a, stream) : launch5_w<16, false>(ctx, ds, a, stream);
    if (W == 32) return direct ? launch5_w<32, true>(ctx, ds, a, stream) : launch5_w<32, false>(ctx, ds, a, stream);
    return RS_ERR_INVALID;
}

// Load the kernels of this file now (CUDA loads a kernel lazily at its first launch, which would
// otherwise land on the first request that needs it).
void preload_hard5_kernels()
{
    cudaFuncAttributes fa;
    cudaFuncGetAttributes(&fa, k_hard5<16, false, false, false>);
    cudaFuncGetAttributes(&fa, k_hard5<16, false, false, true>);
    cudaFuncGetAttributes(&fa, k_hard5<16, false, true, false>);
    cudaFuncGetAttributes(&fa, k_hard5<16, false, true, true>);
    cudaFuncGetAttributes(&fa, k_hard5<16, true, false, false>);
    cudaFuncGetAttributes(&fa, k_hard5<16, true, false, true>);
    cudaFuncGetAttributes(&fa, k_hard5<16, true, true, false>);
    cudaFuncGetAttributes(&fa, k_hard5<16, true, true, true>);
    cudaFuncGetAttributes(&fa, k_hard5<32, false, false, false>);
    cudaFuncGetAttributes(&fa, k_hard5<32, false, false, true>);
    cudaFuncGetAttributes(&fa, k_hard5<32, false, true, false>);
    cudaFuncGetAttributes(&fa, k_hard5<32, false, true, true>);
    cudaFuncGetAttributes(&fa, k_hard5<32, true, false, false>);
    cudaFuncGetAttributes(&fa, k_hard5<32, true, false, true>);
    cudaFuncGetAttributes(&fa, k_hard5<32, true, true, false>);
    cudaFuncGetAttributes(&fa, k_hard5<32, true, true, true>);
}

}  // namespace rs
