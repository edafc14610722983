// The sparse tail of a walk, shared by the rank-coded, the direct and the sign-mask evaluators.
//
// The first rules claim most samples (each of the ragged workload's claims an eighth of
// what is left), so that a set's last chunks are walked for a handful of samples: once at most
// MAX samples are unclaimed, the roles turn (tail). The unclaimed samples are listed, one
// per lane; each lane keeps one record of the chunk, and for one sample after another every lane tests
// its condition (the original compare on the float tile: no cut search, no pass rows, no stage) and a
// vote hands the 32 outcomes to the sample's lane. Each lane then finds its sample's first firing
// rule with one addition.
#pragma once
#include "rs_internal.cuh"

namespace rs {
namespace sparse {

constexpr uint32_t FULL = 0xFFFFFFFFu;

// Unclaimed samples up to which the rest of a set is walked sample by sample (tail). 4096 ragged
// sets on 2^20 x 128: 53.4 ms without it, 46.5 / 45.0 / 45.2 / 45.4 ms with a limit of 8 / 16 / 24 /
// 32; ten evolution generations of 10,000 sets of up to 32 rules on 100,000 x 32: 100.0 and 93.2 /
// 92.2 / 92.5 / 92.5 ms.
constexpr int MAX = 20;

// A dataset's label. LIVE: read through L2 in a kernel that may outlive the dataset at this address: an
// evicted dataset's memory can hold another one's labels while the serving kernel runs on, and a line of
// the read-only or L1 cache would then be stale.
template <bool LIVE, class T>
__device__ __forceinline__ T load_label(const T *p) { return LIVE ? __ldcg(p) : __ldg(p); }

// Work a walk did: records, pair / product / membership conditions and rule ends (profiling counters).
struct WalkCount {
    uint32_t records = 0, rows = 0, ends = 0;
};

// Row of feature f in a shared float tile of BYTES bytes a row: its 16-byte pieces are permuted by
// piece ^ (f & 7), so that one sample's values of 32 features fall on eight groups of banks instead
// of one (the tail reads them so); a warp reading whole rows is unaffected. A staged offset carries
// (f & 7) << 4, and the byte b of the row is at (offset ^ b).
template <int BYTES>
__device__ __host__ __forceinline__ uint32_t row_off(uint32_t f) { return f * BYTES | (f & 7u) << 4; }

// A condition as the tail tests it: fl(A x) > fl(B z), negated by inv; or a membership test (set).
struct Rec {
    uint32_t xo, zo;       // row offsets of x and z (a row of 1.0 where there is no second feature)
    float A, B;
    bool inv, set, row, end;    // row: not a cut (counted); end: the last condition of its rule
    int cls;               // the rule's class (last condition)
};

// The rest of a walk from record c0 (a rule's first) on, for at most 32 unclaimed samples of the tile.
// With P the outcomes of a window's records on a sample, E the ends and S the first records of its
// rules, (P & ~E) + S carries into a rule's end exactly when all records before it hold. A window
// ends with a rule's last record; in a rule of more than 32 records a lane remembers that its sample
// has failed (over). About 12 instructions and 10 shared-memory wavefronts a sample and 80
// instructions a window, against about 500 and 140 for a dense chunk. Returns the lane's hits (UNI);
// otherwise they go to the samples' words. PRED (four samples a lane): `hit` holds the predicted
// classes, a byte a sample, and receives those of the tail through 32 words after the list.
template <int V, bool UNI, bool CAT, bool PRED, bool LIVE = false, class Decode>
__device__ __forceinline__ int tail(uint32_t *list, const uint4 *recs, int rb, int c0, int nrec, int lane, int kmine,
                                    const unsigned char *xs, const int32_t *yl, uint32_t claimed, int deflt,
                                    uint32_t &hit, WalkCount &wc, const Decode &decode)
{
    const uint32_t below = (1u << lane) - 1u;
    uint4 raw = c0 + lane < nrec ? __ldcg(recs + rb + c0 + lane) : make_uint4(0u, 0u, 0u, 0u);
    // list the samples: entry i in lane i, the byte offset 4 n of sample n in a (permuted) row
    int n = 0;
    __syncwarp();
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const bool mine = ((claimed >> (8 * v)) & 0x80u) == 0u;
        const uint32_t b = __ballot_sync(FULL, mine);
        if (mine) list[n + __popc(b & below)] = (uint32_t)(lane * V + v) * 4u;
        n += __popc(b);
    }
    __syncwarp();
    uint32_t at = lane < n ? list[lane] : 0u;
    static_assert(!PRED || V == 4, "a word of four classes per lane");
    if (PRED) {
        list[32 + lane] = hit;
        __syncwarp();
    }
    int hits = 0;
    bool over = false;
    const auto give_back = [&](uint32_t b) {           // the samples of lanes b have hit
        for (; b; b &= b - 1u) {
            const uint32_t a = __shfl_sync(FULL, at, __ffs(b) - 1);
            if (lane == (int)(a / (4u * V))) hit |= 0x80u << (8u * (a / 4u % V));
        }
    };
    while (c0 < nrec && n) {
        const Rec r = decode(raw);
        const uint32_t lo = raw.z, hi = raw.w;
        const uint32_t E = __ballot_sync(FULL, r.end);                        // records from nrec on are 0
        const int cnt = E ? 32 - __clz(E) : 32;
        const uint32_t I = __ballot_sync(FULL, r.inv);
        const uint32_t K = UNI ? __ballot_sync(FULL, r.end && r.cls == kmine) : 0u;
        c0 += cnt;
        wc.records += min(cnt, nrec - c0 + cnt);
        wc.rows += __popc(__ballot_sync(FULL, lane < cnt && r.row));
        wc.ends += __popc(E);
        raw = c0 + lane < nrec ? __ldcg(recs + rb + c0 + lane) : make_uint4(0u, 0u, 0u, 0u);
        uint32_t P = 0;
#pragma unroll 2
        for (int i = 0; i < n; ++i) {
            const uint32_t ai = __shfl_sync(FULL, at, i);
            const float x = *reinterpret_cast<const float *>(xs + (r.xo ^ ai));
            const float z = *reinterpret_cast<const float *>(xs + (r.zo ^ ai));
            bool holds = __fmul_rn(r.A, x) > __fmul_rn(r.B, z);
            if (CAT && r.set) holds = category_member(x, lo, hi);
            const uint32_t v = __ballot_sync(FULL, holds);
            if (lane == i) P = v;
        }
        P ^= I;
        if (over) P &= ~1u;
        const uint32_t fired = lane < n ? ((P & ~E) + (E << 1 | 1u)) & E & P : 0u;
        const uint32_t first = fired & (0u - fired);
        over = !E && (over || P != FULL);
        if (PRED) {
            const int k = __shfl_sync(FULL, r.cls, fired ? __ffs(first) - 1 : 0);
            if (fired) reinterpret_cast<unsigned char *>(list + 32)[at >> 2] = (unsigned char)k;
        } else if (UNI) {
            if (first & K) ++hits;
        } else {
            const int k = __shfl_sync(FULL, r.cls, fired ? __ffs(first) - 1 : 0);
            give_back(__ballot_sync(FULL, fired != 0u && k == load_label<LIVE>(yl - V * lane + (at >> 2))));
        }
        const uint32_t stay = __ballot_sync(FULL, lane < n && fired == 0u);
        if (__popc(stay) != n) {                       // close the list's gaps
            n = __popc(stay);
            if (fired == 0u && (stay >> lane & 1u)) list[__popc(stay & below)] = at;
            __syncwarp();
            at = lane < n ? list[lane] : 0u;
            __syncwarp();
        }
    }
    if (PRED) {
        __syncwarp();
        hit = list[32 + lane];
        __syncwarp();
        return 0;
    }
    if (UNI) return hits + (lane < n && deflt == kmine ? 1 : 0);
    give_back(__ballot_sync(FULL, lane < n && deflt == load_label<LIVE>(yl - V * lane + (at >> 2))));
    return 0;
}

}  // namespace sparse
}  // namespace rs
