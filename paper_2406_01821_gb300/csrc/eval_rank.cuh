// Device code of the rank-coded evaluator (record format v5), shared by the batch evaluator and
// the serving kernel.
//
// A threshold condition has been rewritten exactly as x > c or x < c (pack.cu). Within one
// 128-sample tile, let rank(x) be the position of x in the tile's values (same feature) in
// ascending order, equal values in sample order: #{values below x} + #{equal values before it}.
// Because x is itself one of the tile's values, and a group of equal values is either wholly
// <= c or wholly > c,
//     x >  c  <=>  rank(x) >= L,   L = #{tile values <= c}
//     x <= c  <=>  rank(x) <  L
// (a '<' cut x < c arrives as x <= nextdown(c)). L is counted once per tile and condition, by a
// binary search over the tile's sorted values, when the condition's record is staged. The test
// of a lane's four samples is then one 32-bit subtraction on four rank bytes (0..127), with the
// failure in bit 7 of each byte:
//     '>':  byte (L + 127) - rank          >= 128  <=>  rank <  L   (fails)
//     '<=': byte (255 - L) - (127 - rank)  >= 128  <=>  rank >= L   (fails)
// Each byte difference lies in [0, 255], so no borrow crosses a byte. The second form reads a
// table of reversed ranks (127 - rank), built in shared memory from the first, so that both
// forms are "constant minus table word". A rule's failures are ORed into one word per lane; pair
// and product conditions are compared on the float tile and packed into the same byte layout.
// Claims, per-class hits and the all-claimed exit work on these words (bit 7 of byte v belongs
// to the lane's sample v). A set's records are one flat stream (each rule's conditions, the last
// one flagged) walked 32 records at a time.
#pragma once
#include "eval_sparse.cuh"
#include "rs_internal.cuh"

namespace rs {
namespace rank {

using sparse::WalkCount;
constexpr uint32_t FULL = 0xFFFFFFFFu;
constexpr uint32_t HIGH = 0x80808080u;          // bit 7 of every byte
constexpr uint32_t ONES = 0x01010101u;
constexpr int T = RANK_TILE;                     // samples per tile (= one warp, four per lane)

// #{j : row[j] <= c} over the 128 ascending values of a row in shared memory: each step is a load at a
// fixed offset from a 32-bit address, a compare and a predicated add on the address (the XOR-swizzled
// column it replaced took two operations more a step; ten generations of 10,000 sets 92.0 -> 89.3 ms).
__device__ __forceinline__ int count_below(const float *row, float c)
{
    const uint32_t a0 = (uint32_t)__cvta_generic_to_shared(row);
    uint32_t a = a0;
    float u;
#pragma unroll
    for (uint32_t step = 64; step >= 1; step >>= 1) {
        asm volatile("ld.shared.f32 %0, [%1];" : "=f"(u) : "r"(a + (step - 1) * 4u));
        if (u <= c) a += step * 4u;
    }
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(u) : "r"(a));
    if (u <= c) a += 4u;                         // at most 127 so far: one more for a full count
    return (int)((a - a0) >> 2);
}

// Floats per sorted column: one more than its values, so that searches of different features start
// in different banks.
constexpr int US = T + 1;

// pass rows per warp for pair / product conditions of one chunk
constexpr int VSLOTS = 12, VSLOTS_CAT = 10;
constexpr uint32_t NOOP_K = 127u * ONES;     // constant - rank never has bit 7 set: never fails

// A staged row offset of the float tile (eval_sparse.cuh).
__device__ __forceinline__ uint32_t row_off(uint32_t f) { return sparse::row_off<T * 4>(f); }

// The per-tile tables built in shared memory by the whole block once the tile's features xs
// [F][T] and rank bytes rs [Frows][T] have landed: the reversed ranks (127 - rank) at rs + rev_off,
// each feature's sorted column us[f][pos] = x[f][n] (US floats a row) with pos the rank of x[f][n] (its
// position in the tile's stable ascending order: a permutation, so every slot is written), and the
// float rows permuted in place (row_off). One warp per row.
// With code_of (a row number per feature, CODE_NONE for none): the code rows of features that hold
// category codes only, two words a lane: {nibble v = high three bits of sample v's code, byte v = 1 <<
// its low three bits}.
constexpr uint32_t CODE_NONE = 0xFFu;
__device__ __forceinline__ void build_tile_tables(float *xs, unsigned char *rs, uint32_t rev_off, float *us, int F,
                                                  const unsigned char *code_of = nullptr, uint2 *codes = nullptr)
{
    const int lane = threadIdx.x & 31, warps = blockDim.x >> 5;
    for (int f = threadIdx.x >> 5; f < F; f += warps) {
        float4 *row = reinterpret_cast<float4 *>(xs + f * T);
        const float4 x = row[lane];
        const uint32_t r = reinterpret_cast<const uint32_t *>(rs)[f * 32 + lane];
        reinterpret_cast<uint32_t *>(rs + rev_off)[f * 32 + lane] = r ^ 0x7F7F7F7Fu;
        float *u = us + f * US;
        u[r & 0x7Fu] = x.x;
        u[r >> 8 & 0x7Fu] = x.y;
        u[r >> 16 & 0x7Fu] = x.z;
        u[r >> 24] = x.w;
        if (code_of && code_of[f] != CODE_NONE) {
            const uint32_t c[4] = {(uint32_t)x.x, (uint32_t)x.y, (uint32_t)x.z, (uint32_t)x.w};
            uint2 w = make_uint2(0u, 0u);
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                w.x |= (c[v] >> 3 & 7u) << (4 * v);
                w.y |= (1u << (c[v] & 7u)) << (8 * v);
            }
            codes[code_of[f] * 32 + lane] = w;
        }
        __syncwarp();
        row[lane ^ (f & 7)] = x;
    }
}

// The staged form of a cut for this tile: {rank-table byte offset of the row, per-byte constant}.
__device__ __forceinline__ uint2 stage_cut(uint4 r, const float *us, uint32_t rev_off, int F)
{
    const uint32_t f = min(r.x & R5_F_MASK, (uint32_t)(F - 1));
    const bool le = (r.x >> R5_TAG_SHIFT) == R5_CUT_LT;
    const int L = count_below(us + f * US, __uint_as_float(r.z));
    return make_uint2((le ? rev_off : 0u) + f * T, (uint32_t)(le ? 255 - L : L + 127) * ONES);
}

// The direct walk (finite datasets without rank tables: more than RANK_MAX_F features, or tables that
// do not fit) takes the same records in the same chunks, but tests a cut on the float row: with s =
// +-1 the sign of s x + n is set exactly where the cut fails,
//     '>':  x - c' < 0, c' the float above c        (s = 1,  n = -c')
//     '<=': c - x < 0                               (s = -1, n = c)
// for finite x (a difference of equal floats is +0; n = -0 is made +0), one fused multiply-add a sample,
// and the four signs are gathered into one word. No search, no tables: 12 instructions and a 512-byte
// row read a cut against 7 and a 128-byte one, so the rank-coded walk stays the faster where it fits
// (600 sets on 150,001 samples: 1.34 ms at F = 128, the direct walk 1.59 at F = 233, where the sign-mask
// form takes 1.95). Staged: {row_off of f | le, n}.
__device__ __forceinline__ uint2 stage_cut_direct(uint4 r, int F)
{
    const uint32_t f = min(r.x & R5_F_MASK, (uint32_t)(F - 1));
    const bool le = (r.x >> R5_TAG_SHIFT) == R5_CUT_LT;
    const float c = __uint_as_float(r.z);
    const float n = (le ? c : -nextafterf(c, __uint_as_float(0x7F800000u))) + 0.f;
    return make_uint2(row_off(f) | (le ? 1u : 0u), __float_as_uint(n));
}

__device__ __forceinline__ uint32_t cut_word(uint32_t off, uint32_t n, const unsigned char *xs, uint32_t lane16)
{
    const float4 x = *reinterpret_cast<const float4 *>(xs + ((off & ~15u) ^ lane16));
    const float s = __uint_as_float(0x3F800000u | off << 31), b = __uint_as_float(n);
    const float d0 = __fmaf_rn(s, x.x, b), d1 = __fmaf_rn(s, x.y, b), d2 = __fmaf_rn(s, x.z, b), d3 = __fmaf_rn(s, x.w, b);
    const uint32_t s01 = __byte_perm(__float_as_uint(d0), __float_as_uint(d1), 0x0073);
    const uint32_t s23 = __byte_perm(__float_as_uint(d2), __float_as_uint(d3), 0x0073);
    return __byte_perm(s01, s23, 0x5410);
}

// Bit 7 of byte v where the lane's sample v (labels yl[0..3]) has label k. Only tiles that hold
// more than one label need it, so the labels are read again instead of kept in registers.
// LIVE: see sparse::load_label.
template <bool LIVE = false>
__device__ __forceinline__ uint32_t class_bytes(const int32_t *yl, int k)
{
    const int4 y = sparse::load_label<LIVE>(reinterpret_cast<const int4 *>(yl));
    return ((y.x == k) ? 0x80u : 0u) | ((y.y == k) ? 0x8000u : 0u) | ((y.z == k) ? 0x800000u : 0u) |
           ((y.w == k) ? 0x80000000u : 0u);
}

// Pass row of a pair condition fl(a * x[f]) > fl(b * x[g]) or a product condition
// fl(a * x[f]) > b, staged as {row_off of f, row_off of g (a row of 1.0 for a
// product: fl(b * 1) = b), a, b}: bit 7 of byte v is set exactly where the condition holds for the
// lane's sample v (bits 0..6 carry no meaning; the walk's constant 0xFFFFFFFF minus the word puts
// the failure in bit 7 without a borrow). The products p, q are separately rounded (packed
// two-lane multiplies); p > q is read as the sign of d = fl(fl(q - p) + 0): for p, q finite or
// infinite, fl(q - p) is negative exactly when p > q (gradual underflow keeps the sign of a tiny
// difference; equal values give +0) except q = -0, p = +0, whose -0 the added +0 turns into +0;
// a NaN operand or inf - inf gives the canonical NaN, whose sign bit is clear (false, as the
// IEEE compare). Used on finite datasets only (rank tables), where the products are finite or
// +-inf.
__device__ __forceinline__ uint32_t pass_row(const uint4 *e, const unsigned char *xs, uint32_t lane16)
{
    const uint4 q = *e;
    const float4 x = *reinterpret_cast<const float4 *>(xs + (q.x ^ lane16));
    const float4 z = *reinterpret_cast<const float4 *>(xs + (q.y ^ lane16));
    const float2 a2 = make_float2(__uint_as_float(q.z), __uint_as_float(q.z));
    const float2 b2 = make_float2(__uint_as_float(q.w), __uint_as_float(q.w));
    const float2 m1 = make_float2(-1.f, -1.f), z2 = make_float2(0.f, 0.f);
    const float2 p01 = __fmul2_rn(make_float2(x.x, x.y), a2), p23 = __fmul2_rn(make_float2(x.z, x.w), a2);
    const float2 q01 = __fmul2_rn(make_float2(z.x, z.y), b2), q23 = __fmul2_rn(make_float2(z.z, z.w), b2);
    const float2 d01 = __fadd2_rn(__ffma2_rn(p01, m1, q01), z2);      // fl(q - p) + 0, exactly rounded
    const float2 d23 = __fadd2_rn(__ffma2_rn(p23, m1, q23), z2);
    const uint32_t s01 = __byte_perm(__float_as_uint(d01.x), __float_as_uint(d01.y), 0x0073);
    const uint32_t s23 = __byte_perm(__float_as_uint(d23.x), __float_as_uint(d23.y), 0x0073);
    return __byte_perm(s01, s23, 0x5410);
}

// Pass row of a membership condition, staged as {row_off of f, code row or
// CODE_NONE, set bits 0..31, set
// bits 32..63}: 0xFF in byte v where the lane's sample v holds a category code in the set.
__device__ __forceinline__ uint32_t set_row(uint4 q, const unsigned char *xs, uint32_t lane16)
{
    const float4 x = *reinterpret_cast<const float4 *>(xs + (q.x ^ lane16));
    return (category_member(x.x, q.z, q.w) ? 0x000000FFu : 0u) | (category_member(x.y, q.z, q.w) ? 0x0000FF00u : 0u) |
           (category_member(x.z, q.z, q.w) ? 0x00FF0000u : 0u) | (category_member(x.w, q.z, q.w) ? 0xFF000000u : 0u);
}

// The same from the feature's code row: the set's byte that holds a sample's code is picked by its
// high bits, four samples at once (a byte permute of the set's eight bytes), its bit by its low ones;
// a byte with that bit set carries into bit 7. Three operations where the floats take about forty.
__device__ __forceinline__ uint32_t code_row(uint4 q, const uint2 *codes, int lane)
{
    const uint2 w = codes[q.y * 32u + lane];
    uint32_t m;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(m) : "r"(q.z), "r"(q.w), "r"(w.x));
    return (m & w.y) + 0x7F7F7F7Fu;
}

// One group of four staged records with end-of-rule flags M (bit u: record u ends its rule).
// PRED: the class words are the class in every byte, and hit holds the predicted classes, a byte a sample.
template <uint32_t M, bool UNI, bool PRED, bool LIVE>
__device__ __forceinline__ void group4(const uint32_t (&e)[4], const uint32_t *sw, const int32_t *yl,
                                       uint32_t &fail, uint32_t &claimed, uint32_t &hit)
{
    uint4 w4 = make_uint4(0u, 0u, 0u, 0u);
    if (M) w4 = *reinterpret_cast<const uint4 *>(sw);       // the group's four class words at once
    const uint32_t ws[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        fail |= e[u];
        if (M & (1u << u)) {
            const uint32_t w = ws[u];
            const uint32_t newly = ~fail & HIGH;
            if (PRED) {
                uint32_t m;                                              // bit 7 spread over its byte
                asm("prmt.b32 %0, %1, 0, 0xBA98;" : "=r"(m) : "r"(newly));
                hit = (w & m) | (hit & ~m);
            } else if (UNI) hit |= newly & w;
            else hit |= newly & class_bytes<LIVE>(yl, (int)w);
            claimed |= newly;
            fail = claimed;
        }
    }
}

// Walk the rules of one set (records [rb, rb + nrec)) over the lane's four samples; returns the
// hit bits (bit 7 of byte v: sample v predicted correctly, default included). UNI: the tile holds
// one label (kmine) and end records carry the class mask. CAT: the records may hold membership
// tests (without it, a membership record is never packed: the packer rejects op 2 without sets).
//
// The set is walked in chunks of up to 32 records. Staging turns every record of a chunk into the
// same form {byte offset from the lane's rank word, per-byte constant}: a cut points at its rank
// row; a pair or product condition is first evaluated by the whole warp into a pass row
// (0xFF / 0x00 per sample, constant 0xFFFFFFFF) in the warp's `vrow` slots, from a table of the
// chunk's pairs that the lanes build in parallel; padding records are no-ops. The chunk is then one
// straight run of identical steps, with the first-fire claim applied after each rule's last record
// (a warp vote gives their positions); the all-claimed exit is tested once per chunk.
// PRED: instead of hits, the predicted class of each of the lane's samples, a byte each (classes below
// 256), the default where no rule fires.
// A record of format v5 on the sparse tail: fl(A x) > fl(B z), z = 1 but for pairs; a '<=' cut is the
// negation of x > c.
struct Decode5 {
    int F;
    uint32_t ones_off;
    __device__ __forceinline__ sparse::Rec operator()(const uint4 raw) const
    {
        const uint32_t tag = raw.x >> R5_TAG_SHIFT;
        const bool cut = tag == R5_CUT_GT || tag == R5_CUT_LT, none = tag == R5_NONE;
        sparse::Rec r;
        r.xo = row_off(min(raw.x & R5_F_MASK, (uint32_t)(F - 1)));
        r.zo = tag == R5_PAIR ? row_off(min(raw.y, (uint32_t)(F - 1))) : ones_off;
        r.A = cut ? 1.f : (none ? 0.f : __uint_as_float(raw.z));
        r.B = cut ? __uint_as_float(raw.z) : (none ? -1.f : __uint_as_float(raw.w));
        r.inv = tag == R5_CUT_LT;
        r.set = tag == R5_SET;
        r.row = tag >= R5_PAIR;
        r.end = (raw.x & R5_END_BIT) != 0u;
        r.cls = (int)((raw.x >> R5_CLS_SHIFT) & 0xFFFu);
        return r;
    }
};

// Returns the hit bits; `more` receives the lane's hits of the sparse tail that are not in them.
// DIRECT: the direct walk (us, rl and rev_off unused, vrow_off relative to xs).
template <bool UNI, int VS, bool CAT, bool PRED = false, bool DIRECT = false, bool LIVE = false>
__device__ __forceinline__ uint32_t walk_set(uint4 *st, uint32_t *vrow, uint32_t vrow_off, int lane,
                                             const uint4 *recs, int rb, int nrec, const float *us,
                                             uint32_t rev_off, int F, int kmine, const unsigned char *rl,
                                             const unsigned char *xs, uint32_t ones_off, const int32_t *yl,
                                             uint32_t claimed, int deflt, WalkCount &wc, int &more,
                                             const unsigned char *code_of = nullptr, const uint2 *codes = nullptr)
{
    static_assert(VS <= 16, "pair table and staged records share the warp's 512-byte stage");
    const uint4 zero4 = make_uint4(0u, 0u, 0u, 0u);
    const uint32_t lane16 = (uint32_t)lane << 4;
    uint2 *s8 = reinterpret_cast<uint2 *>(st);            // staged {offset, constant}, 32 entries
    uint32_t *sw = reinterpret_cast<uint32_t *>(st) + 64;  // end-of-rule class mask / class
    uint4 pf = lane < nrec ? __ldcg(recs + rb + lane) : zero4;
    uint32_t hit = PRED ? (uint32_t)deflt * ONES : 0u, fail = claimed;
    more = 0;
    int c0 = 0;
    while (c0 < nrec) {
        const uint4 raw = pf;
        const uint32_t tag = raw.x >> R5_TAG_SHIFT;
        int cnt = min(32, nrec - c0);
        uint32_t pm = __ballot_sync(FULL, lane < cnt && (tag == R5_PAIR || tag == R5_GEN));
        uint32_t sm = CAT ? __ballot_sync(FULL, lane < cnt && tag == R5_SET) : 0u;   // membership tests
        if (__popc(pm | sm) > VS) {         // end the chunk before the pass row that finds no slot
            uint32_t m = pm | sm;
            for (int k = 0; k < VS; ++k) m &= m - 1u;
            cnt = __ffs(m) - 1;
            pm &= (1u << cnt) - 1u;
            sm &= (1u << cnt) - 1u;
        }
        const uint32_t ends = __ballot_sync(FULL, lane < cnt && (raw.x & R5_END_BIT) != 0u);
        pf = (c0 + cnt + lane < nrec) ? __ldcg(recs + rb + c0 + cnt + lane) : zero4;

        __syncwarp();                       // the previous chunk's readers of the stage are done
        // every lane runs the cut search (branch-free staging); other records then take their form.
        // A pair or product condition gets a pass-row slot and a pair-table entry.
        const uint32_t cls = (raw.x >> R5_CLS_SHIFT) & 0xFFFu;
        const uint32_t ew = PRED ? cls * ONES : (UNI ? ((int)cls == kmine ? 0xFFFFFFFFu : 0u) : cls);
        uint2 sr = DIRECT ? stage_cut_direct(raw, F) : stage_cut(raw, us, rev_off, F);
        const int np = __popc(pm);
        if ((pm >> lane) & 1u) {
            const uint32_t slot = __popc(pm & ((1u << lane) - 1u));
            const uint32_t f = min(raw.x & R5_F_MASK, (uint32_t)(F - 1));
            const uint32_t g = min(raw.y, (uint32_t)(F - 1));
            st[slot] = make_uint4(row_off(f), tag == R5_PAIR ? row_off(g) : ones_off, raw.z, raw.w);
            sr = make_uint2(vrow_off + 128u * slot, FULL);
        } else if (CAT && ((sm >> lane) & 1u)) {
            const uint32_t slot = np + __popc(sm & ((1u << lane) - 1u));
            const uint32_t f = min(raw.x & R5_F_MASK, (uint32_t)(F - 1));
            st[slot] = make_uint4(row_off(f), code_of ? code_of[f] : CODE_NONE, raw.z, raw.w);
            sr = make_uint2(vrow_off + 128u * slot, FULL);
        } else if (lane >= cnt || tag == R5_NONE) {
            sr = DIRECT ? make_uint2(0u, 0x7F800000u) : make_uint2(0u, NOOP_K);     // +inf: never fails
        }
        __syncwarp();
        {                                             // pass rows, one warp-wide evaluation each
            uint32_t *vr = vrow + lane;
            for (int j = 0; j < np; j += 2) {
                const uint32_t v0 = pass_row(st + j, xs, lane16);
                if (j + 1 < np) vr[32] = pass_row(st + j + 1, xs, lane16);
                vr[0] = v0;
                vr += 64;
            }
            if (CAT)
                for (int j = np; j < np + __popc(sm); ++j) {
                    const uint4 q = st[j];
                    vrow[j * 32 + lane] = q.y != CODE_NONE ? code_row(q, codes, lane) : set_row(q, xs, lane16);
                }
        }
        __syncwarp();
        s8[lane] = sr;
        sw[lane] = ew;
        __syncwarp();

        for (int g = 0; g < cnt; g += 4) {
            const uint4 ra = *reinterpret_cast<const uint4 *>(s8 + g);
            const uint4 rc = *reinterpret_cast<const uint4 *>(s8 + g + 2);
            uint32_t e[4];
            if (DIRECT) {
                const uint32_t rows = (pm | sm) >> g;
                const uint32_t off[4] = {ra.x, ra.z, rc.x, rc.z}, val[4] = {ra.y, ra.w, rc.y, rc.w};
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    if (rows & (1u << u)) e[u] = ~*reinterpret_cast<const uint32_t *>(xs + off[u] + 4 * lane);
                    else e[u] = cut_word(off[u], val[u], xs, lane16);
                }
            } else {
                e[0] = ra.y - *reinterpret_cast<const uint32_t *>(rl + ra.x);
                e[1] = ra.w - *reinterpret_cast<const uint32_t *>(rl + ra.z);
                e[2] = rc.y - *reinterpret_cast<const uint32_t *>(rl + rc.x);
                e[3] = rc.w - *reinterpret_cast<const uint32_t *>(rl + rc.z);
            }
            const uint32_t *swg = sw + g;
            switch ((ends >> g) & 0xFu) {
#define RS_GROUP4(M) case M: group4<M, UNI, PRED, LIVE>(e, swg, yl, fail, claimed, hit); break;
            RS_GROUP4(0) RS_GROUP4(1) RS_GROUP4(2) RS_GROUP4(3) RS_GROUP4(4) RS_GROUP4(5) RS_GROUP4(6)
            RS_GROUP4(7) RS_GROUP4(8) RS_GROUP4(9) RS_GROUP4(10) RS_GROUP4(11) RS_GROUP4(12)
            RS_GROUP4(13) RS_GROUP4(14) RS_GROUP4(15)
#undef RS_GROUP4
            }
        }
        c0 += cnt;
        wc.rows += __popc(pm | sm);
        wc.ends += __popc(ends);
        if (c0 >= nrec) break;
        const int live = __reduce_add_sync(FULL, __popc(~claimed & HIGH));    // 0: the set is decided
        if (!live) break;
        if (live <= sparse::MAX && ends) {                   // from the first rule not finished yet
            const int tail = cnt - (32 - __clz(ends));
            wc.records += c0 - tail;
            more = sparse::tail<4, UNI, CAT, PRED, LIVE>(sw, recs, rb, c0 - tail, nrec, lane, kmine, xs, yl, claimed, deflt, hit, wc,
                                             Decode5{F, ones_off});
            return hit;
        }
    }
    wc.records += c0;
    if (PRED) return hit;
    const uint32_t left = ~claimed & HIGH;
    if (UNI) hit |= (deflt == kmine) ? left : 0u;
    else hit |= left & class_bytes<LIVE>(yl, deflt);
    return hit;
}

}  // namespace rank
}  // namespace rs
