// The soft path: sigmoid-relaxed first-fire evaluation (forward) and its hand-written adjoint.
//
// Per condition  u = s*(a*x[f] - rhs)/tau  (s = +1 for '>', -1 for '<'; rhs = t or b*x[g]).
// Per rule       lq_r = sum_c log sigmoid(u_c)      (log of the firing probability q_r)
//                l1q_r = log(1 - q_r) = log(-expm1(lq_r))
//                lu_r = sum_{j<r} l1q_j             (log probability that no earlier rule fired)
// Class k        log p_k = logsumexp over rules of class k of (lq_r + lu_r), plus lu_R for the
//                default class.  Loss  L_p = (1/N) sum_n -log p_{y_n}.
// Adjoint        S_r = P(outcome y | evaluation starts at rule r), T_r = 1 - S_r, both kept as logs
//                and both sums of positive terms:
//                  lS_R = 0 if default = y else -inf;  lS_r = logsumexp([cls_r = y] lq_r, l1q_r + lS_{r+1})
//                  lT_R = 0 if default != y else -inf; lT_r = logsumexp([cls_r != y] lq_r, l1q_r + lT_{r+1})
//                dl/dlq_r = exp(lq_r + lu_r - lp) * (S_{r+1} - [cls_r = y])
//                         =  exp(lq_r + lu_r + lS_{r+1} - lp)   if cls_r != y
//                         = -exp(lq_r + lu_r + lT_{r+1} - lp)   if cls_r  = y
//                (the second form avoids the cancellation of S_{r+1} - 1 when S_{r+1} is near 1)
//                dl/du_c  = dl/dlq_r * sigmoid(-u_c);  du/da = s x_f / tau, du/dt = -s / tau,
//                du/db = -s x_g / tau.
// These are the formulas in logs; the float kernels evaluate them as products and sums of positive
// numbers in the linear domain (see "the float path" below), whose relative errors do not grow with the
// margins, and a group of samples in which some sample's p_y is below e^-32 (or is not a number) is
// evaluated again in float-float logs (about 48 significant bits), with the margins formed exactly,
// 1 - q_r taken as a log-sum-exp of -u_c when q_r rounds to 1, and each d ell / d u_c formed in the
// exponent (soft_group_ff): there the exponentials of margins of that size carry the margins' rounding
// (2^-24 of 32 and more), and a probability comes near float32's range.
//
// Work: one warp owns a (rule set, sample chunk) pair and walks the chunk in groups of 64 or 128
// samples (two or four neighbouring ones per lane), so each partial sum has a fixed summation order.
// The forward keeps U_r per rule and sample; the adjoint computes q_r again from the conditions.
// Chunks are a function of the call's shape only; partial losses and gradients per chunk are reduced
// in a second kernel in a fixed order, which makes results bit-reproducible run to run and
// independent of scheduling.
#include "rs_internal.cuh"
#include "soft_step.cuh"
#include "block_scan.cuh"

namespace rs {

namespace {

constexpr uint32_t FULL = 0xFFFFFFFFu;
constexpr int SOFT_W = 4;                 // warps per CTA of the per-warp kernel
constexpr int FF_W = 16, FF_W_PROBS = 8;  // and of the float-float pass, without and with class probabilities
constexpr int SOFT_MAX_RULES = 64;        // rules per set held in shared memory
constexpr int SOFT_MAX_CONDS = 512;       // conditions per set accumulated in shared memory
constexpr int SOFT_MAX_CHUNKS = 128;
constexpr int SOFT_G = 64;                // chunks are whole multiples of it
constexpr int SOFT_FF_GROUP = 64;         // samples that go to the float-float pass together
// the call's counters: tasks taken, [1..2] most rules / conditions of a set, length of the
// float-float list, list items taken
constexpr int SOFT_NEXT_FF_LEN = 3, SOFT_NEXT_FF = 4, SOFT_NEXT_N = 8;

// Floats of a float-float warp's shared arrays: acc [maxC][4], and lu [maxR + 1][32] and lq [maxR][32]
// when the class probabilities are written.
__host__ __device__ constexpr size_t soft_ff_floats(int maxR, int maxC, bool probs)
{
    return (size_t)maxC * 4 + (probs ? (size_t)(2 * maxR + 1) * 32 : 0);
}

// Largest sets the entry points take: four times these floats fit an SM's shared memory (the size of an
// earlier layout of the per-warp arrays, kept as the limit; the present ones are smaller).
__host__ constexpr size_t soft_limit_floats(int maxR, int maxC, bool probs)
{
    return (size_t)(maxR + 1) * SOFT_G + (size_t)maxC * 4 + (probs ? (size_t)maxR * SOFT_G : 0);
}

struct __align__(16) SoftRec {
    uint32_t meta;    // bit 0: pair condition, bit 1: '<', bit 2: category membership
    uint16_t f, g;
    float a, bt;      // bt = threshold t, or the pair coefficient b; a membership test holds the
                      // bits of its category set (0..31 in a, 32..63 in bt)
};

// Single-CTA counting sort of the sets by size (rules + conditions, most first), so that the
// warps of one CTA group walk sets of similar length. Malformed offsets count as size 0 (the
// check kernel rejects the batch).
constexpr int SOFT_ORDER_BUCKETS = 1024;
__global__ void k_soft_order(BatchDev b, int32_t *order)
{
    __shared__ int hist[SOFT_ORDER_BUCKETS];
    const int R = b.dR ? *b.dR : b.R, C = b.dC ? *b.dC : b.C;
    for (int i = threadIdx.x; i < SOFT_ORDER_BUCKETS; i += blockDim.x) hist[i] = 0;
    __syncthreads();
    auto bucket = [&](int p) {
        const int rb = b.set_rule_off[p], re = b.set_rule_off[p + 1];
        int cost = 0;
        if (rb >= 0 && re >= rb && re <= R) {
            const int cb = b.rule_cond_off[rb], ce = b.rule_cond_off[re];
            if (cb >= 0 && ce >= cb && ce <= C) cost = (re - rb) + (ce - cb);
        }
        return SOFT_ORDER_BUCKETS - 1 - min(cost, SOFT_ORDER_BUCKETS - 1);
    };
    for (int p = threadIdx.x; p < b.P; p += blockDim.x) atomicAdd(&hist[bucket(p)], 1);
    __syncthreads();
    block_exclusive_scan_array(hist, SOFT_ORDER_BUCKETS);
    for (int p = threadIdx.x; p < b.P; p += blockDim.x) order[atomicAdd(&hist[bucket(p)], 1)] = p;
}

// Validation of set p's structure by one warp, a rule a lane.
__device__ void check_set_soft(const BatchDev &b, int p, int lane, int K, uint32_t *status, int32_t *maxima, int maxR,
                               int maxC)
{
    const int rb = b.set_rule_off[p], re = b.set_rule_off[p + 1];
    const int d = b.set_default[p];
    if (lane == 0 && (d < 0 || d >= K)) atomicOr(status, ST_BAD_CLASS);
    if (rb < 0 || re < rb || re > b.R) { if (lane == 0) atomicOr(status, ST_BAD_OFFSETS); return; }
    if (re - rb > SOFT_MAX_RULES) { if (lane == 0) atomicOr(status, ST_TOO_LARGE); return; }
    bool bad = false;
    for (int r = rb + lane; r < re; r += 32) {
        const int c0 = b.rule_cond_off[r], c1 = b.rule_cond_off[r + 1];
        bad |= c0 < 0 || c1 < c0 || c1 > b.C;
        const int cls = b.rule_class[r];
        if (cls < 0 || cls >= K) atomicOr(status, ST_BAD_CLASS);
    }
    if (__any_sync(FULL, bad)) { if (lane == 0) atomicOr(status, ST_BAD_OFFSETS); return; }
    if (lane != 0) return;
    const int nc = re > rb ? b.rule_cond_off[re] - b.rule_cond_off[rb] : 0;
    if (nc > SOFT_MAX_CONDS || re - rb > maxR || nc > maxC) atomicOr(status, ST_TOO_LARGE);
    atomicMax(&maxima[0], re - rb);
    atomicMax(&maxima[1], nc);
}

// The record of condition c.
__device__ void pack_soft_one(const BatchDev &b, int c, int F, SoftRec *recs, uint32_t *status)
{
    const int f = b.cond_f[c], g = b.cond_g[c], op = b.cond_op[c];
    SoftRec r{0, 0, 0, 0.f, 0.f};
    if (f < 0 || f >= F || g < -1 || g >= F) atomicOr(status, ST_BAD_FEATURE);
    else if (op == RS_OP_IN && b.cond_set && g == -1) {
        const uint64_t set = b.cond_set[c];
        r.meta = 4u;
        r.f = (uint16_t)f;
        r.a = __uint_as_float((uint32_t)set);
        r.bt = __uint_as_float((uint32_t)(set >> 32));
    } else if (op != 0 && op != 1) atomicOr(status, ST_BAD_OP);
    else {
        r.meta = (g >= 0 ? 1u : 0u) | (op == 1 ? 2u : 0u);
        r.f = (uint16_t)f;
        r.g = (uint16_t)(g >= 0 ? g : 0);
        r.a = b.cond_a[c];
        r.bt = g >= 0 ? b.cond_b[c] : b.cond_t[c];
    }
    recs[c] = r;
}

// One launch: blocks [0, set_blocks) validate the sets, a warp each; the others pack the conditions
// and reset the call's counters. (A thread per set walking its rules took 12 us in a launch of its own.)
constexpr int SOFT_PREP_BLOCK = 256;
__global__ void k_soft_prep(BatchDev b, int F, int K, SoftRec *recs, uint32_t *status, int32_t *counters,
                            int32_t *maxima, int maxR, int maxC, int set_blocks)
{
    if (b.dR) { b.R = *b.dR; b.C = *b.dC; }
    if ((int)blockIdx.x < set_blocks) {
        const int p = (int)((blockIdx.x * SOFT_PREP_BLOCK + threadIdx.x) >> 5);
        if (blockIdx.x == 0 && threadIdx.x == 0 &&
            (b.set_rule_off[0] != 0 || b.set_rule_off[b.P] != b.R || b.rule_cond_off[0] != 0 ||
             b.rule_cond_off[b.R] != b.C))
            atomicOr(status, ST_BAD_OFFSETS);
        if (p < b.P) check_set_soft(b, p, threadIdx.x & 31, K, status, maxima, maxR, maxC);
        return;
    }
    const int64_t c = (int64_t)(blockIdx.x - set_blocks) * SOFT_PREP_BLOCK + threadIdx.x;
    if (c == 0) counters[0] = counters[SOFT_NEXT_FF_LEN] = counters[SOFT_NEXT_FF] = 0;
    if (recs && c < b.C) pack_soft_one(b, (int)c, F, recs, status);
}

static int soft_set_blocks(int P) { return (int)(((int64_t)P * 32 + SOFT_PREP_BLOCK - 1) / SOFT_PREP_BLOCK); }

// log(1 + e) for 0 <= e <= 1 as e p(e), with p the polynomial of degree 8 of least maximum
// relative error against log1p(e) / e on [0, 1] (Remez exchange, 3.0e-8 before its coefficients
// were rounded to float32), evaluated by Horner's rule in fused multiply-adds: within 2 ulp of
// log1p over the interval, and e p(e) keeps the relative accuracy of log1p(e) = e (1 - e/2 + ...)
// as e goes to 0. No division and no special case.
__device__ __forceinline__ float log1p_unit(float e)
{
    float p = 5.232694093e-03f;
    p = fmaf(p, e, -2.950523794e-02f);
    p = fmaf(p, e, 7.822595537e-02f);
    p = fmaf(p, e, -1.366324574e-01f);
    p = fmaf(p, e, 1.910600662e-01f);
    p = fmaf(p, e, -2.484298199e-01f);
    p = fmaf(p, e, 3.331909776e-01f);
    p = fmaf(p, e, -4.999949336e-01f);
    p = fmaf(p, e, 9.999999404e-01f);
    return e * p;
}

// The hardware exponential (ex2.approx of x log2(e)) of a non-positive argument: for |x| up to about
// 100 its relative error stays below a few 1e-6. Used by the class probabilities of the float-float
// pass and by log1m_exp.
__device__ __forceinline__ float exp_np(float x) { return __expf(x); }

// log(1 - e^s) for s <= 0: the log-probability that a rule whose conditions hold with
// probability q = e^s does not fire. For the entry point rs_selftest_log1m_exp only: the float path works
// in the linear domain, the float-float pass has rule_log1mq_ff. Both pieces are evaluated and one is
// selected:
// * q <= e^(-1/2): log1p(-q) = -q a(q), a the degree-10 polynomial of least maximum relative
//   error against -log1p(-q) / q on [0, e^(-1/2)] (Remez exchange; within 2 ulp given q). q comes
//   from the hardware exponential, whose relative error (a few 1e-6 at most for the arguments
//   that matter) becomes that of the result: an absolute error below 1e-7 in the log domain.
// * t = -s < 1/2: log t + t b(t), b the degree-3 polynomial of least maximum relative error
//   against log((1 - e^-t) / t) / t on [0, 1/2]; log t = k ln 2 + log m for t = m 2^k, 1 <= m < 2,
//   with log m from the hardware logarithm, whose error on [1, 2] is at most 2^-21.41 absolute,
//   whatever k: as t goes to 0 the absolute error stays at that level instead of growing with
//   |log t| (lu, a sum of these terms, is an absolute quantity in the log domain).
// s = 0 gives -inf (the rule fires for certain), s = -inf gives -0.
__device__ __forceinline__ float log1m_exp(float s)
{
    const float t = -s;
    const float q = exp_np(s);
    float pa = 5.805101871e+00f;
    pa = fmaf(pa, q, -1.336368465e+01f);
    pa = fmaf(pa, q, 1.424522972e+01f);
    pa = fmaf(pa, q, -8.279889107e+00f);
    pa = fmaf(pa, q, 3.204409838e+00f);
    pa = fmaf(pa, q, -5.293834209e-01f);
    pa = fmaf(pa, q, 2.968223989e-01f);
    pa = fmaf(pa, q, 2.422454804e-01f);
    pa = fmaf(pa, q, 3.336488008e-01f);
    pa = fmaf(pa, q, 4.999950230e-01f);
    pa = fmaf(pa, q, 1.000000000e+00f);
    const float ra = -q * pa;
    float pb = -3.432709782e-04f;
    pb = fmaf(pb, t, -1.679248726e-06f);
    pb = fmaf(pb, t, 4.166686162e-02f);
    pb = fmaf(pb, t, -5.000000000e-01f);
    const bool sub = t < 0x1p-126f;                  // subnormal t: scaled by 2^24 first
    const int it = __float_as_int(sub ? t * 0x1p24f : t);
    const float k = (float)((it >> 23) - (sub ? 127 + 24 : 127));
    const float m = __int_as_float((it & 0x007FFFFF) | 0x3F800000);
    const float lt = fmaf(k, 6.931471825e-01f, fmaf(k, -1.904654212e-09f, __logf(m)));   // ln 2 as hi + lo
    const float rb = t == 0.f ? -INFINITY : fmaf(t, pb, lt);
    return t >= 0.5f ? ra : rb;
}

// Elementary functions evaluated on the device (test hooks): 0 = log1p_unit, 1 = log1m_exp.
__global__ void k_selftest_soft_math(const float *in, int n, float *out, int which)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        out[i] = which == 0 ? log1p_unit(in[i]) : log1m_exp(in[i]);
}

__device__ __forceinline__ float log_add(float a, float b)
{
    if (a == -INFINITY) return b;
    if (b == -INFINITY) return a;
    const float m = fmaxf(a, b);
    return m + log1p_unit(exp_np(-fabsf(a - b)));
}

// Kahan-compensated accumulation.
__device__ __forceinline__ void kadd(float &s, float &c, float v)
{
    const float y = v - c;
    const float t = s + y;
    c = (t - s) - y;
    s = t;
}

// The same for the loss, whose terms may be +inf (a label no path reaches): an infinite sum stays
// infinite rather than turning NaN.
__device__ __forceinline__ void kadd_loss(float &s, float &c, float v)
{
    const float y = v - c;
    const float t = s + y;
    c = isinf(t) ? 0.f : (t - s) - y;
    s = t;
}

struct SoftKArgs {
    const SoftRec *recs;
    const int32_t *set_rule_off, *rule_cond_off, *rule_class, *set_default;
    int32_t P;
    const float *Xt;
    const int32_t *y;
    const int32_t *perm;
    int64_t N, n_pad;
    int32_t K;
    float inv_tau;
    float inv_tau_lo;                // 1/tau - inv_tau (float-float path)
    int32_t nchunks, chunk;          // chunk = samples per chunk (multiple of 32)
    float *part_loss;                // [nchunks][P]
    float *part_ga, *part_gbt;       // [nchunks][C]
    float *probs;                    // [P*N*K] or null
    int32_t *next;                   // [8] counters (SOFT_NEXT_*)
    int32_t maxR, maxC;              // shared-memory capacity per warp (rules, conditions)
    int64_t Ccap;                    // row stride of the gradient partials
    const uint32_t *status;          // no work if non-zero (malformed batch)
    const int32_t *order;            // sets by decreasing size (schedule only; results do not depend on it)
    int32_t *fflist;                 // [nchunks * P]: tasks (ch * P + p) with groups left to the float-float pass
    uint32_t *ffbits;                // [nchunks][P][ff_wpt]: bit g of a task: its g-th SOFT_FF_GROUP samples are among them
    int32_t ff_wpt;                  // words per task (SOFT_FF_GROUPs per chunk / 32, rounded up)
    int32_t pslots;                  // class-probability slots per warp (0: not written)
    int32_t teams;                   // teams per CTA (staged-tile kernel)
    uint32_t tm_cols;                // tensor-memory columns of a CTA (staged-tile adjoint)
};

// Feature access of the float-float pass: the lane's sample column in global memory, x[f] at col[f * stride].
struct XView {
    const float *col;
    int64_t stride;
    // x[f] of the lane's sample
    __device__ __forceinline__ float operator()(int f) const { return col[(int64_t)f * stride]; }
};

// ------------------------------------------------------------------ float-float arithmetic
// A value held as the unevaluated sum hi + lo of two floats (Dekker, "A floating-point technique
// for extending the available precision", 1971; Knuth's TwoSum): about 48 significant bits. The
// transformations below are written with explicitly rounded operations so that no contraction
// or reassociation can change them. Non-finite values carry lo = 0 and bypass the
// transformations (which would turn an infinity into NaN).
struct ff {
    float hi, lo;
};

__device__ __forceinline__ ff ff_two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}

__device__ __forceinline__ ff ff_fast_sum(float a, float b)     // |a| >= |b| or a == 0
{
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}

__device__ __forceinline__ float ff_f(ff x) { return __fadd_rn(x.hi, x.lo); }
__device__ __forceinline__ ff ff_neg(ff x) { return {-x.hi, -x.lo}; }

__device__ __forceinline__ ff ff_add(ff x, ff y)
{
    if (!isfinite(x.hi) || !isfinite(y.hi)) return {__fadd_rn(x.hi, y.hi), 0.f};
    const ff s = ff_two_sum(x.hi, y.hi);
    return ff_fast_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(x.lo, y.lo)));
}

__device__ __forceinline__ ff ff_add_f(ff x, float y) { return ff_add(x, ff{y, 0.f}); }

__device__ __forceinline__ ff ff_two_prod(float a, float b)
{
    const float p = __fmul_rn(a, b);
    if (!isfinite(p)) return {p, 0.f};
    return {p, __fmaf_rn(a, b, -p)};
}

__device__ __forceinline__ ff ff_mul(ff x, ff y)
{
    const float p = __fmul_rn(x.hi, y.hi);
    if (!isfinite(p)) return {p, 0.f};
    float e = __fmaf_rn(x.hi, y.hi, -p);
    e = __fadd_rn(e, __fadd_rn(__fmul_rn(x.hi, y.lo), __fmul_rn(x.lo, y.hi)));
    return ff_fast_sum(p, e);
}

__device__ __forceinline__ bool ff_less(ff x, ff y) { return x.hi < y.hi || (x.hi == y.hi && x.lo < y.lo); }

// log(e^a + e^b): the larger term plus log1p of the exponential of the (float) difference
__device__ __forceinline__ ff ff_log_add(ff a, ff b)
{
    if (a.hi == -INFINITY) return b;
    if (b.hi == -INFINITY) return a;
    const bool ab = ff_less(b, a);
    const ff m = ab ? a : b, o = ab ? b : a;
    return ff_add_f(m, log1p_unit(expf(ff_f(ff_add(o, ff_neg(m))))));
}

// log y for 0 < y <= 1 in float-float: y = m 2^k with m in [sqrt(1/2), sqrt(2)), log y = k ln 2 +
// log m; ln 2 split into a head of 15 significant bits (k * head is exact for |k| < 512) and a tail.
__device__ __forceinline__ ff ff_log_unit(float y)
{
    int k;
    float m = frexpf(y, &k);
    if (m < 0.70710678f) { m = __fmul_rn(m, 2.f); --k; }
    constexpr float LN2_HI = 0.693145751953125f, LN2_LO = 1.42860682030941723e-6f;
    const ff kl = ff_fast_sum(__fmul_rn((float)k, LN2_HI), __fmul_rn((float)k, LN2_LO));
    return ff_add_f(kl, logf(m));
}

// A condition's record with the lane's feature values (xg: the second feature of a pair).
struct CondIn {
    SoftRec rc;
    float xf, xg;
};

__device__ __forceinline__ CondIn load_cond(const SoftKArgs &a, int c, const XView &x)
{
    CondIn t;
    t.rc = a.recs[c];
    t.xf = x(t.rc.f);
    t.xg = x((t.rc.meta & 1u) ? t.rc.g : t.rc.f);
    return t;
}

// The signed scaled margin u = s * (a * x[f] - rhs) / tau of a condition for the lane's sample, in
// float-float: the products are exact (a float times a float), 1/tau is a float-float.
__device__ __forceinline__ ff margin_ff(const SoftKArgs &a, const CondIn &t)
{
    const ff lhs = ff_two_prod(t.rc.a, t.xf);
    const ff rhs = (t.rc.meta & 1u) ? ff_two_prod(t.rc.bt, t.xg) : ff{t.rc.bt, 0.f};
    ff u = ff_mul(ff_add(lhs, ff_neg(rhs)), ff{a.inv_tau, a.inv_tau_lo});
    if (t.rc.meta & 2u) u = ff_neg(u);
    return u;
}

// log sigmoid(u) = min(u, 0) - log1p(e^-|u|); l1pe returns log1p(e^-|u|), which log sigmoid(-u) =
// -max(u, 0) - log1p(e^-|u|) shares.
__device__ __forceinline__ ff log_sigmoid_ff(ff u, float &l1pe)
{
    l1pe = log1p_unit(expf(-fabsf(ff_f(u))));
    return u.hi < 0.f ? ff_add_f(u, -l1pe) : ff{-l1pe, 0.f};
}

// log q of one rule for the lane's sample in float-float (membership tests: 0 or -inf).
template <bool CAT>
__device__ ff rule_logq_ff(const SoftKArgs &a, int c0, int c1, const XView &x)
{
    ff s{0.f, 0.f};
    for (int c = c0; c < c1; ++c) {
        const CondIn t = load_cond(a, c, x);
        if (CAT && (t.rc.meta & 4u)) {
            if (!category_member(t.xf, __float_as_uint(t.rc.a), __float_as_uint(t.rc.bt))) s = ff_add(s, ff{-INFINITY, 0.f});
            continue;
        }
        float l1pe;
        s = ff_add(s, log_sigmoid_ff(margin_ff(a, t), l1pe));
    }
    return s;
}

// log(1 - q) of one rule from its log q (float-float). Where q <= 1/2 the float value is exact to
// its last bit's scale; below that, 1 - q = -expm1(log q) and its log is taken in float-float;
// where log q is within 2^-24 of 0, every condition's margin exceeds ~16.6 tau and
// 1 - q = sum_c softplus(-u_c) = sum_c e^{-u_c} to float precision, whose log is the
// log-sum-exp of -u_c with the largest term factored out. A rule of holding membership tests
// only has q = 1 exactly and log(1 - q) = -inf.
template <bool CAT>
__device__ ff rule_log1mq_ff(const SoftKArgs &a, int c0, int c1, const XView &x, ff lq)
{
    if (lq.hi == -INFINITY) return {0.f, 0.f};
    const float lqf = ff_f(lq);
    if (isnan(lqf)) return {lqf, 0.f};
    if (lqf < -0.69314718f) return {log1pf(-expf(lqf)), 0.f};
    if (lqf < -0x1p-24f) return ff_log_unit(-expm1f(lqf));
    ff m{INFINITY, 0.f};
    for (int c = c0; c < c1; ++c) {
        const CondIn t = load_cond(a, c, x);
        if (CAT && (t.rc.meta & 4u)) continue;
        const ff u = margin_ff(a, t);
        if (ff_less(u, m)) m = u;
    }
    if (m.hi == INFINITY) return {-INFINITY, 0.f};
    float acc = 0.f;
    for (int c = c0; c < c1; ++c) {
        const CondIn t = load_cond(a, c, x);
        if (CAT && (t.rc.meta & 4u)) continue;
        acc += expf(ff_f(ff_add(m, ff_neg(margin_ff(a, t)))));
    }
    return ff_add_f(ff_neg(m), logf(acc));
}

// The four gradient sums of conditions c and c + 1 (g0, g1: this lane's d/da, d/db-or-dt) reduced
// over the warp in one butterfly and added to the warp's accumulators.
__device__ __forceinline__ void reduce_pair(float2 g0, float2 g1, int ci0, bool has1, float (*acc)[4], int lane)
{
    const bool b4 = lane & 16, b3 = lane & 8;
    // lanes 0..15 gather the first condition's two sums, lanes 16..31 the second's
    float k0 = b4 ? g1.x : g0.x, k1 = b4 ? g1.y : g0.y;
    k0 += __shfl_xor_sync(FULL, b4 ? g0.x : g1.x, 16);
    k1 += __shfl_xor_sync(FULL, b4 ? g0.y : g1.y, 16);
    // then lanes with bit 3 clear the d/da sum, set the other
    float t = (b3 ? k1 : k0) + __shfl_xor_sync(FULL, b3 ? k0 : k1, 8);
    t += __shfl_xor_sync(FULL, t, 4);
    t += __shfl_xor_sync(FULL, t, 2);
    t += __shfl_xor_sync(FULL, t, 1);
    // lanes 0, 8, 16, 24 hold the totals; each condition's sums always land in the same lanes
    if ((lane & 7) == 0 && (!b4 || has1)) {
        const int ci = ci0 + (b4 ? 1 : 0), k = b3 ? 2 : 0;
        kadd(acc[ci][k], acc[ci][k + 1], t);
    }
}

// Class probabilities of the lane's sample n from its per-rule log q and log "no earlier rule fired"
// (lq, lu; lu[R] for the default).
__device__ __forceinline__ void write_probs(const SoftKArgs &a, int p, int rb, int R, int deflt, int64_t n, int lane,
                                            float (*lq)[32], float (*lu)[32])
{
    const int64_t orig = a.perm[n];
    for (int k = 0; k < a.K; ++k) {
        float lpk = (deflt == k) ? lu[R][lane] : -INFINITY;
        for (int j = 0; j < R; ++j)
            if (a.rule_class[rb + j] == k) lpk = log_add(lpk, lq[j][lane] + lu[j][lane]);
        a.probs[((int64_t)p * a.N + orig) * a.K + k] = expf(lpk);
    }
}

// soft_group in float-float arithmetic, one sample n to a lane (all lanes walk the same
// rules and conditions, so the gradient butterflies stay warp-wide). Forward: log q_r and
// log(1 - q_r) of every rule, lu and log p_y accumulated in float-float. Adjoint: lu_r recovered
// backwards as lu_{r+1} - log(1 - q_r) (exact to float-float precision; from the saved value at
// the first rule with q_r = 1, after which lu is -inf), the S and T recursions in float-float, and
// d ell / d u_c = -+exp(lq_r + lu_r + lT_{r+1} or lS_{r+1} - lp_y + log sigmoid(-u_c)) formed in the
// exponent. Per-set sums keep a fixed order: the loss in the caller's Kahan sum, the gradients
// through one butterfly per two conditions and fixed lanes. lq, lu: only with class probabilities.
template <bool BWD, bool CAT>
__device__ __forceinline__ void soft_group_ff(const SoftKArgs &a, int p, int rb, int R, int cb, int deflt, int64_t n,
                                           bool ok, const XView &x, float (*lq)[32], float (*lu)[32],
                                           float (*acc)[4], int lane, float &loss_s, float &loss_c)
{
    const int yv = ok ? a.y[n] : -1;
    // ---------------- forward
    ff lur{0.f, 0.f}, lpy{-INFINITY, 0.f}, lu_fin{0.f, 0.f};
    int jinf = R;                          // first rule with q = 1 (log(1 - q) = -inf)
    for (int j = 0; j < R; ++j) {
        const int r = rb + j;
        const int c0 = a.rule_cond_off[r], c1 = a.rule_cond_off[r + 1];
        const ff lqj = rule_logq_ff<CAT>(a, c0, c1, x);
        const ff l1q = rule_log1mq_ff<CAT>(a, c0, c1, x, lqj);
        if (a.rule_class[r] == yv) lpy = ff_log_add(lpy, ff_add(lqj, lur));
        if (lq) { lq[j][lane] = lqj.hi; lu[j][lane] = lur.hi; }
        if (l1q.hi == -INFINITY && jinf == R) { jinf = j; lu_fin = lur; }
        lur = ff_add(lur, l1q);
    }
    if (lq) lu[R][lane] = lur.hi;
    if (deflt == yv) lpy = ff_log_add(lpy, lur);
    if (ok) kadd_loss(loss_s, loss_c, -ff_f(lpy));
    if (lq && ok) write_probs(a, p, rb, R, deflt, n, lane, lq, lu);   // this lane's own slots
    if (!BWD) return;
    // ---------------- adjoint
    ff lS = deflt == yv ? ff{0.f, 0.f} : ff{-INFINITY, 0.f};
    ff lT = deflt == yv ? ff{-INFINITY, 0.f} : ff{0.f, 0.f};
    ff lu_next = lur;
    for (int j = R - 1; j >= 0; --j) {
        const int r = rb + j;
        const int cls = a.rule_class[r];
        const int c0 = a.rule_cond_off[r], c1 = a.rule_cond_off[r + 1];
        const ff lqj = rule_logq_ff<CAT>(a, c0, c1, x);
        const ff l1q = rule_log1mq_ff<CAT>(a, c0, c1, x, lqj);
        const ff luj = j > jinf ? ff{-INFINITY, 0.f} : (j == jinf ? lu_fin : ff_add(lu_next, ff_neg(l1q)));
        lu_next = luj;
        const bool same = cls == yv;
        const ff lw = same ? lT : lS;
        const bool zero = !ok || lw.hi == -INFINITY || lqj.hi == -INFINITY || luj.hi == -INFINITY;
        const ff G = ff_add(ff_add(ff_add(lqj, luj), lw), ff_neg(lpy));
        const float sign = same ? -1.f : 1.f;
        lS = ff_log_add(same ? lqj : ff{-INFINITY, 0.f}, ff_add(l1q, lS));
        lT = ff_log_add(same ? ff{-INFINITY, 0.f} : lqj, ff_add(l1q, lT));
        for (int c = c0; c < c1; c += 2) {
            const bool has1 = c + 1 < c1;
            const CondIn t[2] = {load_cond(a, c, x), load_cond(a, has1 ? c + 1 : c, x)};
            float2 g[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                if (i == 1 && !has1) break;
                const SoftRec &rc = t[i].rc;
                if ((CAT && (rc.meta & 4u)) || zero) continue;
                const ff u = margin_ff(a, t[i]);
                float l1pe;
                log_sigmoid_ff(u, l1pe);
                const ff lsn = u.hi > 0.f ? ff_add_f(ff_neg(u), -l1pe) : ff{-l1pe, 0.f};   // log sigmoid(-u)
                const float sg = (rc.meta & 2u) ? -1.f : 1.f;
                const float du = sign * expf(ff_f(ff_add(G, lsn))) * sg * a.inv_tau;
                g[i] = make_float2(du * t[i].xf, (rc.meta & 1u) ? -du * t[i].xg : -du);
            }
            reduce_pair(g[0], g[1], c - cb, has1, acc, lane);
        }
    }
}

// ------------------------------------------------------------------ the float path
// A condition with margin u has sigmoid(u) = 1 / (1 + E), E = e^-u. Over the conditions of a rule,
// with D = prod (1 + E) and z = D - 1,
//     q = 1 / D,    1 - q = z / D    (taken as 1 - q itself where q < 1/2),
// and z follows its own recursion z' = z + E D of positive terms, so that 1 - q keeps its relative
// accuracy where q rounds to 1. D beyond 1.6e38 counts as q = 0. E enters D and z with the smallest
// subnormal added, which only an E below 2^-124 notices (and 1 - q drops again): an infinite D stays
// infinite when it meets an E that came out 0 (a margin beyond 87), where 0 x inf would make a NaN and
// send the group to the float-float pass, whatever its p_y. (Accurate sets at a temperature of 0.02, 256
// of 6 rules on 100,000 x 32: 25 ms with nearly every group there, 0.93 so.) A group whose margins are
// not numbers still goes there.
// Everything after it is a sum of products of positive numbers as well: U_r = prod_{j<r} (1 - q_j),
// p_y and 1 - p_y over the rules, S_r and T_r backwards (S_r = [same] q + (1 - q) S_{r+1}, T_r with
// the other rules), and d ell / d log q_r = q_r U_r (S_{r+1} or -T_{r+1}) / p_y. No logarithm and no
// log-sum-exp is left: per condition and sample one ex2 forward, and an ex2 and a reciprocal in the
// adjoint, against two ex2, two degree-8 polynomials and a division before; relative errors grow
// by a rounding per factor instead of an ulp of the log-probability. Underflow only meets terms
// below 2^-126 of a sample whose p_y is at least e^-32 (others take the float-float pass), that is parts of
// a gradient below 9e-25 x / tau, which count as 0.
// A rule of more than SOFT_SEG conditions is taken in pieces, q = q1 q2, 1 - q = w1 + q1 w2.
//
// What bounds it: instruction issue. A lane holds 2 NV neighbouring samples, so that a feature is one
// 8- or 16-byte load, the products and sums are packed two-lane instructions, and reading a record
// is shared by all of them; records, with the sign of '<' folded into the coefficients, and rule
// ends sit in the warp's shared memory; U_r is parked in tensor memory by the staged-tile kernel
// (2 NV columns a rule, which leaves shared memory to twice the warps). Gradient sums of 16
// conditions are gathered in a 16 x 32 shared table and summed by all lanes at once: a condition
// costs one store and about two instructions of summing, where a warp butterfly per two conditions
// cost about 13 with its accumulator update. Forward + adjoint of 1024 sets x 32 rules x 4 conditions
// on 262,144 samples: 139.7 ms in the log domain with two samples a lane (238 warp instructions per
// condition and 64 samples), 70.3 ms so with U_r in tensor memory (123), 45.6 ms with E = e^-u in
// place of e^-|u| and its sign and four samples a lane (72, issue slots 68 % busy at 16 warps an SM;
// 44.6 without anything against inf x 0).
constexpr int SOFT_SEG = 32;               // conditions per piece of a rule
constexpr float SOFT_D_MAX = 1.6e38f;      // D from which q is 0 (above 2^126: its reciprocal is subnormal)
constexpr float SOFT_E_MAX = 8e37f;        // cap of E in E / (1 + E), whose reciprocal comes out 0 above 2^126
constexpr float SOFT_E_ADD = 1.4e-45f;     // the smallest subnormal: keeps E above 0 in D and z
constexpr int SOFT_NV_TILE = 2, SOFT_NV = 1;    // float2 per lane: staged-tile and per-warp kernel
constexpr int SOFT_CACHE = 4;              // conditions of a rule whose e the adjoint keeps in registers
constexpr int SOFT_GROWS = 16;             // conditions per gradient table
constexpr int SOFT_GPITCH = 288;           // bytes per table row: 32 lanes x 8, + 32 against bank conflicts
constexpr float SOFT_P_MIN = 1.26642e-14f;   // e^-32: p_y below which samples are evaluated in float-float
constexpr int32_t SREC_THR = -1, SREC_SET = -2;  // SoftRec4.g of a threshold / membership record

// A record staged for the warp's set: v = s (a x[f] - rhs) = a' x[f] + n' (x[g] for a pair).
struct __align__(16) SoftRec4 {
    uint32_t f;        // feature (staged tile: byte offset of its row)
    int32_t g;         // the same for a pair's second feature, SREC_THR, SREC_SET
    float a, n;        // s a and -s t or -s b; a membership test's set words
};

// One warp's shared memory.
struct SoftWarp {
    SoftRec4 *recs;    // [maxC]
    uint32_t *rules;   // [maxR] end of the rule's conditions (set-relative) | class << 16
    float4 *acc;       // [maxC] Kahan sums of d/da (x, y) and d/d(b or t) (z, w), without s / tau (adjoint)
    char *gtab;        // gradient table (adjoint)
    float2 *u;         // [maxR][NV][32] U_r of the lane's samples (per-warp kernel's adjoint)
    float2 *pc;        // [min(K, maxR + 1)][NV][32] class (or rule) probabilities (class probabilities)
};

__host__ __device__ constexpr size_t soft_main_bytes(int maxR, int maxC, bool bwd, bool tile, int pslots)
{
    return (size_t)maxC * sizeof(SoftRec4) + ((size_t)maxR * 4 + 15) / 16 * 16 +
           (bwd ? (size_t)maxC * sizeof(float4) + SOFT_GROWS * SOFT_GPITCH : 0) +
           (bwd && !tile ? (size_t)maxR * SOFT_NV * 32 * sizeof(float2) : 0) +
           (size_t)pslots * (tile ? SOFT_NV_TILE : SOFT_NV) * 32 * sizeof(float2);
}

__device__ __forceinline__ SoftWarp soft_warp(char *base, int maxR, int maxC, bool bwd, bool tile)
{
    SoftWarp m{};
    m.recs = reinterpret_cast<SoftRec4 *>(base);
    base += (size_t)maxC * sizeof(SoftRec4);
    m.rules = reinterpret_cast<uint32_t *>(base);
    base += ((size_t)maxR * 4 + 15) / 16 * 16;
    if (bwd) {
        m.acc = reinterpret_cast<float4 *>(base);
        base += (size_t)maxC * sizeof(float4);
        m.gtab = base;
        base += SOFT_GROWS * SOFT_GPITCH;
        if (!tile) { m.u = reinterpret_cast<float2 *>(base); base += (size_t)maxR * SOFT_NV * 32 * sizeof(float2); }
    }
    m.pc = reinterpret_cast<float2 *>(base);
    return m;
}

// The lane's 2 NV samples of some value, two to a register pair.
template <int NV>
struct Vec {
    float2 v[NV];
};

// The lane's samples of a feature, from the staged tile (o: the row's byte offset) or from global
// memory (o: the feature).
template <bool TILE, int NV>
struct XPair {
    const char *base;
    int64_t row;       // bytes per feature row (global form)
    __device__ __forceinline__ Vec<NV> operator()(uint32_t o) const
    {
        const char *p = TILE ? base + o : base + (int64_t)o * row;
        Vec<NV> r;
        if constexpr (NV == 2) {
            const float4 t = *reinterpret_cast<const float4 *>(p);
            r.v[0] = make_float2(t.x, t.y);
            r.v[1] = make_float2(t.z, t.w);
        } else {
            r.v[0] = *reinterpret_cast<const float2 *>(p);
        }
        return r;
    }
};

__device__ __forceinline__ float ex2_ftz(float x)
{
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ float rcp_ftz(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ float2 f2(float v) { return make_float2(v, v); }

// Products with subnormal operands and results taken as 0.
__device__ __forceinline__ float2 mul2_ftz(float2 a, float2 b)
{
    float2 r;
    asm("{\n\t.reg .b64 a, b, r;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tmul.rn.ftz.f32x2 r, a, b;\n\t"
        "mov.b64 {%0, %1}, r;\n\t}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}

// Tensor memory as a per-warp array of Vec (2 NV columns each; a warp reaches its own 32 lanes).
template <int NV>
__device__ __forceinline__ void tmem_put(uint32_t at, const Vec<NV> &u)
{
    if constexpr (NV == 2)
        asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(at),
                     "r"(__float_as_uint(u.v[0].x)), "r"(__float_as_uint(u.v[0].y)), "r"(__float_as_uint(u.v[1].x)),
                     "r"(__float_as_uint(u.v[1].y))
                     : "memory");
    else
        asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1, %2};" ::"r"(at), "r"(__float_as_uint(u.v[0].x)),
                     "r"(__float_as_uint(u.v[0].y))
                     : "memory");
}
// The load's registers hold the values only after tmem_wait_get on them.
template <int NV>
__device__ __forceinline__ void tmem_get(uint32_t at, uint32_t (&r)[2 * NV])
{
    if constexpr (NV == 2)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                     : "r"(at)
                     : "memory");
    else
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(at) : "memory");
}
template <int NV>
__device__ __forceinline__ void tmem_wait_get(uint32_t (&r)[2 * NV])
{
    if constexpr (NV == 2)
        asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3])::"memory");
    else
        asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(r[0]), "+r"(r[1])::"memory");
}
__device__ __forceinline__ void tmem_wait_put() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// min that keeps a NaN.
__device__ __forceinline__ float min_nan(float a, float b)
{
    float r;
    asm("min.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}

// E = e^-u of the lane's samples under record rc. nc = -log2(e) / tau.
template <bool TILE, int NV>
__device__ __forceinline__ Vec<NV> cond_e(const SoftRec4 &rc, const XPair<TILE, NV> &x, float nc)
{
    const Vec<NV> xf = x(rc.f);
    Vec<NV> t;
    if (rc.g >= 0) {
        const Vec<NV> xg = x((uint32_t)rc.g);
#pragma unroll
        for (int i = 0; i < NV; ++i) t.v[i] = __ffma2_rn(f2(rc.a), xf.v[i], __fmul2_rn(f2(rc.n), xg.v[i]));
    } else {
#pragma unroll
        for (int i = 0; i < NV; ++i) t.v[i] = __ffma2_rn(f2(rc.a), xf.v[i], f2(rc.n));
    }
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        t.v[i] = __fmul2_rn(t.v[i], f2(nc));
        t.v[i] = make_float2(ex2_ftz(t.v[i].x), ex2_ftz(t.v[i].y));
    }
    return t;
}

// D and z of a rule's piece so far, for the lane's samples.
template <int NV>
struct SoftProd {
    float2 D[NV], z[NV];
    uint32_t dead = 0;                               // bit i: a membership test of sample i failed
    __device__ __forceinline__ SoftProd()
    {
#pragma unroll
        for (int i = 0; i < NV; ++i) { D[i] = f2(1.f); z[i] = f2(0.f); }
    }
    __device__ __forceinline__ void add(const Vec<NV> &e)
    {
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            const float2 E = __fadd2_rn(e.v[i], f2(SOFT_E_ADD));
            z[i] = __ffma2_rn(E, D[i], z[i]);
            D[i] = __ffma2_rn(E, D[i], D[i]);
        }
    }
    // a membership test: its exact indicator
    template <bool TILE>
    __device__ __forceinline__ void member(const SoftRec4 &rc, const XPair<TILE, NV> &x)
    {
        const Vec<NV> v = x(rc.f);
        const uint32_t lo = __float_as_uint(rc.a), hi = __float_as_uint(rc.n);
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            if (!category_member(v.v[i].x, lo, hi)) dead |= 1u << (2 * i);
            if (!category_member(v.v[i].y, lo, hi)) dead |= 2u << (2 * i);
        }
    }
    template <bool CAT>
    __device__ __forceinline__ void close(Vec<NV> &q, Vec<NV> &w) const
    {
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            // beyond SOFT_D_MAX the reciprocal is subnormal and comes out 0, which the Newton step keeps
            const float2 d = make_float2(min_nan(D[i].x, SOFT_D_MAX), min_nan(D[i].y, SOFT_D_MAX));
            float2 r = make_float2(rcp_ftz(d.x), rcp_ftz(d.y));
            r = __ffma2_rn(r, __ffma2_rn(__fmul2_rn(d, f2(-1.f)), r, f2(1.f)), r);
            if (CAT && ((dead >> (2 * i)) & 1u)) r.x *= 0.f;     // a NaN stays
            if (CAT && ((dead >> (2 * i)) & 2u)) r.y *= 0.f;
            q.v[i] = r;
            // 1 - q rounded once where q < 1/2, else the quotient, which keeps a small 1 - q
            w.v[i] = mul2_ftz(z[i], r);                  // the added subnormals alone: 0
            const float2 v = __ffma2_rn(r, f2(-1.f), f2(1.f));
            if (r.x < 0.5f) w.v[i].x = v.x;
            if (r.y < 0.5f) w.v[i].y = v.y;
        }
    }
};

// The conditions [c, c1) of a rule into (q, w), a piece of SOFT_SEG at a time; (q, w) holds the rule
// so far.
template <bool CAT, bool TILE, int NV>
__device__ __forceinline__ void rule_more(const SoftRec4 *recs, int c, int c1, const XPair<TILE, NV> &x, float nc,
                                       Vec<NV> &q, Vec<NV> &w)
{
    while (c < c1) {
        const int end = min(c1, c + SOFT_SEG);
        SoftProd<NV> d;
        for (; c < end; ++c) {
            const SoftRec4 rc = recs[c];
            if (CAT && rc.g == SREC_SET) d.member(rc, x);
            else d.add(cond_e(rc, x, nc));
        }
        Vec<NV> q2, w2;
        d.template close<CAT>(q2, w2);
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            w.v[i] = __ffma2_rn(q.v[i], w2.v[i], w.v[i]);
            q.v[i] = __fmul2_rn(q.v[i], q2.v[i]);
        }
    }
}

// Sum a block of the gradient table (rows of conditions [16 blk, 16 blk + 16) of the set) over the
// warp into their accumulators: lane 2 s + h adds half of row s (16-byte pieces 2 i + h: eight lanes
// of a phase fall on distinct banks), the halves meet, and lane 2 s + h keeps component h.
__device__ __forceinline__ void grad_block(const SoftWarp &m, int blk, int nc, int lane)
{
    __syncwarp();
    const char *row = m.gtab + (lane >> 1) * SOFT_GPITCH + (lane & 1) * 16;
    float2 s0 = f2(0.f), s1 = f2(0.f);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float4 t = *reinterpret_cast<const float4 *>(row + 32 * i);
        s0 = __fadd2_rn(s0, make_float2(t.x, t.y));
        s1 = __fadd2_rn(s1, make_float2(t.z, t.w));
    }
    s0 = __fadd2_rn(s0, s1);
    const bool odd = lane & 1;
    const float other = __shfl_xor_sync(FULL, odd ? s0.x : s0.y, 1);
    const float v = (odd ? s0.y : s0.x) + other;
    const int ci = blk * SOFT_GROWS + (lane >> 1);
    if (ci < nc) {
        float2 *p = reinterpret_cast<float2 *>(m.acc + ci) + (lane & 1);
        float2 k = *p;
        kadd(k.x, k.y, v);
        *p = k;
    }
    __syncwarp();
}

// The lane's part of condition ci's two gradient sums into the table; the table is summed after the
// block's first condition (conditions arrive in descending order).
template <bool CAT, bool TILE, int NV>
__device__ __forceinline__ void cond_grads(const SoftWarp &m, int ci, int nconds, const Vec<NV> &e, const Vec<NV> &G,
                                           const XPair<TILE, NV> &x, int lane)
{
    const SoftRec4 rc = m.recs[ci];
    float2 g = f2(0.f);
    if (!(CAT && rc.g == SREC_SET)) {
        float2 h[NV];
#pragma unroll
        for (int i = 0; i < NV; ++i) {        // sigmoid(-u) = E / (1 + E)
            const float2 c = make_float2(fminf(e.v[i].x, SOFT_E_MAX), fminf(e.v[i].y, SOFT_E_MAX));
            const float2 d = __fadd2_rn(c, f2(1.f));
            h[i] = __fmul2_rn(__fmul2_rn(G.v[i], c), make_float2(rcp_ftz(d.x), rcp_ftz(d.y)));
        }
        const Vec<NV> xf = x(rc.f);
        float2 ga = __fmul2_rn(h[0], xf.v[0]), gb = h[0];
#pragma unroll
        for (int i = 1; i < NV; ++i) ga = __ffma2_rn(h[i], xf.v[i], ga);
        if (rc.g >= 0) {
            const Vec<NV> xg = x((uint32_t)rc.g);
            gb = __fmul2_rn(h[0], xg.v[0]);
#pragma unroll
            for (int i = 1; i < NV; ++i) gb = __ffma2_rn(h[i], xg.v[i], gb);
        } else {
#pragma unroll
            for (int i = 1; i < NV; ++i) gb = __fadd2_rn(gb, h[i]);
        }
        g = make_float2(ga.x + ga.y, gb.x + gb.y);
    }
    *reinterpret_cast<float2 *>(m.gtab + (ci & (SOFT_GROWS - 1)) * SOFT_GPITCH + lane * 8) = g;
    if ((ci & (SOFT_GROWS - 1)) == 0) grad_block(m, ci / SOFT_GROWS, nconds, lane);
}

// Forward (and adjoint) of a set of R rules over one group of 64 NV samples: lane l holds samples
// n0 + 2 NV l + i (bit i of valid: the sample exists). tm: the warp's tensor-memory base
// (staged-tile adjoint). Returns a bit for each SOFT_FF_GROUP of its samples from which nothing was added,
// since some sample's p_y in it is below e^-32 (all of them when something is not a number): the bits go
// to the task's list, and k_soft_ff evaluates these samples in float-float after this kernel.
template <bool BWD, bool CAT, bool TILE, int NV>
__device__ __forceinline__ uint32_t soft_group(const SoftKArgs &a, const SoftWarp &m, int p, int R, int nconds, int deflt,
                                           int64_t n0, uint32_t valid, const XPair<TILE, NV> &x, float nc, uint32_t tm,
                                           int lane, float &loss_s, float &loss_c)
{
    const int64_t n = n0 + 2 * NV * lane;
    int y[2 * NV];
#pragma unroll
    for (int i = 0; i < 2 * NV; ++i) y[i] = ((valid >> i) & 1u) ? a.y[n + i] : -1;
    const bool by_class = a.K <= a.maxR + 1;
    float2 *const pc = m.pc + lane;
    Vec<NV> U, py, po;
#pragma unroll
    for (int i = 0; i < NV; ++i) { U.v[i] = f2(1.f); py.v[i] = f2(0.f); po.v[i] = f2(0.f); }
    if (!BWD && a.probs && by_class)
        for (int k = 0; k < a.K * NV; ++k) pc[k * 32] = f2(0.f);
    const auto add_class = [&](int cls, const Vec<NV> &pr) {
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            if (cls == y[2 * i]) py.v[i].x += pr.v[i].x; else po.v[i].x += pr.v[i].x;
            if (cls == y[2 * i + 1]) py.v[i].y += pr.v[i].y; else po.v[i].y += pr.v[i].y;
        }
    };
    int c0 = 0;
    for (int j = 0; j < R; ++j) {
        const uint32_t ru = m.rules[j];
        const int c1 = ru & 0xFFFFu, cls = ru >> 16;
        Vec<NV> q, w;
        {
            SoftProd<NV> d;
            const int end = min(c1, c0 + SOFT_SEG);
#pragma unroll 2
            for (int c = c0; c < end; ++c) {
                const SoftRec4 rc = m.recs[c];
                if (CAT && rc.g == SREC_SET) d.member(rc, x);
                else d.add(cond_e(rc, x, nc));
            }
            d.template close<CAT>(q, w);
            if (end < c1) rule_more<CAT>(m.recs, end, c1, x, nc, q, w);
        }
        if (BWD) {
            if constexpr (TILE) tmem_put<NV>(tm + 2 * NV * j, U);
            else
#pragma unroll
                for (int i = 0; i < NV; ++i) m.u[(j * NV + i) * 32 + lane] = U.v[i];
        }
        Vec<NV> pr;
#pragma unroll
        for (int i = 0; i < NV; ++i) pr.v[i] = __fmul2_rn(q.v[i], U.v[i]);
        add_class(cls, pr);
        if (!BWD && a.probs) {
#pragma unroll
            for (int i = 0; i < NV; ++i) {
                float2 *s = pc + ((by_class ? cls : j) * NV + i) * 32;
                *s = by_class ? __fadd2_rn(*s, pr.v[i]) : pr.v[i];
            }
        }
#pragma unroll
        for (int i = 0; i < NV; ++i) U.v[i] = __fmul2_rn(U.v[i], w.v[i]);
        c0 = c1;
    }
    add_class(deflt, U);
    // every q_r went into p_y or 1 - p_y: a NaN anywhere shows in one of them (looked for beyond the
    // data's end too, where a NaN times a weight of 0 would spoil the sums)
    bool nan = false, far = false;
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        nan |= !(py.v[i].x >= 0.f && po.v[i].x >= 0.f) || !(py.v[i].y >= 0.f && po.v[i].y >= 0.f);
        far |= (((valid >> (2 * i)) & 1u) && py.v[i].x < SOFT_P_MIN) ||
               (((valid >> (2 * i + 1)) & 1u) && py.v[i].y < SOFT_P_MIN);
    }
    if (BWD && TILE) tmem_wait_put();
    uint32_t left = 0;
    {
        constexpr uint32_t ALL = (1u << NV) - 1u;    // SOFT_FF_GROUP is 32 / NV lanes
        const uint32_t f = __ballot_sync(FULL, far);
        if (NV == 1) left = f ? 1u : 0u;
        else left = ((f & 0xFFFFu) ? 1u : 0u) | ((f >> 16) ? 2u : 0u);
        if (__any_sync(FULL, nan)) left = ALL;
        if (left == ALL) return ALL;
        if ((left >> (NV == 1 ? 0 : lane >> 4)) & 1u) valid = 0;     // finite: a weight of 0 leaves them out
    }
    // -log p_y; near 1 from 1 - p_y, which is its own sum of positive terms
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        if ((valid >> (2 * i)) & 1u) kadd_loss(loss_s, loss_c, py.v[i].x < 0.5f ? -logf(py.v[i].x) : -log1pf(-po.v[i].x));
        if ((valid >> (2 * i + 1)) & 1u)
            kadd_loss(loss_s, loss_c, py.v[i].y < 0.5f ? -logf(py.v[i].y) : -log1pf(-po.v[i].y));
    }
    if (!BWD) {
        if (a.probs) {
            int64_t o[2 * NV];
#pragma unroll
            for (int i = 0; i < 2 * NV; ++i) o[i] = ((valid >> i) & 1u) ? ((int64_t)p * a.N + a.perm[n + i]) * a.K : -1;
            for (int k = 0; k < a.K; ++k) {
#pragma unroll
                for (int i = 0; i < NV; ++i) {
                    float2 v = f2(0.f);
                    if (by_class) v = pc[(k * NV + i) * 32];
                    else
                        for (int j = 0; j < R; ++j)
                            if ((int)(m.rules[j] >> 16) == k) v = __fadd2_rn(v, pc[(j * NV + i) * 32]);
                    if (k == deflt) v = __fadd2_rn(v, U.v[i]);
                    if (o[2 * i] >= 0) a.probs[o[2 * i] + k] = v.x;
                    if (o[2 * i + 1] >= 0) a.probs[o[2 * i + 1] + k] = v.y;
                }
            }
        }
        return left;
    }
    // ---------------- adjoint
    __syncwarp();
    Vec<NV> rp, S, T;
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        rp.v[i] = make_float2(((valid >> (2 * i)) & 1u) ? 1.f / py.v[i].x : 0.f,
                              ((valid >> (2 * i + 1)) & 1u) ? 1.f / py.v[i].y : 0.f);
        S.v[i] = make_float2(deflt == y[2 * i] ? 1.f : 0.f, deflt == y[2 * i + 1] ? 1.f : 0.f);
        T.v[i] = make_float2(1.f - S.v[i].x, 1.f - S.v[i].y);
    }
    uint32_t ru = R > 0 ? m.rules[R - 1] : 0u;
    for (int j = R - 1; j >= 0; --j) {
        const int c1 = ru & 0xFFFFu, cls = ru >> 16;
        ru = j > 0 ? m.rules[j - 1] : 0u;
        const int b0 = ru & 0xFFFFu;                 // the rule's first condition
        uint32_t ur[2 * NV];
        if constexpr (TILE) tmem_get<NV>(tm + 2 * NV * j, ur);
        Vec<NV> q, w, ce[SOFT_CACHE];
        {
            SoftProd<NV> d;
#pragma unroll
            for (int k = 0; k < SOFT_CACHE; ++k) {
                if (b0 + k >= c1) break;
                const SoftRec4 rc = m.recs[b0 + k];
                if (CAT && rc.g == SREC_SET) d.member(rc, x);
                else {
                    ce[k] = cond_e(rc, x, nc);
                    d.add(ce[k]);
                }
            }
            const int end = min(c1, b0 + SOFT_SEG);
            for (int c = b0 + SOFT_CACHE; c < end; ++c) {
                const SoftRec4 rc = m.recs[c];
                if (CAT && rc.g == SREC_SET) d.member(rc, x);
                else d.add(cond_e(rc, x, nc));
            }
            d.template close<CAT>(q, w);
            if (end < c1) rule_more<CAT>(m.recs, end, c1, x, nc, q, w);
        }
        if constexpr (TILE) tmem_wait_get<NV>(ur);
        Vec<NV> G;
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            float2 Uj;
            if constexpr (TILE) Uj = make_float2(__uint_as_float(ur[2 * i]), __uint_as_float(ur[2 * i + 1]));
            else Uj = m.u[(j * NV + i) * 32 + lane];
            const bool s0 = cls == y[2 * i], s1 = cls == y[2 * i + 1];
            const float2 pr = __fmul2_rn(__fmul2_rn(Uj, rp.v[i]), q.v[i]);
            G.v[i] = __fmul2_rn(pr, make_float2(s0 ? -T.v[i].x : S.v[i].x, s1 ? -T.v[i].y : S.v[i].y));
            S.v[i] = __ffma2_rn(w.v[i], S.v[i], make_float2(s0 ? q.v[i].x : 0.f, s1 ? q.v[i].y : 0.f));
            T.v[i] = __ffma2_rn(w.v[i], T.v[i], make_float2(s0 ? 0.f : q.v[i].x, s1 ? 0.f : q.v[i].y));
        }
        for (int c = c1 - 1; c >= b0 + SOFT_CACHE; --c) {
            const SoftRec4 rc = m.recs[c];
            Vec<NV> e = {};
            if (!(CAT && rc.g == SREC_SET)) e = cond_e(rc, x, nc);
            cond_grads<CAT>(m, c, nconds, e, G, x, lane);
        }
#pragma unroll
        for (int k = SOFT_CACHE - 1; k >= 0; --k)
            if (b0 + k < c1) cond_grads<CAT>(m, b0 + k, nconds, ce[k], G, x, lane);
    }
    return left;
}

// Stage a set's records and rule ends for the warp (row: bytes of a staged feature row, or 1 for
// plain feature numbers) and clear its accumulators. Returns the number of conditions.
template <bool BWD>
__device__ __forceinline__ int soft_stage(const SoftKArgs &a, const SoftWarp &m, int rb, int R, uint32_t row, int lane)
{
    const int cb = a.rule_cond_off[rb], nc = a.rule_cond_off[rb + R] - cb;
    __syncwarp();
    for (int i = lane; i < nc; i += 32) {
        const SoftRec r = a.recs[cb + i];
        const bool pair = r.meta & 1u, lt = r.meta & 2u, set = r.meta & 4u;
        SoftRec4 o;
        o.f = r.f * row;
        o.g = set ? SREC_SET : (pair ? (int32_t)(r.g * row) : SREC_THR);
        o.a = set ? r.a : (lt ? -r.a : r.a);
        o.n = set ? r.bt : (lt ? r.bt : -r.bt);
        m.recs[i] = o;
        if (BWD) m.acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    for (int j = lane; j < R; j += 32)
        m.rules[j] = (uint32_t)(a.rule_cond_off[rb + j + 1] - cb) | (uint32_t)a.rule_class[rb + j] << 16;
    __syncwarp();
    return nc;
}

// Write a task's chunk partials (loss; gradient sums when BWD, with the factor s / tau of
// du/da = s x / tau and -s / tau of du/dt that the table's sums leave out).
template <bool BWD>
__device__ __forceinline__ void soft_flush(const SoftKArgs &a, const SoftWarp &m, int p, int ch, int cb, int nc,
                                           float loss_s, int lane)
{
    float ls = loss_s;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ls += __shfl_xor_sync(FULL, ls, o);
    if (lane == 0) a.part_loss[(int64_t)ch * a.P + p] = ls;
    if (BWD) {
        __syncwarp();
        for (int i = lane; i < nc; i += 32) {
            const float sc = (a.recs[cb + i].meta & 2u) ? -a.inv_tau : a.inv_tau;
            const float4 g = m.acc[i];
            a.part_ga[(int64_t)ch * a.Ccap + cb + i] = g.x * sc;
            a.part_gbt[(int64_t)ch * a.Ccap + cb + i] = -g.z * sc;
        }
        __syncwarp();
    }
}

constexpr float LOG2E = 1.44269504f;

// Bit i: the lane's sample i exists, `left` samples being left from its first one on.
template <int NV>
__device__ __forceinline__ uint32_t valid_mask(int64_t left)
{
    return left >= 2 * NV ? (1u << (2 * NV)) - 1u : (left <= 0 ? 0u : (1u << (int)left) - 1u);
}

template <bool BWD, bool CAT>
__global__ void __launch_bounds__(SOFT_W * 32) k_soft(SoftKArgs a)
{
    extern __shared__ __align__(16) char smc[];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t tasks = (int64_t)a.P * a.nchunks;
    const SoftWarp m = soft_warp(smc + soft_main_bytes(a.maxR, a.maxC, BWD, false, a.pslots) * w, a.maxR, a.maxC, BWD, false);
    const float nc = -a.inv_tau * LOG2E;
    if (*a.status) return;

    while (true) {
        int64_t task = 0;
        if (lane == 0) task = atomicAdd(a.next, 1);
        task = __shfl_sync(FULL, task, 0);
        if (task >= tasks) break;
        const int p = a.order[task / a.nchunks];
        const int ch = (int)(task % a.nchunks);
        const int rb = a.set_rule_off[p], R = a.set_rule_off[p + 1] - rb;
        const int nconds = soft_stage<BWD>(a, m, rb, R, 1u, lane);
        float loss_s = 0.f, loss_c = 0.f;
        const int64_t s0 = (int64_t)ch * a.chunk;
        const int64_t s1 = min(s0 + a.chunk, a.N);
        uint32_t *fbits = a.ffbits + ((int64_t)ch * a.P + p) * a.ff_wpt;
        uint32_t fw = 0, ff = 0;
        int gi = 0;
        for (int64_t nb = s0; nb < s1; nb += 64 * SOFT_NV, ++gi) {
            const int64_t n = nb + 2 * SOFT_NV * lane;
            const uint32_t valid = valid_mask<SOFT_NV>(s1 - n);
            // the dataset is padded to a multiple of 256 samples: every read stays inside it
            const XPair<false, SOFT_NV> x{reinterpret_cast<const char *>(a.Xt + n), a.n_pad * (int64_t)sizeof(float)};
            fw |= soft_group<BWD, CAT, false, SOFT_NV>(a, m, p, R, nconds, a.set_default[p], nb, valid, x, nc, 0u, lane,
                                                       loss_s, loss_c) << (gi & 31);
            if ((gi & 31) == 31 || nb + 64 * SOFT_NV >= s1) {
                if (lane == 0) fbits[gi >> 5] = fw;
                ff |= fw;
                fw = 0;
            }
        }
        soft_flush<BWD>(a, m, p, ch, a.rule_cond_off[rb], nconds, loss_s, lane);
        if (lane == 0 && ff) a.fflist[atomicAdd(a.next + SOFT_NEXT_FF_LEN, 1)] = (int32_t)((int64_t)ch * a.P + p);
    }
}

// The same evaluation with the warps of a team on as many neighbouring sets (in size order) over
// the same chunk, four samples a lane: the features of each group of 128 are staged once per team in
// shared memory (double-buffered asynchronous copies), so condition loads are shared-memory reads.
constexpr int SOFT_TW_MIN = 4, SOFT_TW_MAX = 16;   // warps per CTA (and sets per team) of the staged-tile kernel
constexpr int SOFT_GT = 64 * SOFT_NV_TILE;    // samples per group of the staged-tile kernel
constexpr int SOFT_TILE_STATIC = 256;   // bytes kept for the kernel's static shared memory

__device__ __forceinline__ void stage_group(float *dst, const float *Xt, int64_t n_pad, int F, int64_t nb, int thread,
                                            int threads)
{
    // F rows x G samples, 16-byte pieces
    constexpr int PR = SOFT_GT / 4;   // pieces per row
    for (int i = thread; i < F * PR; i += threads) {
        const int f = i / PR, q = i % PR;
        const float *src = Xt + (int64_t)f * n_pad + nb + 4 * q;
        const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst + f * SOFT_GT + 4 * q);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// A CTA is a.teams teams of TW warps, each taking tasks of its own with its own buffers and named
// barrier (a kernel that allocates tensor memory runs one CTA per SM: teams take the place of
// further CTAs; the forward, which needs none, runs one team per CTA). The adjoint's CTA allocates
// a.tm_cols tensor-memory columns for U_r: warp w holds rule r of its set at columns
// (w / 4) 2 NV maxR + 2 NV r of its own 32 lanes. One barrier per group: a warp that has passed it is done
// with the buffer that is restaged after it.
template <bool BWD, bool CAT>
__global__ void __maxnreg__(128) k_soft_tile(SoftKArgs a, int F)
{
    extern __shared__ __align__(16) char smc[];
    __shared__ int64_t s_tasks[SOFT_TW_MAX / SOFT_TW_MIN];
    __shared__ uint32_t s_tm;
    const int lane = threadIdx.x & 31;
    const int TW = (int)(blockDim.x >> 5) / a.teams;  // sets per team
    const int team = (int)(threadIdx.x >> 5) / TW, w = (int)(threadIdx.x >> 5) - team * TW;
    const int64_t set_groups = (a.P + TW - 1) / TW;
    const int64_t tasks = set_groups * a.nchunks;
    const size_t per_warp = soft_main_bytes(a.maxR, a.maxC, BWD, true, a.pslots);
    char *const team_sm = smc + (per_warp * TW + sizeof(float) * 2 * SOFT_GT * (size_t)F) * team;
    const SoftWarp m = soft_warp(team_sm + per_warp * w, a.maxR, a.maxC, BWD, true);
    float *xbuf = reinterpret_cast<float *>(team_sm + per_warp * TW);     // [2][F][G]
    const float nc = -a.inv_tau * LOG2E;
    const auto team_sync = [&] { asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "r"(TW * 32) : "memory"); };
    if (*a.status) return;
    uint32_t tm = 0;
    if (BWD) {
        const uint32_t cw = threadIdx.x >> 5;
        if (cw == 0) {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                             (uint32_t)__cvta_generic_to_shared(&s_tm)),
                         "r"(a.tm_cols)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        tm = s_tm + ((cw & 3u) << 21) + (cw >> 2) * (2u * SOFT_NV_TILE) * (uint32_t)a.maxR;
    }

    while (true) {
        team_sync();
        if (w == 0 && lane == 0) s_tasks[team] = atomicAdd(a.next, 1);
        team_sync();
        const int64_t task = s_tasks[team];
        if (task >= tasks) break;
        const int g = (int)(task / a.nchunks);
        const int ch = (int)(task % a.nchunks);
        const int64_t s0 = (int64_t)ch * a.chunk;
        const int64_t s1 = min(s0 + a.chunk, a.N);
        stage_group(xbuf, a.Xt, a.n_pad, F, s0, w * 32 + lane, TW * 32);
        // the CTA's warps move through the chunk in step: sets of one group have similar sizes
        const bool active = g * TW + w < a.P;
        const int p = active ? a.order[g * TW + w] : 0;
        int rb = 0, R = 0, nconds = 0, deflt = 0;
        if (active) {
            rb = a.set_rule_off[p];
            R = a.set_rule_off[p + 1] - rb;
            deflt = a.set_default[p];
            nconds = soft_stage<BWD>(a, m, rb, R, SOFT_GT * (uint32_t)sizeof(float), lane);
        }
        float loss_s = 0.f, loss_c = 0.f;
        uint32_t fw = 0, ff = 0;
        const int ngroups = (int)((s1 - s0 + SOFT_GT - 1) / SOFT_GT);
        uint32_t *fbits = a.ffbits + ((int64_t)ch * a.P + p) * a.ff_wpt;
        for (int gi = 0; gi < ngroups; ++gi) {
            const int64_t nb = s0 + SOFT_GT * (int64_t)gi;
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            team_sync();
            if (gi + 1 < ngroups)
                stage_group(xbuf + ((gi + 1) & 1) * F * SOFT_GT, a.Xt, a.n_pad, F, nb + SOFT_GT, w * 32 + lane, TW * 32);
            if (active) {
                constexpr int NV = SOFT_NV_TILE;
                const uint32_t valid = valid_mask<NV>(s1 - nb - 2 * NV * lane);
                const XPair<true, NV> x{reinterpret_cast<const char *>(xbuf + (gi & 1) * F * SOFT_GT + 2 * NV * lane), 0};
                fw |= soft_group<BWD, CAT, true, NV>(a, m, p, R, nconds, deflt, nb, valid, x, nc, tm, lane, loss_s, loss_c)
                      << (NV * gi & 31);
                if ((NV * (gi + 1) & 31) == 0 || gi + 1 == ngroups) {
                    if (lane == 0) fbits[NV * gi >> 5] = fw;
                    ff |= fw;
                    fw = 0;
                }
            }
        }
        if (active) {
            soft_flush<BWD>(a, m, p, ch, a.rule_cond_off[rb], nconds, loss_s, lane);
            if (lane == 0 && ff) a.fflist[atomicAdd(a.next + SOFT_NEXT_FF_LEN, 1)] = (int32_t)((int64_t)ch * a.P + p);
        }
    }
    if (BWD) {
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (threadIdx.x < 32)
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(s_tm), "r"(a.tm_cols));
    }
}

// The float-float pass: the CTAs take the (set, chunk) tasks that the main kernel listed, all warps of
// a CTA on one task: warp i of W evaluates every W-th 32 samples of those whose bits the main kernel set
// (SOFT_FF_GROUP samples each, left out there) in float-float (soft_group_ff), its loss and gradient sums
// Kahan-summed in their order; the warps' sums are added to the task's partials in warp order, so that
// results do not depend on the order of the list. Runs after the main kernel on the same stream; features
// are read from global memory, one sample to a lane. Few marked samples are bound by the chain of one
// warp's conditions (a record, its features, the arithmetic, one after another), hence FF_W = 16 warps to
// a task (FF_W_PROBS = 8 for class probabilities, whose arrays leave room for fewer warps an SM); many by
// the warps that an SM holds, so that as many CTAs run as fit. With 4 / 8 / 16 warps: class probabilities
// of 48 sets on 20,000 x 30 (9 % of the samples marked) 231 / 187 / 226 us a call; the autograd step of 64
// sets on 100,000 x 32 (two seeds; many marked samples in a few sets) 1.70 and 3.10 / 1.59 and 2.40 / 1.53
// and 1.92 ms; nearly every sample of 256 sets of 6 rules on 100,000 x 32 10.5 / 11.0 / 10.5 ms (with the
// loads of four conditions issued together, whose unrolled code is four times as long, twice that).
template <bool BWD, bool CAT>
__global__ void __launch_bounds__(FF_W * 32, 2) k_soft_ff(SoftKArgs a)
{
    extern __shared__ __align__(16) float sm[];
    __shared__ int s_item;
    __shared__ float s_loss[FF_W];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, W = blockDim.x >> 5;
    if (*a.status) return;
    const int items = a.next[SOFT_NEXT_FF_LEN];
    const size_t per_warp = soft_ff_floats(a.maxR, a.maxC, a.probs != nullptr);
    float *base_w = sm + per_warp * w;
    float(*acc)[4] = reinterpret_cast<float(*)[4]>(base_w);
    float(*lu)[32] = a.probs ? reinterpret_cast<float(*)[32]>(base_w + (size_t)a.maxC * 4) : nullptr;
    float(*lq)[32] = a.probs ? lu + a.maxR + 1 : nullptr;
    while (true) {
        __syncthreads();
        if (threadIdx.x == 0) s_item = atomicAdd(a.next + SOFT_NEXT_FF, 1);
        __syncthreads();
        if (s_item >= items) break;
        const int64_t task = a.fflist[s_item];         // ch * P + p
        const int p = (int)(task % a.P), ch = (int)(task / a.P);
        const int rb = a.set_rule_off[p], re = a.set_rule_off[p + 1];
        const int cb = a.rule_cond_off[rb], ce = a.rule_cond_off[re];
        const int deflt = a.set_default[p];
        if (BWD) {
            for (int i = lane; i < (ce - cb); i += 32) {
                acc[i][0] = 0.f; acc[i][1] = 0.f; acc[i][2] = 0.f; acc[i][3] = 0.f;
            }
            __syncwarp();
        }
        float loss_s = 0.f, loss_c = 0.f;
        const int64_t s0 = (int64_t)ch * a.chunk;
        const int64_t s1 = min(s0 + a.chunk, a.N);
        const uint32_t *fbits = a.ffbits + task * a.ff_wpt;
        uint32_t fw = 0;
        int k = 0;                                     // 32-sample pieces of marked groups so far
        for (int64_t nb = s0; nb < s1; nb += 32) {
            const int gi = (int)((nb - s0) / SOFT_FF_GROUP);
            if ((nb - s0) % (32 * SOFT_FF_GROUP) == 0) fw = fbits[gi >> 5];
            if (!((fw >> (gi & 31)) & 1u)) continue;
            if ((k++ & (W - 1)) != w) continue;
            const int64_t n = nb + lane;
            soft_group_ff<BWD, CAT>(a, p, rb, re - rb, cb, deflt, n, n < s1, XView{a.Xt + n, a.n_pad}, lq, lu, acc,
                                    lane, loss_s, loss_c);
        }
        float ls = loss_s;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ls += __shfl_xor_sync(FULL, ls, o);
        if (lane == 0) s_loss[w] = ls;
        __syncthreads();
        if (threadIdx.x == 0) {
            float t = s_loss[0];
            for (int i = 1; i < W; ++i) t += s_loss[i];
            a.part_loss[task] += t;
        }
        if (BWD) {
            for (int i = threadIdx.x; i < (ce - cb); i += W * 32) {
                float ga = 0.f, gbt = 0.f;
                for (int v = 0; v < W; ++v) {
                    const float *t = sm + per_warp * v + 4 * (size_t)i;
                    ga += t[0];
                    gbt += t[2];
                }
                a.part_ga[(int64_t)ch * a.Ccap + cb + i] += ga;
                a.part_gbt[(int64_t)ch * a.Ccap + cb + i] += gbt;
            }
        }
    }
}

__device__ __forceinline__ float tree_sum_strided(const float *base, int64_t stride, int n)
{
    // pairwise sum of base[0], base[stride], ... (n <= SOFT_MAX_CHUNKS) in a fixed order
    float v[SOFT_MAX_CHUNKS];
#pragma unroll
    for (int i = 0; i < SOFT_MAX_CHUNKS; ++i) v[i] = (i < n) ? base[(int64_t)i * stride] : 0.f;
#pragma unroll
    for (int w = 1; w < SOFT_MAX_CHUNKS; w <<= 1)
#pragma unroll
        for (int i = 0; i + w < SOFT_MAX_CHUNKS; i += 2 * w) v[i] += v[i + w];
    return v[0];
}

__global__ void k_soft_reduce_loss(const float *part_loss, int nchunks, int P, float inv_n, float *loss,
                                   const uint32_t *status)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= P || *status) return;
    loss[p] = tree_sum_strided(part_loss + p, P, nchunks) * inv_n;
}

// One Adam update of parameter *p with gradient g and moments *m, *v; every operation separately
// rounded, so that the result does not depend on the file's contraction setting.
__device__ __forceinline__ void adam_one(float *p, float g, float *m, float *v, float bc1, float bc2,
                                         const SoftAdam &ad)
{
    const float mk = __fadd_rn(__fmul_rn(ad.b1, *m), __fmul_rn(1.0f - ad.b1, g));
    const float vk = __fadd_rn(__fmul_rn(ad.b2, *v), __fmul_rn(__fmul_rn(1.0f - ad.b2, g), g));
    *m = mk;
    *v = vk;
    const float mh = __fdiv_rn(mk, bc1), vh = __fdiv_rn(vk, bc2);
    *p = __fsub_rn(*p, __fdiv_rn(__fmul_rn(ad.lr, mh), __fadd_rn(sqrtf(vh), ad.eps)));
}

// One CTA per set, its threads looping over the set's conditions (grads scaled by dloss[p] / N);
// thread 0 also writes the set's loss when `loss` is given; with adam.a the Adam update of the
// set's conditions follows at once.
__global__ void k_soft_reduce_grad(const float *part_ga, const float *part_gbt, const float *part_loss,
                                   int nchunks, const int32_t *set_rule_off, const int32_t *rule_cond_off,
                                   const SoftRec *recs, int P, int64_t C, const float *dloss,
                                   float inv_n, float *grad_a, float *grad_b, float *grad_t, float *loss,
                                   SoftAdam adam, const uint32_t *status)
{
    const int p = blockIdx.x;
    if (p >= P || *status) return;
    if (loss && threadIdx.x == 0) loss[p] = tree_sum_strided(part_loss + p, P, nchunks) * inv_n;
    const float bc1 = 1.0f - powf(adam.b1, (float)adam.step), bc2 = 1.0f - powf(adam.b2, (float)adam.step);
    const int cb = rule_cond_off[set_rule_off[p]], ce = rule_cond_off[set_rule_off[p + 1]];
    const float scale = dloss[p] * inv_n;
    for (int c = cb + threadIdx.x; c < ce; c += blockDim.x) {
        const float ga = tree_sum_strided(part_ga + c, C, nchunks) * scale;
        const float gbt = tree_sum_strided(part_gbt + c, C, nchunks) * scale;
        const bool pair = recs[c].meta & 1u;
        grad_a[c] = ga;
        grad_b[c] = pair ? gbt : 0.f;
        grad_t[c] = pair ? 0.f : gbt;
        if (adam.a) {
            adam_one(adam.a + c, ga, adam.m + 2 * c, adam.v + 2 * c, bc1, bc2, adam);
            adam_one((pair ? adam.b : adam.t) + c, gbt, adam.m + 2 * c + 1, adam.v + 2 * c + 1, bc1, bc2, adam);
        }
    }
}

}  // namespace

// Shared body of both entry points. `known` = bounds given by the caller (no host readback).
template <bool CAT>
static void set_soft_attributes(Ctx *ctx)
{
    cudaFuncSetAttribute(k_soft<true, CAT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ctx->smem_optin);
    cudaFuncSetAttribute(k_soft<false, CAT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ctx->smem_optin);
    // the staged-tile and float-float kernels have a little static shared memory of their own
    cudaFuncSetAttribute(k_soft_tile<true, CAT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)ctx->smem_optin - SOFT_TILE_STATIC);
    cudaFuncSetAttribute(k_soft_tile<false, CAT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)ctx->smem_optin - SOFT_TILE_STATIC);
    cudaFuncSetAttribute(k_soft_ff<true, CAT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)ctx->smem_optin - SOFT_TILE_STATIC);
    cudaFuncSetAttribute(k_soft_ff<false, CAT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)ctx->smem_optin - SOFT_TILE_STATIC);
    cudaGetLastError();
}

// Tensor-memory columns of a staged-tile CTA of tw warps: U_r takes 2 NV per rule and group of four
// warps; allocations are powers of two from 32 to the SM's 512.
constexpr int TMEM_COLS = 512;
static int soft_tm_cols(int tw, int maxR)
{
    const int need = (tw + 3) / 4 * 2 * SOFT_NV_TILE * maxR;
    int cols = 32;
    while (cols < need) cols *= 2;
    return cols;
}

// Launch shape of the soft kernel: warps per team and teams per CTA (staged-tile form), resident CTAs
// per SM.
struct SoftShape {
    int tw = SOFT_TW_MIN;
    int teams = 1;
    int per_sm = 1;
};

// Shared memory of a team of tw warps: the warps' arrays and two feature tiles.
static size_t soft_team_bytes(int tw, size_t per_warp, int F)
{
    return per_warp * tw + sizeof(float) * 2 * SOFT_GT * (size_t)F;
}

// Resident teams per SM of the staged-tile kernel with tw warps to a team (0 when one does not fit):
// CTAs of one team in the forward, teams of one CTA in the adjoint (tensor memory: one CTA per SM).
template <bool BWD, bool CAT>
static int soft_teams_per_sm(Ctx *ctx, int tw, size_t per_warp, int F, int maxR)
{
    const size_t bytes = soft_team_bytes(tw, per_warp, F);
    if (bytes + SOFT_TILE_STATIC > ctx->smem_optin) return 0;
    if (BWD) {
        int n = std::min(SOFT_TW_MAX / tw, (int)((ctx->smem_optin - SOFT_TILE_STATIC) / bytes));
        while (n > 0 && (n * tw + 3) / 4 * 2 * SOFT_NV_TILE * maxR > TMEM_COLS) --n;
        return n;
    }
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_soft_tile<BWD, CAT>, tw * 32, bytes) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return per_sm;
}

// The staged-tile form takes the number of warps per team that keeps the most warps resident for
// this batch's per-warp arrays (ties: fewer warps per team, so that a team's sets are closer in
// size); small populations keep at most P / 8 warps per team, since a team walks its sets in step
// and a wide one over few sets of uneven size waits for the longest.
template <bool CAT>
static SoftShape soft_shape(Ctx *ctx, bool tiled, bool bwd, int F, size_t smem, size_t per_warp, int P, int maxR)
{
    SoftShape sh;
    if (tiled) {
        int best = 0;
        const int tw_max = std::max(SOFT_TW_MIN, std::min(SOFT_TW_MAX, P / 8));
        for (int t = SOFT_TW_MIN; t <= tw_max; ++t) {
            const int c = bwd ? soft_teams_per_sm<true, CAT>(ctx, t, per_warp, F, maxR)
                              : soft_teams_per_sm<false, CAT>(ctx, t, per_warp, F, maxR);
            if (c * t > best) {
                best = c * t;
                sh.tw = t;
                sh.teams = bwd ? c : 1;
                sh.per_sm = bwd ? 1 : c;
            }
        }
    } else {
        if (bwd) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&sh.per_sm, k_soft<true, CAT>, SOFT_W * 32, smem);
        else cudaOccupancyMaxActiveBlocksPerMultiprocessor(&sh.per_sm, k_soft<false, CAT>, SOFT_W * 32, smem);
    }
    sh.per_sm = std::max(1, sh.per_sm);
    return sh;
}

// One persistent wave of the soft kernel: the staged-tile form or the per-warp form, forward only
// or forward + adjoint, with or without membership conditions (CAT).
template <bool CAT>
static void launch_soft_kernel(Ctx *ctx, const SoftKArgs &k, bool tiled, bool bwd, int F, size_t smem,
                               size_t per_warp, const SoftShape &sh, cudaStream_t stream)
{
    const int grid = ctx->sm_count * sh.per_sm;
    if (tiled) {
        const size_t smem_tile = soft_team_bytes(sh.tw, per_warp, F) * sh.teams;
        if (bwd) k_soft_tile<true, CAT><<<grid, sh.tw * sh.teams * 32, smem_tile, stream>>>(k, F);
        else k_soft_tile<false, CAT><<<grid, sh.tw * sh.teams * 32, smem_tile, stream>>>(k, F);
    } else {
        if (bwd) k_soft<true, CAT><<<grid, SOFT_W * 32, smem, stream>>>(k);
        else k_soft<false, CAT><<<grid, SOFT_W * 32, smem, stream>>>(k);
    }
}

// The float-float pass: as many CTAs as the SMs hold, or as there are tasks. The largest sets fit.
static_assert(sizeof(float) * soft_ff_floats(SOFT_MAX_RULES, SOFT_MAX_CONDS, false) * FF_W <= SMEM_CTA - SOFT_TILE_STATIC &&
              sizeof(float) * soft_ff_floats(SOFT_MAX_RULES, SOFT_MAX_CONDS, true) * FF_W_PROBS <= SMEM_CTA - SOFT_TILE_STATIC);
template <bool BWD, bool CAT>
static void launch_soft_ff(Ctx *ctx, const SoftKArgs &k, cudaStream_t stream)
{
    const int W = k.probs ? FF_W_PROBS : FF_W;
    const size_t smem = sizeof(float) * soft_ff_floats(k.maxR, k.maxC, k.probs != nullptr) * W;
    static std::atomic<uint64_t> asked{0};
    const int resident = std::max(1, resident_ctas(asked, k_soft_ff<BWD, CAT>, W * 32, smem));
    const int64_t grid = std::min<int64_t>((int64_t)k.P * k.nchunks, (int64_t)ctx->sm_count * resident);
    k_soft_ff<BWD, CAT><<<(unsigned)grid, W * 32, smem, stream>>>(k);
}

// Words of the float-float group bits for P sets over N samples, for any chunking of at most
// SOFT_MAX_CHUNKS chunks: chunks x ceil(groups per chunk / 32) <= N / 2048 + 2 * SOFT_MAX_CHUNKS.
static size_t ff_words(int P, int64_t N)
{
    return (size_t)P * (size_t)(N / 2048 + 2 * SOFT_MAX_CHUNKS + 1);
}

// Scratch layout of one soft call: records [C], order [P], per-chunk losses [chunks][P], the work
// counter and maxima [4], per-chunk gradient sums [chunks][C] twice (adjoint only), the tasks'
// float-float list [chunks * P] and group bits.
struct SoftScratchLayout {
    size_t recs, order, part_loss, next, part_ga, part_gbt, fflist, ffbits, total;
};

static SoftScratchLayout soft_layout(int64_t C, int P, int nchunks, bool bwd, int64_t N)
{
    auto up = [](size_t x) { return (x + 255) / 256 * 256; };
    SoftScratchLayout L{};
    size_t o = 0;
    L.recs = o; o += up(sizeof(SoftRec) * (size_t)C);
    L.order = o; o += up(sizeof(int32_t) * (size_t)P);
    L.part_loss = o; o += up(sizeof(float) * (size_t)nchunks * P);
    L.next = o; o += 256;
    L.part_ga = o; o += bwd ? up(sizeof(float) * (size_t)nchunks * C) : 0;
    L.part_gbt = o; o += bwd ? up(sizeof(float) * (size_t)nchunks * C) : 0;
    L.fflist = o; o += up(sizeof(int32_t) * (size_t)nchunks * P);
    L.ffbits = o; o += up(sizeof(uint32_t) * ff_words(P, N));
    L.total = o;
    return L;
}

size_t soft_scratch_bytes(int64_t cap_c, int cap_p, int64_t N)
{
    return soft_layout(std::max<int64_t>(cap_c, 1), std::max(cap_p, 1), SOFT_MAX_CHUNKS, true, N).total;
}

// `repeat`: a later step on the caller's scratch over the same structure as the step before it
// (only coefficients and thresholds changed), whose validation and set order still stand.
static rs_status soft_run(Ctx *ctx, const SoftArgs &s, int known_maxR, int known_maxC, cudaStream_t stream,
                          char *pre = nullptr, bool repeat = false, const SoftAdam *adam = nullptr)
{
    const BatchDev &b = s.b;
    const int P = b.P;
    const int64_t Ccap = std::max<int64_t>(b.C, 1);     // capacity when sizes are device-side
    if (P == 0) return RS_OK;
    // Sample chunks: about 1024 samples each, and for small problems as many as it takes to give
    // every SM some 64 (set, chunk) items, down to one 64-sample group per chunk. The chunking is
    // a function of (N, P, SM count) only, so repeated calls sum in the same order.
    const int64_t groups = (s.N + SOFT_G - 1) / SOFT_G;
    const int64_t want = std::max<int64_t>((s.N + 1023) / 1024, ((int64_t)ctx->sm_count * 64 + P - 1) / P);
    int nchunks = (int)std::min<int64_t>(std::min<int64_t>(SOFT_MAX_CHUNKS, groups), want);
    if (nchunks < 1) nchunks = 1;
    int64_t chunk = (s.N + nchunks - 1) / nchunks;
    chunk = (chunk + SOFT_G - 1) / SOFT_G * SOFT_G;
    nchunks = (int)((s.N + chunk - 1) / chunk);

    SoftRec *recs = nullptr;
    float *part_loss = nullptr, *part_ga = nullptr, *part_gbt = nullptr;
    int32_t *next = nullptr;   // the call's counters (SOFT_NEXT_*)
    int32_t *order = nullptr;
    int32_t *fflist = nullptr;
    uint32_t *ffbits = nullptr;
    const bool bwd = s.dloss != nullptr;
    cudaError_t ae = cudaSuccess;
    if (pre) {                       // the caller's scratch, laid out for at most SOFT_MAX_CHUNKS chunks
        const SoftScratchLayout L = soft_layout(Ccap, P, SOFT_MAX_CHUNKS, bwd, s.N);
        recs = reinterpret_cast<SoftRec *>(pre + L.recs);
        order = reinterpret_cast<int32_t *>(pre + L.order);
        part_loss = reinterpret_cast<float *>(pre + L.part_loss);
        next = reinterpret_cast<int32_t *>(pre + L.next);
        part_ga = bwd ? reinterpret_cast<float *>(pre + L.part_ga) : nullptr;
        part_gbt = bwd ? reinterpret_cast<float *>(pre + L.part_gbt) : nullptr;
        fflist = reinterpret_cast<int32_t *>(pre + L.fflist);
        ffbits = reinterpret_cast<uint32_t *>(pre + L.ffbits);
    } else {
        ae = dev_alloc_async(&recs, sizeof(SoftRec) * Ccap, stream);
        if (ae == cudaSuccess) ae = dev_alloc_async(&order, sizeof(int32_t) * (size_t)P, stream);
        if (ae == cudaSuccess) ae = dev_alloc_async(&part_loss, sizeof(float) * (size_t)nchunks * P, stream);
        if (ae == cudaSuccess) ae = dev_alloc_async(&next, sizeof(int32_t) * SOFT_NEXT_N, stream);
        if (ae == cudaSuccess && bwd) ae = dev_alloc_async(&part_ga, sizeof(float) * (size_t)nchunks * Ccap, stream);
        if (ae == cudaSuccess && bwd) ae = dev_alloc_async(&part_gbt, sizeof(float) * (size_t)nchunks * Ccap, stream);
        if (ae == cudaSuccess) ae = dev_alloc_async(&fflist, sizeof(int32_t) * (size_t)nchunks * P, stream);
        if (ae == cudaSuccess) ae = dev_alloc_async(&ffbits, sizeof(uint32_t) * ff_words(P, s.N), stream);
    }
    if (ae != cudaSuccess) {         // release what was taken before the failure
        for (void *q : {(void *)recs, (void *)order, (void *)part_loss, (void *)next, (void *)part_ga, (void *)part_gbt,
                        (void *)fflist, (void *)ffbits})
            if (q) cudaFreeAsync(q, stream);
        return cuda_fail(ae, "soft scratch");
    }
    const bool known = known_maxR > 0;
    repeat = repeat && pre && known;
    if (!repeat) RS_CUDA(cudaMemsetAsync(next, 0, sizeof(int32_t) * SOFT_NEXT_N, stream));
    const int set_blocks = repeat ? 0 : soft_set_blocks(P);
    k_soft_prep<<<set_blocks + (unsigned)((Ccap + SOFT_PREP_BLOCK - 1) / SOFT_PREP_BLOCK), SOFT_PREP_BLOCK, 0, stream>>>(
        b, s.F, s.K, recs, s.status, next, next + 1, known ? known_maxR : SOFT_MAX_RULES,
        known ? known_maxC : SOFT_MAX_CONDS, set_blocks);
    count_launch(ctx);
    if (!repeat) {
        k_soft_order<<<1, 1024, 0, stream>>>(b, order);
        count_launch(ctx);
    }
    SoftKArgs k{};
    k.recs = recs;
    k.set_rule_off = b.set_rule_off;
    k.rule_cond_off = b.rule_cond_off;
    k.rule_class = b.rule_class;
    k.set_default = b.set_default;
    k.P = P;
    k.Xt = s.Xt;
    k.y = s.y;
    k.perm = s.perm;
    k.N = s.N;
    k.n_pad = s.n_pad;
    k.K = s.K;
    k.inv_tau = 1.0f / s.tau;
    k.inv_tau_lo = (float)(1.0 / (double)s.tau - (double)k.inv_tau);
    k.nchunks = nchunks;
    k.chunk = (int32_t)chunk;
    k.part_loss = part_loss;
    k.part_ga = part_ga;
    k.part_gbt = part_gbt;
    k.order = order;
    k.fflist = fflist;
    k.ffbits = ffbits;
    k.probs = s.probs;
    k.next = next;
    k.Ccap = Ccap;
    k.status = s.status;
    rs_status rc = RS_OK;
    if (known) {
        k.maxR = known_maxR;
        k.maxC = known_maxC;
    } else {
        // validation must finish before the launch is sized: read the status and the maxima
        uint32_t *hs = host_status_slot();
        if (!hs) return RS_ERR_OOM;
        RS_CUDA(cudaMemcpyAsync(hs, s.status, sizeof(uint32_t), cudaMemcpyDeviceToHost, stream));
        RS_CUDA(cudaMemcpyAsync(hs + 1, next + 1, sizeof(int32_t) * 2, cudaMemcpyDeviceToHost, stream));
        RS_CUDA(cudaStreamSynchronize(stream));
        k.maxR = std::max<int32_t>(1, (int32_t)hs[1]);
        k.maxC = std::max<int32_t>(1, (int32_t)hs[2]);
        if (*hs) {
            rc = (*hs & ST_TOO_LARGE) ? RS_ERR_TOO_LARGE : RS_ERR_INVALID;
            set_error("soft evaluation rejected the batch: %s", status_text(*hs).c_str());
        }
    }
    k.pslots = k.probs ? std::min(k.K, k.maxR + 1) : 0;
    const size_t smem = soft_main_bytes(k.maxR, k.maxC, bwd, false, k.pslots) * SOFT_W;
    const size_t per_warp = soft_main_bytes(k.maxR, k.maxC, bwd, true, k.pslots);
    // the staged-tile kernel when its smallest per-CTA footprint (and two feature tiles) fits
    const size_t smem_tile = soft_team_bytes(SOFT_TW_MIN, per_warp, s.F);
    const bool tiled = s.F <= 128 && smem_tile + SOFT_TILE_STATIC <= ctx->smem_optin;
    const size_t limit = sizeof(float) * soft_limit_floats(k.maxR, k.maxC, k.probs != nullptr) * SOFT_W;
    if (rc == RS_OK && (smem > ctx->smem_optin || limit > ctx->smem_optin)) {
        rc = RS_ERR_TOO_LARGE;
        set_error("soft evaluation: sets too large for shared memory");
    }
    if (rc == RS_OK) {
        static std::once_flag once;
        std::call_once(once, [&] {
            set_soft_attributes<false>(ctx);
            set_soft_attributes<true>(ctx);
        });
        const SoftShape sh = b.cond_set ? soft_shape<true>(ctx, tiled, bwd, s.F, smem, per_warp, P, k.maxR)
                                        : soft_shape<false>(ctx, tiled, bwd, s.F, smem, per_warp, P, k.maxR);
        if (tiled) {
            // The staged-tile kernel's CTAs take (set group, chunk) tasks until none is left. When
            // the tasks make only a few rounds of the resident CTAs, the last round decides the
            // time: take the chunk count (at most the one chosen above, whose partial sums the
            // scratch holds) that minimises rounds x samples per chunk, preferring more chunks.
            const int64_t set_groups = (P + sh.tw - 1) / sh.tw;
            const int64_t workers = (int64_t)ctx->sm_count * sh.per_sm * sh.teams;
            int64_t best_cost = INT64_MAX;
            for (int n = 1; n <= k.nchunks; ++n) {
                int64_t ch = (s.N + n - 1) / n;
                ch = (ch + SOFT_GT - 1) / SOFT_GT * SOFT_GT;
                const int64_t nc = (s.N + ch - 1) / ch;
                // one round more for the tail: the sets of a group are alike, the groups are not
                const int64_t cost = ((set_groups * nc + workers - 1) / workers + 1) * ch;
                if (cost < best_cost || (cost == best_cost && nc > nchunks)) {
                    best_cost = cost;
                    nchunks = (int)nc;
                    chunk = ch;
                }
            }
            k.nchunks = nchunks;
            k.chunk = (int32_t)chunk;
        }
        k.teams = sh.teams;
        k.tm_cols = (uint32_t)soft_tm_cols(sh.tw * sh.teams, k.maxR);
        k.ff_wpt = (int32_t)(((k.chunk + SOFT_FF_GROUP - 1) / SOFT_FF_GROUP + 31) / 32);
        {
            TimedLaunch tl(ctx, TK_SOFT, stream);
            if (b.cond_set) launch_soft_kernel<true>(ctx, k, tiled, bwd, s.F, smem, per_warp, sh, stream);
            else launch_soft_kernel<false>(ctx, k, tiled, bwd, s.F, smem, per_warp, sh, stream);
        }
        // groups beyond float32's resolution (usually none: the kernel's warps exit at once)
        if (b.cond_set) {
            if (bwd) launch_soft_ff<true, true>(ctx, k, stream);
            else launch_soft_ff<false, true>(ctx, k, stream);
        } else {
            if (bwd) launch_soft_ff<true, false>(ctx, k, stream);
            else launch_soft_ff<false, false>(ctx, k, stream);
        }
        count_launch(ctx);
        if (bwd)                      // the gradients and (when asked) the loss in one launch
            k_soft_reduce_grad<<<P, 128, 0, stream>>>(part_ga, part_gbt, part_loss, nchunks, b.set_rule_off,
                                                     b.rule_cond_off, recs, P, Ccap, s.dloss,
                                                     1.0f / (float)s.N, s.grad_a, s.grad_b, s.grad_t,
                                                     s.loss, adam ? *adam : SoftAdam{}, s.status);
        else
            k_soft_reduce_loss<<<(P + 255) / 256, 256, 0, stream>>>(part_loss, nchunks, P,
                                                                   1.0f / (float)s.N, s.loss, s.status);
        count_launch(ctx, 2);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) rc = cuda_fail(e, "soft kernels");
    }
    if (!pre) {
        cudaFreeAsync(recs, stream);
        cudaFreeAsync(order, stream);
        cudaFreeAsync(part_loss, stream);
        cudaFreeAsync(next, stream);
        if (bwd) { cudaFreeAsync(part_ga, stream); cudaFreeAsync(part_gbt, stream); }
        cudaFreeAsync(fflist, stream);
        cudaFreeAsync(ffbits, stream);
    }
    return rc;
}

// The soft kernels' log1p on [0, 1] (which = 0) or log(1 - e^s) (which = 1) evaluated on the
// device for host inputs (a test hook).
rs_status selftest_soft_math(int which, const float *e_h, int n, float *out_h, cudaStream_t stream)
{
    float *d = nullptr;
    RS_CUDA(dev_alloc_async(&d, sizeof(float) * 2 * (size_t)n, stream));
    rs_status rc = RS_OK;
    cudaError_t e = cudaMemcpyAsync(d, e_h, sizeof(float) * n, cudaMemcpyHostToDevice, stream);
    if (e == cudaSuccess) {
        k_selftest_soft_math<<<std::min((n + 255) / 256, 4096), 256, 0, stream>>>(d, n, d + n, which);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(out_h, d + n, sizeof(float) * n, cudaMemcpyDeviceToHost, stream);
    cudaFreeAsync(d, stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    if (e != cudaSuccess) rc = cuda_fail(e, "soft math self-test");
    return rc;
}

rs_status launch_soft(Ctx *ctx, const SoftArgs &s, cudaStream_t stream)
{
    return soft_run(ctx, s, 0, 0, stream);
}

rs_status soft_step_known(Ctx *ctx, const SoftArgs &a, int maxR, int maxC, cudaStream_t stream)
{
    return soft_run(ctx, a, std::max(1, maxR), std::max(1, maxC), stream);
}

rs_status soft_validate(Ctx *ctx, const SoftArgs &a, int *maxR, int *maxC, cudaStream_t stream)
{
    const BatchDev &b = a.b;
    if (b.P == 0) { *maxR = *maxC = 1; return RS_OK; }
    int32_t *maxima = nullptr;
    RS_CUDA(dev_alloc_async(&maxima, sizeof(int32_t) * 4, stream));
    RS_CUDA(cudaMemsetAsync(maxima, 0, sizeof(int32_t) * 4, stream));
    k_soft_prep<<<soft_set_blocks(b.P), SOFT_PREP_BLOCK, 0, stream>>>(b, a.F, a.K, nullptr, a.status, nullptr, maxima,
                                                                      SOFT_MAX_RULES, SOFT_MAX_CONDS, soft_set_blocks(b.P));
    count_launch(ctx);
    uint32_t *hs = host_status_slot();
    if (!hs) { cudaFreeAsync(maxima, stream); return RS_ERR_OOM; }
    RS_CUDA(cudaMemcpyAsync(hs, a.status, sizeof(uint32_t), cudaMemcpyDeviceToHost, stream));
    RS_CUDA(cudaMemcpyAsync(hs + 1, maxima, sizeof(int32_t) * 2, cudaMemcpyDeviceToHost, stream));
    cudaFreeAsync(maxima, stream);
    RS_CUDA(cudaStreamSynchronize(stream));
    *maxR = std::max<int32_t>(1, (int32_t)hs[1]);
    *maxC = std::max<int32_t>(1, (int32_t)hs[2]);
    if (*hs) {
        set_error("soft evaluation rejected the batch: %s", status_text(*hs).c_str());
        return (*hs & ST_TOO_LARGE) ? RS_ERR_TOO_LARGE : RS_ERR_INVALID;
    }
    return RS_OK;
}

rs_status soft_step_scratch(Ctx *ctx, const SoftArgs &a, int maxR, int maxC, void *scratch, int64_t cap_c,
                            int cap_p, bool repeat, const SoftAdam *adam, cudaStream_t stream)
{
    if (adam && !a.dloss) {
        set_error("soft step: an Adam update needs the adjoint");
        return RS_ERR_INVALID;
    }
    if (!scratch || a.b.P > cap_p || std::max<int64_t>(a.b.C, 1) > std::max<int64_t>(cap_c, 1)) {
        set_error("soft step: scratch smaller than the batch");
        return RS_ERR_INVALID;
    }
    return soft_run(ctx, a, std::max(1, maxR), std::max(1, maxC), stream, static_cast<char *>(scratch), repeat,
                    adam);
}

// Load the kernels of this file now (CUDA loads a kernel lazily at its first launch, which would
// otherwise land on the first request that needs it).
void preload_soft_kernels()
{
    cudaFuncAttributes fa;
    cudaFuncGetAttributes(&fa, k_soft<false, false>);
    cudaFuncGetAttributes(&fa, k_soft<true, false>);
    cudaFuncGetAttributes(&fa, k_soft<false, true>);
    cudaFuncGetAttributes(&fa, k_soft<true, true>);
    cudaFuncGetAttributes(&fa, k_soft_tile<false, false>);
    cudaFuncGetAttributes(&fa, k_soft_tile<true, false>);
    cudaFuncGetAttributes(&fa, k_soft_tile<false, true>);
    cudaFuncGetAttributes(&fa, k_soft_tile<true, true>);
    cudaFuncGetAttributes(&fa, k_soft_ff<false, false>);
    cudaFuncGetAttributes(&fa, k_soft_ff<true, false>);
    cudaFuncGetAttributes(&fa, k_soft_ff<false, true>);
    cudaFuncGetAttributes(&fa, k_soft_ff<true, true>);
    cudaFuncGetAttributes(&fa, k_soft_prep);
    cudaFuncGetAttributes(&fa, k_soft_order);
    cudaFuncGetAttributes(&fa, k_soft_reduce_grad);
    cudaFuncGetAttributes(&fa, k_soft_reduce_loss);
}

}  // namespace rs
