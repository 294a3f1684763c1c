// pairs.cuh -- steps A2-A4 for every (lambda, jhat, k): ratios, exact
// weighted median (Lemma 1) and per-pair residual (Algorithm 1).
//
// Layout: one CTA per (jhat, k-chunk).  Column jhat is staged once in shared
// memory -- x_ijhat, its float reciprocal and its fixed-point weight -- and
// shared by the CTA's warps; each warp owns one k at a time and keeps a small
// histogram of its own.
//
// Per pair the warp never divides per row.  It orders rows by a COARSE key,
// the 32-bit order-preserving image of the ratio rounded to float, and
// approximates it by one multiply, fl(x_ik * fl(1/x_ijhat)) (both rounded to
// float first for double input).  The approximation is within G keys of the
// coarse key of the correctly rounded ratio (G = 8 float, 16 double; the bound
// is derived in the design notes), so a row whose approximate key is more than
// G away from a pivot is classified exactly without dividing; the final <= 31
// candidates are divided exactly and decide the median by exact integer
// arithmetic (the test of Lemma 1).
//
// The selection proper is in select32.cuh (32-bit weights, two passes over
// the rows).  What it cannot settle -- a decision inside the certainty band of the
// 32-bit weights, or more rows around the median than a warp's lanes -- is listed
// for the kernel behind (exact.cuh), which first looks at the coarse keys that the
// selection has left with 64-bit weights (narrow.cuh).  Then the residual sum_i
// |x_ik - v x_ijhat| over all rows (Algorithm 1, objective).
//
// Also listed, for the exact wide-accumulator search: a column whose magnitudes fall
// outside the approximation's range, and a decision that the 64-bit fixed-point
// weights, truncated too, cannot settle.
#pragma once
#include <algorithm>
#include <cmath>

#include "checks.cuh"
#include "common.cuh"

namespace l1l {

__host__ __device__ inline size_t al16(size_t x) { return (x + 15) & ~size_t(15); }

__device__ __forceinline__ uint32_t ckey(float r) { return Traits<float>::key(r); }
// Key of an approximate ratio: -0 is not folded onto +0 (the two keys are
// adjacent, well inside the guard band), which saves two instructions.
__device__ __forceinline__ uint32_t akey(float r) {
    const uint32_t u = __float_as_uint(r);
    return u ^ ((uint32_t)((int32_t)u >> 31) | 0x80000000u);
}

template <typename T> struct Approx;
template <> struct Approx<float> {
    static constexpr uint32_t G = 8;
    static __device__ __forceinline__ float inv_of(float b) { return __frcp_rn(b); }
    static __device__ __forceinline__ uint32_t exact_ck(float a, float b) {
        return ckey(__fdiv_rn(a, b));
    }
};
template <> struct Approx<double> {
    static constexpr uint32_t G = 16;
    static __device__ __forceinline__ float inv_of(double b) {
        return __frcp_rn(__double2float_rn(b));
    }
    static __device__ __forceinline__ uint32_t exact_ck(double a, double b) {
        return ckey(__double2float_rn(__ddiv_rn(a, b)));
    }
};

constexpr int NSAMP = 64;   // weight-proportional sample rows per column
constexpr int HIST_WORDS = 256;  // per-warp histogram

template <typename T> struct PairSmem {
    // per CTA: x_ijhat (T; only when `cs`, else it is read from the column
    // copy in global memory), 1/x_ijhat (float, NaN marks x_ijhat == 0), the
    // 32-bit weights q32_i, the 64 sample rows (uint16)
    __host__ __device__ static size_t col_bytes(int64_t npad, bool cs) {
        return (cs ? al16(npad * sizeof(T)) : 0) + al16(npad * 4) + al16(npad * 4) +
               al16(NSAMP * 2);
    }
    // per warp: the histogram, and room that the planner's shapes were measured with
    // (six bytes for each of `cap` slots; nothing is kept there)
    __host__ __device__ static size_t warp_bytes(int64_t cap) {
        return al16(HIST_WORDS * 4) + al16(cap * 4) + al16(cap * 2);
    }
};

constexpr uint32_t CK0 = 0x80000000u;      // coarse key of 0
constexpr uint32_t CKNONE = 0xFFFFFFFFu;

// ---------------------------------------------------------------------------
// Warp sorts.
// ---------------------------------------------------------------------------
template <typename K, typename W>
__device__ __forceinline__ void warp_sort32(K &key, W &w, int lane) {
#pragma unroll
    for (int size = 2; size <= 32; size <<= 1) {
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            K ok = __shfl_xor_sync(0xFFFFFFFFu, key, stride);
            W ow = __shfl_xor_sync(0xFFFFFFFFu, w, stride);
            bool up = (lane & size) == 0 || size == 32;
            bool lower = (lane & stride) == 0;
            bool take = lower == up ? (ok < key) : (ok > key);
            if (take) {
                key = ok;
                w = ow;
            }
        }
    }
}

template <typename V> __device__ __forceinline__ V warp_scan_add(V x, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        V y = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= o) x += y;
    }
    return x;
}

// Residual over the padded rows: Xt and the staged column are zero past n, so
// a padding row adds |0 - v 0| = 0.  np is a multiple of ROW_PAD.
//   float:  eight rows per lane per step, all eight global loads issued before
//           any is summed, four accumulators (a load issued a step ahead
//           measured slower at low occupancy);
//   double: four rows per lane per step, the next step's loads issued before
//           this step is summed (eight double loads in flight spill at the
//           kernel's register cap).
template <typename T>
__device__ __forceinline__ T warp_residual_pad(const T *__restrict__ xk, const T *__restrict__ xj,
                                               int n, T v, int lane) {
    const int np = (n + ROW_PAD - 1) & ~(ROW_PAD - 1);
    T acc[4] = {T(0), T(0), T(0), T(0)};
    if constexpr (sizeof(T) == 4) {
        constexpr int U = 8;
        static_assert(32 * U == 2 * ROW_PAD, "a step is two row pads");
        int i0 = 0;
        for (; i0 + 32 * U <= np; i0 += 32 * U) {
            T ac[U];
#pragma unroll
            for (int u = 0; u < U; ++u) ac[u] = xk[i0 + u * 32 + lane];
#pragma unroll
            for (int u = 0; u < U; ++u)
                acc[u & 3] += fabs(fma(-v, xj[i0 + u * 32 + lane], ac[u]));
        }
        if (i0 < np) {  // one row pad left
            T ac[U / 2];
#pragma unroll
            for (int u = 0; u < U / 2; ++u) ac[u] = xk[i0 + u * 32 + lane];
#pragma unroll
            for (int u = 0; u < U / 2; ++u) acc[u] += fabs(fma(-v, xj[i0 + u * 32 + lane], ac[u]));
        }
    } else {
        constexpr int U = 4;
        static_assert(U * 32 == ROW_PAD, "one step = one row pad");
        T an[U];
#pragma unroll
        for (int u = 0; u < U; ++u) an[u] = xk[u * 32 + lane];
        for (int i0 = 0; i0 < np; i0 += 32 * U) {
            T ac[U];
#pragma unroll
            for (int u = 0; u < U; ++u) ac[u] = an[u];
            if (i0 + 32 * U < np) {
#pragma unroll
                for (int u = 0; u < U; ++u) an[u] = xk[i0 + 32 * U + u * 32 + lane];
            }
#pragma unroll
            for (int u = 0; u < U; ++u) acc[u] += fabs(fma(-v, xj[i0 + u * 32 + lane], ac[u]));
        }
    }
    T s = (acc[0] + acc[1]) + (acc[2] + acc[3]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
    return s;
}

// Outcomes of a selection.  Every code >= SEL_SLOW hands the pair to the kernel
// behind; the code says why (kept in the slow list).
enum {
    SEL_OK = 0,
    SEL_INTERNAL = 1,
    SEL_SLOW = 2,    // column outside the approximate-key range / forced
    SEL_SLOW_BAND,   // truncated weights cannot settle a decision
    SEL_W64 = 16,    // not settled on 32-bit weights
    SEL_MANY,        // rows too close together for the bins (listed: of a batch of lambdas)
    SEL_BELOW,       // narrow(): the median lies below the range looked at, above it
    SEL_ABOVE
};

__device__ __forceinline__ uint32_t sat_sub(uint32_t a, uint32_t b) { return a > b ? a - b : 0u; }
__device__ __forceinline__ uint32_t sat_add(uint32_t a, uint32_t b) {
    return a < CKNONE - b ? a + b : CKNONE;
}

constexpr uint16_t ROW_MASK = 0x7FFFu;

// The exact test on the 32-bit weights q32 (scale sigma - shift32), with its thresholds
// as whole weights: S passes at a negative ratio when S >= tneg, at a ratio >= 0 when
// S >= tpos (untruncated weights; the search steers by them, the test decides).
//
// The band: of the weights' remainders, R < e in all, S lacks some r of 0 .. R, so the
// true 2S - Q is D + 2r - R, within e of D.  The 64-bit total tells R to within its own
// truncation; a remainder of up to 1 for each row, in S and in Q (Decide), is a band
// three times as wide, and as many more pairs go to the list.
struct Dec32 : Decide {
    uint32_t tneg, tpos;
    float fneg, fpos, Qf;  // for the sample: the same, and Q / 32
    __device__ __forceinline__ void set(const ColInfo &ci, double lambda) {
        // R is less than this
        const int64_t R = ((ci.Q + ci.n_inexact) >> ci.shift32) + 1 - (int64_t)ci.Q32;
        init_at((int64_t)ci.Q32, ci.sigma - ci.shift32, ci.n_inexact32 ? R : 0, lambda);
        auto clamp = [](int64_t x) -> uint32_t {
            return x < 0 ? 0u : (x > 0xFFFFFFFFll ? 0xFFFFFFFFu : (uint32_t)x);
        };
        tneg = clamp(((Q + Lf) >> 1) + 1);
        tpos = clamp(((Q - Lc) >> 1) + 1);
        fneg = (float)tneg;
        fpos = (float)tpos;
        Qf = (float)Q * (1.0f / 32.0f);
    }
    // 1 = true, 0 = false, -1 = undecidable at this precision.
    __device__ __forceinline__ int cond(int64_t S, bool t_nonneg) const {
        int64_t D = 2 * S - Q;
        if (e == 0) return t_nonneg ? (D > -Lc) : (D > Lf);
        if (t_nonneg) {
            if (D - e >= -Lf) return 1;
            if (D + e <= -Lc) return 0;
        } else {
            if (D - e >= Lc) return 1;
            if (D + e <= Lf) return 0;
        }
        return -1;
    }
};

// The lambdas of one launch (or of one instance of a batch).
struct LamView {
    const double *lam;
    int tl_min, tl_max;  // positions of the smallest and largest lambda
};

// What one warp needs to solve the pairs of its CTA's column jhat.
// The fast path's weights are the 32-bit q32 (both input types); s_dec and
// decide_for use the same scale.
template <typename T> struct WarpCtx {
    const T *colb;
    const float *inv;
    const uint32_t *q32;
    uint32_t *hist;       // the warp's histogram
    const Dec32 *s_dec;   // per-lambda thresholds for the first NDEC lambdas
    const ColInfo *ci;    // of column jhat
    int n;
    int d0;               // first-bracket half-width in sample positions
    int srow;             // this lane's sample row and its 1/x_ijhat
    float sinv;
};
constexpr int NDEC = 32;
// Static shared memory of the pair kernels, for the planner: s_dec and the counters.
constexpr int PAIR_STATIC = NDEC * (int)sizeof(Dec32) + 16;

// The place in s_all, whose values are never negative, of a pair that the selection
// has not settled: the sign bit, whether the median lies in the range that follows, among
// few rows or many (or those of a whole batch do), and that range of coarse keys, rounded
// outward to 2 and 4 keys to fit.
enum : int { OFF_NONE = 0, OFF_RANGE, OFF_MANY, OFF_BATCH };
__device__ __forceinline__ int64_t off_mark(int why, uint32_t lo, uint32_t hi) {
    uint64_t range = (uint64_t)(lo >> 1) << 30 | min((hi >> 2) + 1u, (1u << 30) - 1u);
    if (lo > hi) {  // not known
        range = 0;
        if (why != OFF_BATCH) why = OFF_NONE;
    }
    return (int64_t)(1ull << 63 | (uint64_t)why << 61 | range);
}
__device__ __forceinline__ int off_why(int64_t mark) { return (int)((uint64_t)mark >> 61) & 3; }
// Whether it holds a range.
__device__ __forceinline__ bool off_range(int64_t mark, uint32_t &lo, uint32_t &hi) {
    lo = (uint32_t)((uint64_t)mark >> 30 & 0x7FFFFFFFu) << 1;
    hi = ((uint32_t)mark & 0x3FFFFFFFu) << 2;
    return hi != 0;
}

// The coarse key of an exact key.
template <typename T>
__device__ __forceinline__ uint32_t coarse_of(typename Traits<T>::K k) {
    if constexpr (sizeof(T) == 4)
        return k;
    else
        return ckey(__double2float_rn(Traits<T>::value(k)));
}

}  // namespace l1l

#include "select32.cuh"
#include "narrow.cuh"

namespace l1l {

// The exact test of lambda tl on the fast path's weight scale (q32).
template <typename T>
__device__ __forceinline__ Dec32 decide_for(const WarpCtx<T> &w, const LamView &lp, int tl) {
    Dec32 dc;
    if (tl < NDEC)
        dc = w.s_dec[tl];
    else
        dc.set(*w.ci, lp.lam[tl]);
    return dc;
}

// ---------------------------------------------------------------------------
// Residual of a double pair in float-float arithmetic (the double pipe of
// this GPU runs at 1/64 of the float rate; summed in double, the residual's
// two double operations per row made that pipe the bound of the double fit).  Each double x is held as two floats, x1 = fl(x) and
// x2 = fl(x - x1) (the staged copies Xf and Xlo), so |x - x1 - x2| <= u^2|x|
// with u = 2^-24; v likewise.  Per row, with K = |v||x_ijhat|:
//   p1 = fl(v1 b1), e1 = fma(v1, b1, -p1) (exact), c = fma(v1, b2, fma(v2, b1, e1));
//   (s, t) = TwoSum(a1, -p1) (exact), d = fl(fl(a2 - c) + t);
// then s + d = x_ik - v x_ijhat within u^2 (4.04|x_ik| + 15.12 K) + 8 eta
// (eta = 2^-150, the products' underflow), and |s + d| is the pair negated
// when fl(s + d) < 0.  A lane sums its rows in blocks of 8: (H, e) =
// TwoSum(H, s'), L = fl(L + fl(d' + e)), error <= 9.02 u sum|d| + 72.1 u^2
// T_block with |d| <= u (2.04|x_ik| + 4.06 K); each block goes to a double
// accumulator (two roundings of 2^-53 per block), the lanes' sums are added
// in double.  In all, with C_k = sum_i |x_ik|, W = sum_i |x_ijhat|, T the
// exact residual and ldn the padded rows,
//   |T_ff - T| <= E = u^2 (24 C_k + 56 |v| W + (76 + ldn/4096) T) + ldn 2^-146.
// ff_certified accepts T_ff when E (with 77 T_ff in place of 76 T, and C_k, W
// bounded above from the fixed-point column totals) is at most 2^-40 T_ff,
// i.e. a relative error of at most 9.1e-13; any other pair (a near-exact
// fit, v outside [2^-60, 2^60]) is summed again in double.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void ff_row(float a1, float a2, float b1, float b2, float v1, float v2,
                                       float &H, float &L) {
    const float p1 = __fmul_rn(v1, b1);
    const float e1 = __fmaf_rn(v1, b1, -p1);
    const float c = __fmaf_rn(v1, b2, __fmaf_rn(v2, b1, e1));
    const float s = __fsub_rn(a1, p1);
    const float sb = __fsub_rn(s, a1);
    const float t = __fadd_rn(__fsub_rn(a1, __fsub_rn(s, sb)), __fsub_rn(-p1, sb));
    const float d = __fadd_rn(__fsub_rn(a2, c), t);
    // |s + d|: both halves take the sign of fl(s + d)
    const uint32_t sg = __float_as_uint(__fadd_rn(s, d)) & 0x80000000u;
    const float sp = __uint_as_float(__float_as_uint(s) ^ sg);
    const float dp = __uint_as_float(__float_as_uint(d) ^ sg);
    const float h = __fadd_rn(H, sp);
    const float hb = __fsub_rn(h, H);
    const float e = __fadd_rn(__fsub_rn(H, __fsub_rn(h, hb)), __fsub_rn(sp, hb));
    H = h;
    L = __fadd_rn(L, __fadd_rn(dp, e));
}
__device__ __forceinline__ void ff_group(const float4 &a1, const float4 &a2, const float4 &b1,
                                         const float4 &b2, float v1, float v2, float &H, float &L) {
    ff_row(a1.x, a2.x, b1.x, b2.x, v1, v2, H, L);
    ff_row(a1.y, a2.y, b1.y, b2.y, v1, v2, H, L);
    ff_row(a1.z, a2.z, b1.z, b2.z, v1, v2, H, L);
    ff_row(a1.w, a2.w, b1.w, b2.w, v1, v2, H, L);
}
// The sum over the ldn padded rows (zero in both columns past n); a1p, a2p:
// column k's float pair, b1p, b2p: column jhat's.  Every lane returns it.
__device__ __forceinline__ double residual_ff(const float *__restrict__ a1p,
                                              const float *__restrict__ a2p,
                                              const float *__restrict__ b1p,
                                              const float *__restrict__ b2p, int64_t ldn,
                                              float v1, float v2, int lane) {
    const float4 *A1 = reinterpret_cast<const float4 *>(a1p) + lane;
    const float4 *A2 = reinterpret_cast<const float4 *>(a2p) + lane;
    const float4 *B1 = reinterpret_cast<const float4 *>(b1p) + lane;
    const float4 *B2 = reinterpret_cast<const float4 *>(b2p) + lane;
    const int ng = (int)(ldn >> 7);  // 128-row groups; a lane takes 4 rows of each
    const float4 z4 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    double D = 0.0;
    for (int g = 0; g < ng; g += 2) {  // blocks of 8 rows per lane
        // an odd last group is paired with zero rows, which add exactly 0
        const bool two = g + 1 < ng;
        const int o0 = g * 32, o1 = (g + 1) * 32;
        const float4 xa = __ldg(A1 + o0), xb = two ? __ldg(A1 + o1) : z4;
        const float4 la = __ldg(A2 + o0), lb = two ? __ldg(A2 + o1) : z4;
        const float4 ya = __ldg(B1 + o0), yb = two ? __ldg(B1 + o1) : z4;
        const float4 ma = __ldg(B2 + o0), mb = two ? __ldg(B2 + o1) : z4;
        float H = 0.0f, L = 0.0f;
        ff_group(xa, la, ya, ma, v1, v2, H, L);
        ff_group(xb, lb, yb, mb, v1, v2, H, L);
        D = __dadd_rn(D, (double)H);
        D = __dadd_rn(D, (double)L);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) D = __dadd_rn(D, __shfl_xor_sync(0xFFFFFFFFu, D, o));
    return D;
}
// The certificate, divided by 2^-48 and evaluated in float (off the double
// pipe): accept T_ff when
//   24 C_k + 56 |v| W + (77 + ldn/4096) T_ff + ldn 2^-98 <= 256 T_ff,
// with C_k, W rounded up, |v| from its float rounding and both sides given a
// 2^-20 relative margin for the float roundings of this test.  A huge,
// infinite or NaN sum is not accepted.
__device__ __forceinline__ bool ff_certified(double Tff, float Ck, float W, float av,
                                             int64_t ldn) {
    const float T = (float)Tff;
    if (!(T < 0x1p100f)) return false;
    const float ln = (float)ldn;
    const float lhs = 24.0f * Ck + 56.0f * av * W + (77.0f + ln * (1.0f / 4096.0f)) * T +
                      ln * 0x1p-98f;
    return lhs * (1.0f + 0x1p-20f) <= 256.0f * T * (1.0f - 0x1p-20f);
}

// Residual of one pair (CS: x_ijhat staged in shared memory); j, k: the
// pair's columns in a (double input reads their float pairs and totals).
template <typename T, bool CS>
__device__ __forceinline__ T pair_residual(const ScanArgs<T> &a, int64_t j, int64_t k,
                                           const T *xk, const T *colb, int n, T v, int lane) {
    if constexpr (sizeof(T) == 4) {
        (void)a, (void)j, (void)k;
        return warp_residual_f4<CS>(xk, colb, n, v, lane);
    } else {
        // one 128-row group: the double sum's 8 double operations per lane
        // cost less than the float-float sum's fixed part (measured: 100 x 100
        // double fits 30% slower in float-float)
        const ColInfo &ck = a.ci[k], &cj = a.ci[j];
        const float v1 = (float)v;
        const float av = fabsf(v1);
        if (a.ldn > ROW_PAD && ((ck.flags | cj.flags) & COL_WIDE) == 0 &&
            (av == 0.0f || (av >= 0x1p-60f && av <= 0x1p60f))) {
            const float v2 = (float)(v - (double)v1);
            const int64_t ldn = a.ldn, lo = a.m * ldn;  // Xlo follows Xf
            const double Tff = residual_ff(a.Xf + k * ldn, a.Xf + lo + k * ldn, a.Xf + j * ldn,
                                           a.Xf + lo + j * ldn, ldn, v1, v2, lane);
            if (ff_certified(Tff, ck.l1_up, cj.l1_up, av, ldn)) return Tff;
        }
        return warp_residual_pad<T>(xk, colb, n, v, lane);
    }
}

// Writes v and s of (lambda t0+tl, jhat, k), or lists the pair for the exact path.
// VO: the launch may ask for medians only (the float kernels of one or two
// lambdas).
template <typename T, bool CS, bool VO>
__device__ void emit_pair(const ScanArgs<T> &a, int t, int64_t j, int64_t k, int st,
                          typename Traits<T>::K ts, const T *xk, const T *colb, int n,
                          double lam, int lane) {
    using Tr = Traits<T>;
    const int64_t m = a.m;
    const int64_t o = L1L_CHK(((int64_t)t * m + j) * m + k, (int64_t)a.n_lambda * m * m);
    if (st >= SEL_SLOW) {
        if (lane == 0) {
            uint32_t slot = atomicAdd(a.slow_count, 1u);
            SlowEntry e;
            e.t = t;
            e.j = (int32_t)j;
            e.k = (int32_t)k;
            e.inst = (int16_t)a.inst;
            e.reason = (int16_t)st;
            a.slow[slot] = e;
            a.s_all[o] = 0.0;  // no mark of a pair put off
        }
        return;
    }
    if (st == SEL_INTERNAL) {
        if (lane == 0) {
            atomicOr(a.status, ST_INTERNAL);
            a.v_all[o] = T(NAN);
            a.s_all[o] = NAN;
        }
        return;
    }
    const T v = Tr::value(ts);
    const T res = VO && sizeof(T) == 4 && a.v_only
                      ? T(0)
                      : pair_residual<T, CS>(a, j, k, xk, colb, n, v, lane);
    if (lane == 0) {
        a.v_all[o] = v;
        a.s_all[o] = (double)res + lam * (double)fabs(v);
    }
}

// Lists pair (t, j, k), not settled by the selection: `why` SEL_W64, or SEL_MANY for all
// lambdas of the launch.
template <typename T>
__device__ __forceinline__ void list_off(const ScanArgs<T> &a, int t, int64_t j, int64_t k,
                                         int why, int64_t mark, int lane) {
    if (lane == 0) {
        reinterpret_cast<int64_t *>(a.s_all)[((int64_t)t * a.m + j) * a.m + k] = mark;
        a.slow[atomicAdd(a.slow_count, 1u)] =
            SlowEntry{t, (int32_t)j, (int32_t)k, (int16_t)a.inst, (int16_t)why};
    }
}

// One lambda of one pair (valid: x_ijhat != 0 somewhere; batch: one of several, whose
// ties are settled together: the mark of that in whole).  What the selection cannot
// settle is listed: with a call here, what lived across it was spilled in the hot
// loop, and a pair that takes several times as long as the others held up its CTA
// (2000 x 2000 float 11.1 ms with the fallback in this place, 10.5 without).  Returns
// whether the batch is listed.
template <typename T, bool CS, bool VO>
__device__ __forceinline__ bool solve_one(const ScanArgs<T> &a, const LamView &lp, int t0, int tl,
                                          int64_t j, int64_t k, const T *xk, const float *xf,
                                          const WarpCtx<T> &w, bool slow_pair, bool valid,
                                          bool batch, int64_t whole, int lane) {
    using Tr = Traits<T>;
    typename Tr::K ts = Tr::KEY0;
    int st = SEL_OK;
    if (slow_pair) {
        st = SEL_SLOW;
    } else if (valid) {
        int64_t mark = 0;
        const int sel = select_w32<T>(xf, xk, w, decide_for(w, lp, tl), ts, mark, lane);
        if (sel != SEL_OK) {
            const bool all = batch && sel == SEL_MANY;
            list_off(a, t0 + tl, j, k, all ? SEL_MANY : SEL_W64, all ? whole : mark, lane);
            return all;
        }
    }
    emit_pair<T, CS, VO>(a, t0 + tl, j, k, st, ts, xk, w.colb, w.n, lp.lam[tl], lane);
    return false;
}

// A batch of lambdas against candidates between two penalties' medians: lane l holds
// the weight P up to its key fk, ascending; `last`: the lanes that end a run of equal
// keys, `nonneg`: those with a key >= 0; L, after_zero: the weight below them and
// whether the penalty point lies there.
template <typename T> struct LamCand {
    typename Traits<T>::K fk;
    int64_t P, L;
    unsigned last, nonneg;
    bool after_zero;
    __device__ __forceinline__ void init(typename Traits<T>::K key, int64_t fq, int64_t below,
                                         bool zero_below, int lane) {
        using Tr = Traits<T>;
        fk = key;
        warp_sort32(fk, fq, lane);
        P = below + warp_scan_add(fq, lane);
        const typename Tr::K nxt = __shfl_down_sync(0xFFFFFFFFu, fk, 1);
        // the last candidate of each key holds the weight up to it
        last = __ballot_sync(0xFFFFFFFFu, fk != Tr::NONE && (lane == 31 || nxt != fk));
        nonneg = __ballot_sync(0xFFFFFFFFu, fk >= Tr::KEY0);
        L = below;
        after_zero = zero_below;
    }
};

// The lambdas of the lanes with `on`, one per lane (t: of the call; lam, dc: its value
// and test), each against every candidate in turn; the residual is summed once per value
// that any of them takes.  Writes what they decide and returns those lanes; for the
// others they are undecided, or none passes.
template <typename T, bool CS, typename D>
__device__ __forceinline__ unsigned lambda_decide(const ScanArgs<T> &a, const LamCand<T> &f,
                                                  const D &dc, int t, double lam, bool on,
                                                  int64_t j, int64_t k,
                                                  const T *__restrict__ xk, const T *colb, int n,
                                                  int lane) {
    using Tr = Traits<T>;
    const unsigned FULL = 0xFFFFFFFFu;
    int first = -1, res = 0;
    const int below = dc.cond(f.L, f.after_zero);
    for (unsigned c = f.last; c; c &= c - 1) {
        const int u = __ffs(c) - 1;
        const int r = dc.cond(__shfl_sync(FULL, f.P, u), (f.nonneg >> u) & 1u);
        if (first < 0 && r != 0) {
            first = u;
            res = r;
        }
    }
    const bool ok = on && first >= 0 && res == 1 && below == 0;
    const T v = Tr::value(__shfl_sync(FULL, f.fk, max(first, 0)));
    T r = T(0);
    const unsigned done = __ballot_sync(FULL, ok);
    for (unsigned todo = done; todo;) {
        const int src = __ffs(todo) - 1;
        const T vs = __shfl_sync(FULL, v, src);
        const int u = __shfl_sync(FULL, first, src);
        const T rs = pair_residual<T, CS>(a, j, k, xk, colb, n, vs, lane);
        if (first == u) r = rs;
        todo &= ~__ballot_sync(FULL, first == u);
    }
    if (ok) {
        const int64_t o = L1L_CHK(((int64_t)t * a.m + j) * a.m + k,
                                  (int64_t)a.n_lambda * a.m * a.m);
        a.v_all[o] = v;
        a.s_all[o] = (double)r + lam * (double)fabs(v);
    }
    return done;
}

// Lambda batch (step A7).  The weighted median moves monotonically toward 0
// as lambda grows (the penalty point only gains weight), so every lambda's
// median lies between those of the smallest and the largest lambda: one
// selection brackets both, and one sort and prefix scan of the candidates
// between them serve every lambda, 32 at a time.  (Deciding one lambda at a time
// by the whole warp took half of the kernel at 32 lambdas: 1000 x 500 float 2.53 ->
// 1.39 ms; 30 x 100 x 100 double with 8 lambdas 1.09 -> 0.79 ms.)  Returns SEL_OK, or
// why not all of them are settled and, where known, the range of their medians.
template <typename T, bool CS>
__device__ __forceinline__ int lambda_whole(const ScanArgs<T> &a, const LamView &lp, int t0,
                                             int nlc, int64_t j, int64_t k,
                                             const T *__restrict__ xk,
                                             const float *__restrict__ xf, const WarpCtx<T> &w,
                                             uint32_t &lo, uint32_t &hi, int lane) {
    Cand32<T> f;
    f.lo = 1;
    f.hi = 0;
    int st = candidates32<T, true>(xf, xk, w, decide_for(w, lp, lp.tl_min),
                                         decide_for(w, lp, lp.tl_max), f, lane);
    if (st == SEL_OK) {
        LamCand<T> c;
        c.init(f.fk, (int64_t)f.fq, f.L, f.lo > CK0, lane);
        for (int cb = 0; cb < nlc; cb += 32) {
            const bool on = cb + lane < nlc;
            const int tl = on ? cb + lane : 0;
            if (lambda_decide<T, CS>(a, c, decide_for(w, lp, tl), t0 + tl, lp.lam[tl], on, j, k,
                                     xk, w.colb, w.n, lane) != __ballot_sync(0xFFFFFFFFu, on))
                st = SEL_W64;
        }
    }
    lo = f.lo;
    hi = f.hi;
    return st;
}

// The batch in parts, where the whole has more than 31 rows between its medians or a
// bracket fails: runs of neighbouring lambdas, halved until a run's rows fit; their
// candidates serve whatever other lambda they decide.  One by one left a CTA's 16 warps
// waiting for the one with such a pair: 1000 x 500 float with 32 lambdas 1.41 -> 1.29 ms;
// in a kernel of its own, so that the first attempt's does not spill, 1.03 ms.  From
// RUN_MIN lambdas on; fewer are taken one by one at once.
constexpr int RUN_MIN = 16;
template <typename T, bool CS>
__device__ void lambda_parts(const ScanArgs<T> &a, const LamView &lp, int t0, int nlc, int64_t j,
                             int64_t k, const T *xk, const float *xf, const WarpCtx<T> &w,
                             int64_t whole, int lane) {
    const unsigned FULL = 0xFFFFFFFFu;
    int tb = -32, cnt = 0;    // the lambdas tb .. tb + cnt, one per lane,
    unsigned left = 0;        // those of them still to do,
    int rank = 0, len = 1;    // this lane's place by size, and the run's length
    for (;;) {
        if (left == 0) {  // the next 32, ranked
            tb += 32;
            if (tb >= nlc) return;
            cnt = min(32, nlc - tb);
            left = FULL >> (32 - cnt);
            const double mine = lane < cnt ? lp.lam[tb + lane] : INFINITY;
            rank = 0;
            for (int u = 0; u < cnt; ++u) {
                const double o = __shfl_sync(FULL, mine, u);
                rank += o < mine || (o == mine && u < lane) ? 1 : 0;
            }
            if (lane >= cnt) rank = lane;
            len = nlc <= 32 ? (cnt + 1) / 2 : cnt;  // all of them just failed
        }
        const bool mine = (left >> lane) & 1u;
        const int r0 = __reduce_min_sync(FULL, mine ? rank : 32);
        const unsigned part = __ballot_sync(FULL, mine && rank < r0 + len);
        const int r1 = __reduce_max_sync(FULL, (part >> lane) & 1u ? rank : 0);
        const int t1 = tb + __ffs(__ballot_sync(FULL, rank == r0)) - 1;
        const int t2 = tb + __ffs(__ballot_sync(FULL, rank == r1)) - 1;
        Cand32<T> f;
        const int st = candidates32<T, true>(xf, xk, w, decide_for(w, lp, t1),
                                             decide_for(w, lp, t2), f, lane, t1 == t2);
        __syncwarp();
        if (st == SEL_MANY) {
            list_off(a, t0 + t1, j, k, SEL_MANY, whole, lane);
            return;
        }
        if (st != SEL_OK && len > 1) {
            len = len > 2 ? (len + 1) / 2 : 1;
            continue;
        }
        unsigned ok = 0;
        if (st == SEL_OK) {
            LamCand<T> c;
            c.init(f.fk, (int64_t)f.fq, f.L, f.lo > CK0, lane);
            const int tl = mine ? tb + lane : 0;
            ok = lambda_decide<T, CS>(a, c, decide_for(w, lp, tl), t0 + tl, lp.lam[tl], mine, j,
                                      k, xk, w.colb, w.n, lane);
        }
        left &= ~(ok | part);
        for (unsigned rest = part & ~ok; rest; rest &= rest - 1) {  // undecided: each by itself
            if (solve_one<T, CS, false>(a, lp, t0, tb + __ffs(rest) - 1, j, k, xk, xf, w, false,
                                        true, true, whole, lane))
                return;
            __syncwarp();
        }
        __syncwarp();
    }
}

// One work unit: column jhat = j of an instance and the k in [k0, k1), all
// lambdas of the launch.  Called by every thread of a CTA; `smem` is laid out
// for lay_npad rows (column arrays, then one histogram per warp).  CS:
// x_ijhat is staged in shared memory; otherwise the warps read it from the
// column copy in global memory (L2-resident), which frees shared memory for
// more resident warps when n is large.
// What a unit is: the lambdas one by one; as a batch; the batches put off by that (where
// `parts` says that such units follow).
enum : int { UNIT_ONE, UNIT_BATCH, UNIT_PARTS };
template <typename T, int WHAT, bool CS>
__device__ void pairs_unit(const ScanArgs<T> &a, const LamView &lp, int t0, int nlc, int j,
                           int64_t k0, int64_t k1, int cap, int lay_npad, bool parts,
                           unsigned char *smem, Dec32 *s_dec) {
    const int n = (int)a.n;
    const int64_t m = a.m, ldn = a.ldn;
    const int npad = lay_npad;  // shared-memory layout stride (>= n rounded up to 32)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;

    auto mark_of = [&](int64_t k) -> int64_t {
        const int64_t o = L1L_CHK(((int64_t)t0 * m + j) * m + k, (int64_t)a.n_lambda * m * m);
        // k = jhat: s is lambda, which may be -0
        return k == j ? 0 : reinterpret_cast<const int64_t *>(a.s_all)[o];
    };
    auto put_off = [](int64_t mark) { return mark < 0 && off_why(mark) == OFF_BATCH; };
    if (WHAT == UNIT_PARTS) {
        int any = 0;
        for (int64_t k = k0 + threadIdx.x; k < k1; k += blockDim.x) any |= put_off(mark_of(k));
        if (!__syncthreads_or(any)) return;
    }
    const T *xj = a.Xt + (int64_t)j * ldn;
    T *colb_s = reinterpret_cast<T *>(smem);
    const T *colb = CS ? colb_s : xj;
    size_t off = CS ? al16((size_t)npad * sizeof(T)) : 0;
    float *inv = reinterpret_cast<float *>(smem + off);
    off += al16((size_t)npad * 4);
    // fast-path weights: 32-bit q32_i
    uint32_t *q32 = reinterpret_cast<uint32_t *>(smem + off);
    off += al16((size_t)npad * 4);
    uint16_t *samp = reinterpret_cast<uint16_t *>(smem + off);
    unsigned char *wbase =
        smem + PairSmem<T>::col_bytes(npad, CS) + (size_t)warp * PairSmem<T>::warp_bytes(cap);
    uint32_t *hist = reinterpret_cast<uint32_t *>(wbase);
    // prologue scratch: the first 256 bytes of warp 0's histogram
    long long *s_wsum = reinterpret_cast<long long *>(smem + PairSmem<T>::col_bytes(npad, CS));

    const ColInfo cinfo = a.ci[j];
    for (int i = threadIdx.x; i < npad; i += blockDim.x) {
        const T b = i < n ? xj[i] : T(0);
        if (CS) colb_s[i] = b;
        // rows with x_ijhat = 0 (and padding rows) get a NaN reciprocal: their
        // approximate key is the NaN key CKNONE, above every bracket (bounds
        // stop at CKMAX), so the passes need no validity test.  Their
        // weight is 0, so even a NaN of the other sign (a key near 0) could
        // only add zero-weight candidates, which never decide the median.
        inv[i] = b != T(0) ? Approx<T>::inv_of(b) : __int_as_float(0x7FFFFFFF);
        int e = 0;
        const int64_t qi = b != T(0) ? fixq(b < T(0) ? -b : b, cinfo.sigma, e) : 0;
        q32[i] = (uint32_t)((uint64_t)qi >> cinfo.shift32);
    }
    for (int q = threadIdx.x; q < NSAMP; q += blockDim.x) samp[q] = 0;  // always a valid row
    __syncthreads();
    // Systematic weight-proportional sample of the rows of column jhat: sample
    // s is the row whose cumulative weight interval contains (s + 1/2) Q / 64.
    if (cinfo.n_valid > 0) {
        const int nt = blockDim.x;
        const int chunk = (n + nt - 1) / nt;
        const int r0 = min(n, threadIdx.x * chunk), r1 = min(n, r0 + chunk);
        auto wq = [&](int r) -> long long { return (long long)q32[r]; };
        long long mine = 0;
        for (int r = r0; r < r1; ++r) mine += wq(r);
        long long incl = warp_scan_add(mine, lane);
        if (lane == 31) s_wsum[warp] = incl;
        __syncthreads();
        long long before = incl - mine;
        for (int w = 0; w < warp; ++w) before += s_wsum[w];
        const double per = (double)NSAMP / (double)cinfo.Q32;
        for (int r = r0; r < r1; ++r) {
            const long long after = before + wq(r);
            const double x0 = (double)before * per - 0.5, x1 = (double)after * per - 0.5;
            int s0 = (int)floor(x0) + 1, s1 = (int)floor(x1);
            s0 = max(s0, 0);
            s1 = min(s1, NSAMP - 1);
            for (int sidx = s0; sidx <= s1; ++sidx) samp[L1L_CHK(sidx, NSAMP)] = (uint16_t)r;
            before = after;
        }
        __syncthreads();
    }
    // per-lambda thresholds of the exact test depend on (jhat, lambda) only
    for (int tl = threadIdx.x; tl < min(nlc, NDEC); tl += blockDim.x)
        s_dec[tl].set(cinfo, lp.lam[tl]);
    __shared__ int s_knext;  // next k of this unit (offset from k0)
    if (threadIdx.x == 0) s_knext = 0;
    __syncthreads();
    WarpCtx<T> wc;
    wc.colb = colb;
    wc.inv = inv;
    wc.q32 = q32;
    wc.hist = hist;
    wc.srow = L1L_CHK((int)samp[2 * lane + 1], npad);
    wc.sinv = inv[wc.srow];
    wc.s_dec = s_dec;
    wc.ci = a.ci + j;
    wc.d0 = a.d0;
    wc.n = n;

    const bool jwide = (cinfo.flags & COL_WIDE) != 0;
    // a warp takes the next k when it is done with its pair: pairs cost
    // different times (bracket misses), and a fixed share per warp
    // leaves the CTA waiting for its slowest warp
    for (;;) {
        int idx = 0;
        if (lane == 0) idx = atomicAdd(&s_knext, 1);
        const int64_t k = k0 + __shfl_sync(0xFFFFFFFFu, idx, 0);
        if (k >= k1) break;
        const T *xk = a.Xt + k * ldn;
        const float *xf = a.Xf + k * ldn;
        if constexpr (WHAT == UNIT_PARTS) {
            const int64_t mark = mark_of(k);
            if (put_off(mark)) lambda_parts<T, CS>(a, lp, t0, nlc, j, k, xk, xf, wc, mark, lane);
            __syncwarp();
            continue;
        }
        if (k == j) {  // v_jhat = 1: zero residual, penalty lambda * 1
            for (int tl = lane; tl < nlc; tl += 32) {
                int64_t o = L1L_CHK(((int64_t)(t0 + tl) * m + j) * m + k,
                                    (int64_t)a.n_lambda * m * m);
                a.v_all[o] = T(1);
                a.s_all[o] = lp.lam[tl];
            }
            continue;
        }
        const bool slow_pair = a.force_exact || jwide ||
                               (sizeof(T) == 8 && (a.ci[k].flags & COL_WIDE));
        const bool batch = WHAT != UNIT_ONE && nlc >= 3 && !slow_pair && cinfo.n_valid > 0;
        int64_t whole = 0;
        if (batch) {
            uint32_t lo, hi;
            const int st = lambda_whole<T, CS>(a, lp, t0, nlc, j, k, xk, xf, wc, lo, hi, lane);
            if (st == SEL_OK) continue;
            whole = off_mark(OFF_BATCH, lo, hi);
            if (st == SEL_MANY) {
                list_off(a, t0, j, k, SEL_MANY, whole, lane);
                continue;
            }
            if (parts && nlc >= RUN_MIN) {
                if (lane == 0) {
                    reinterpret_cast<int64_t *>(a.s_all)[((int64_t)t0 * m + j) * m + k] = whole;
                    a.slow_count[1] = 1;
                }
                continue;
            }
        }
        for (int tl = 0; tl < nlc; ++tl)
            if (solve_one<T, CS, WHAT == UNIT_ONE>(a, lp, t0, tl, j, k, xk, xf, wc, slow_pair,
                                                   cinfo.n_valid > 0, batch, whole, lane))
                break;
        __syncwarp();
    }
    __syncthreads();  // the CTA may stage another column next
}

}  // namespace l1l
