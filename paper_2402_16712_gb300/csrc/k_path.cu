// k_path.cu -- Algorithm 2: the lambda path of every (jhat, k) pair.
//
// As lambda grows the penalty point at 0 gains weight, so the weighted median
// v_k(lambda) moves monotonically from v0 = v_k(0) to 0 through the distinct
// ratios between them.  For v0 > 0, with S(t) the weight of the rows whose
// ratio is <= t and Q the column's total weight, v_k takes the value t just
// above lambda = Q - 2 S(t) (Algorithm 2's lambda_p at the last row of t's
// run) and reaches 0 above Q - 2 S(0) (its lambda_max); for v0 < 0 it leaves
// t at lambda = 2 S(t) - Q.  So a pair's path needs v0 (the exact lambda = 0
// scan), the rows whose ratio lies between v0 and 0, sorted, and prefix sums
// of their exact fixed-point weights.
//
// Count pass: one warp per pair counts the rows in that range (entries <=
// rows + 1).  A device scan turns the counts into offsets.  Write pass: the
// warp collects the rows (exact keys, row index) into its shared-memory list,
// sorts them, and each run of equal keys writes its entry; pairs with more
// rows than the list holds are queued for a second kernel that does the same
// with a list in global scratch.
//
// Both passes look at a row with one multiply-add and two compares, four rows
// per lane and step: z = x_ik / x_ijhat - c, approximately, tells the rows
// that are certainly below or above the range; the few others (3% of the rows
// at 1000 x 500) are queued and divided 32 at a time.
//
// Residuals R(t) = sum_i |x_ik - t x_ijhat| of the entries: R(0) is column
// k's total, and between 0 and t only the rows of the range change sign, so
//     t > 0:  R(t) = R(0) - 2 B(0, t] + t (2 S(t) - Q)
//     t < 0:  R(t) = R(0) - 2 B(t, 0) + t (2 S(t) - Q)
// with B the sum of |x_ik| over the rows whose ratio lies there.  All of them
// are sums of fixed-point integers (column k's and column jhat's), exact
// whatever the order; what truncation to those drops (double input, and float
// columns that span many binary orders) is summed beside them in float, in units
// of the last place.  (The five double sums over all rows that gave R before made
// the double pipe, two operations per SM and cycle, the bound: 1000 x 500 float
// with residuals, write pass 5.07 -> 0.61 ms.  Without them, 2000 x 400: 1.33 ->
// 0.56 ms; count pass 0.42 -> 0.22 ms.)  The write pass is bound by instructions,
// a quarter of them the rows', the rest the order and the prefix sums of the list.
#include <cmath>
#include <type_traits>

#include "checks.cuh"
#include "common.cuh"
#include "launch.h"
#include "pairs.cuh"

namespace l1l {

namespace {

constexpr int PW = 8;          // warps per CTA
constexpr int PATH_CAP = 256;  // shared-memory list entries per warp
constexpr int PATH_CAP_MIN = 128;  // where the column leaves no room for that
constexpr int PEND = 64;       // rows queued for the exact division, per warp
constexpr int PBUCK = 64;      // buckets of the list's sort
constexpr uint32_t BUCK_MAX = 48;

template <typename T> struct PathArgs {
    const T *Xt;
    const float *Xf;
    const ColInfo *ci;
    int64_t n, m, ldn;
    const T *v0;           // [m][m] lambda = 0 medians
    int64_t *bound;        // count pass: [m*m] entries upper bound
    const int64_t *off;    // write pass: [m*m + 1]
    double *lam;           // write pass outputs
    T *val;
    double *res;           // optional: residual sum_i |x_ik - v x_ijhat| of each entry
    float *crem;           // with residuals: [m] remainder of a column's fixed-point total
    int32_t *len;          // [m*m]
    int32_t *big;          // pairs whose rows exceed the warp list
    uint32_t *big_count;
    uint32_t *big_next;    // work counter of the big-pair kernel
    uint32_t *inexact;     // whether any column's remainders are needed
    unsigned char *scratch;  // big-pair lists, one slice per worker warp
    int64_t slice;         // entries per slice (power of two >= n)
    uint32_t *status;
};

// Classification of one row against the range between 0 and v0 (exclusive
// of 0) by its exact key: -1 below it, 0 inside, +1 above.
template <typename K>
__device__ __forceinline__ int classify(K ke, K kv, K key0, bool pos) {
    if (pos) {  // range (KEY0, kv]
        if (ke <= key0) return -1;
        return ke <= kv ? 0 : 1;
    }
    // range [kv, KEY0)
    if (ke < kv) return -1;
    return ke < key0 ? 0 : 1;
}

// Coarse-key range of (0, v0] or [v0, 0), and its exact upper/lower key.
template <typename T>
__device__ __forceinline__ void range_of(T v0, bool &pos, uint32_t &ck_lo, uint32_t &ck_hi,
                                         typename Traits<T>::K &kv) {
    pos = v0 > T(0);
    kv = Traits<T>::key(v0);
    const uint32_t cv = ckey((float)v0);
    if (pos) {
        ck_lo = CK0;
        ck_hi = cv;
    } else {
        ck_lo = cv;
        ck_hi = CK0;
    }
}

// What fixq(w, sigma) truncates, in units of 2^-sigma (double w; [0, 1)).
__device__ __forceinline__ float fix_rem(double w, int sigma) {
    const uint64_t u = (uint64_t)__double_as_longlong(w) & 0x7FFFFFFFFFFFFFFFull;
    const int be = (int)(u >> 52);
    uint64_t f = u & 0xFFFFFFFFFFFFFull;
    if (be) f |= 0x10000000000000ull;
    const int rs = 1075 - sigma - (be ? be : 1);
    if (rs <= 0 || rs > 120) return 0.0f;
    if (rs < 64) f &= (1ull << rs) - 1ull;
    return (float)f * __int_as_float((127 - rs) << 23);
}

// Whether a column's truncated weights may together lack more than 2^-54 of its
// total, and whether a pair's remainders are summed (the same for the warp).
__device__ __forceinline__ bool lacks(const ColInfo &c) {
    return (int64_t)c.n_inexact > (c.Q >> 54);
}
template <typename T>
__device__ __forceinline__ bool with_rem(const PathArgs<T> &a, const ColInfo &cj,
                                         const ColInfo &ck) {
    return a.res != nullptr && (lacks(cj) || lacks(ck));
}

// The column arrays of jhat: float reciprocal, fixed-point weight, and x
// itself (float input, whose remainders are computed where there are any) or
// the weight's remainder (double input, which reads x from the column copy: a
// few rows per pair).
template <typename T> struct Column {
    const T *x;
    float *inv;
    int64_t *q;
    float *rem;
    int sigma;
    __device__ __forceinline__ float rem_of(int i) const {
        if constexpr (sizeof(T) == 8)
            return rem[i];
        else
            return fix_rem(x[i], sigma);
    }
};

// Stage them by `nt` threads; `own` holds x or the remainders.
template <typename T>
__device__ Column<T> stage_column(const PathArgs<T> &a, int64_t j, float *own, float *inv,
                                  int64_t *colq, int npad, int t, int nt) {
    const ColInfo ci = a.ci[j];
    const T *xj = a.Xt + j * a.ldn;
    for (int i = t; i < npad; i += nt) {
        const T b = i < a.n ? xj[i] : T(0);
        if constexpr (sizeof(T) == 4)
            own[i] = b;
        else
            own[i] = a.res ? fix_rem(b, ci.sigma) : 0.0f;
        // NaN: neither inside, below nor above any range
        inv[i] = b != T(0) ? Approx<T>::inv_of(b) : __int_as_float(0x7FFFFFFF);
        int e = 0;
        colq[i] = b != T(0) ? fixq(b < T(0) ? -b : b, ci.sigma, e) : 0;
    }
    if constexpr (sizeof(T) == 4)
        return Column<T>{own, inv, colq, nullptr, ci.sigma};
    else
        return Column<T>{xj, inv, colq, own, ci.sigma};
}

// Remainder of each column's fixed-point total.
template <typename T> __global__ void __launch_bounds__(256) k_colrem(PathArgs<T> a) {
    __shared__ float sm[8];
    const T *x = a.Xt + (int64_t)blockIdx.x * a.ldn;
    const ColInfo ci = a.ci[blockIdx.x];
    float s = 0.0f;
    if (ci.n_inexact > 0)
        for (int64_t i = threadIdx.x; i < a.n; i += 256) s += fix_rem(x[i], ci.sigma);
    s = warp_sum_f32(s);
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int q = 1; q < 8; ++q) s += sm[q];
        a.crem[blockIdx.x] = s;
        if (lacks(ci)) atomicOr(a.inexact, 1u);
    }
}

// The list's sums of one pair: the weight below the range and (negative ranges)
// the |x_ik| in it, in fixed point and the remainders of both.
struct ListSums {
    int64_t Sbelow, Ball;
    float Srem, Brem;
};

// A warp's sort of its list, as an order: bucket counts and two index arrays
// (the first is the queue while the rows are scanned).
struct SortBuf {
    uint32_t *cnt;      // [PBUCK]
    uint16_t *part, *ord;  // [cap]
};
__host__ __device__ constexpr size_t sort_bytes(int cap) { return PBUCK * 4 + (size_t)cap * 4; }

// ord[i] = list position of the i-th smallest (key, position) of c, by one
// warp: the ratios of a list spread evenly between 0 and v0, so 64 equal steps
// hold a few each, and an entry is ranked within its own.  Returns whether two
// keys are equal, or -1, with no order, when a bucket holds over BUCK_MAX (many
// ties, a range with most ratios in one place): ranking within it would take
// longer than the network.  (A bitonic network: 28 steps of 20 instructions and their
// latencies at 65 to 128 entries; 2000 x 400 write pass 0.70 -> 0.61 ms.
// Ranking up to 64 entries among all instead: 0.87 -> 0.91 ms at 1000 x 500.)
template <typename T>
__device__ int warp_bucket_sort(const typename Traits<T>::K *keys, int c, T v0,
                                 const SortBuf &sb, int lane) {
    using Tr = Traits<T>;
    using K = typename Tr::K;
    const bool pos = v0 > T(0);
    const float scale = (float)PBUCK / fabsf((float)v0);
    auto bucket = [&](K k) -> int {  // monotone in the key
        const int b = min(PBUCK - 1, (int)(fabsf((float)Tr::value(k)) * scale));
        return pos ? b : PBUCK - 1 - b;
    };
    static_assert(PBUCK == 64, "two buckets per lane");
    sb.cnt[lane] = sb.cnt[lane + 32] = 0u;
    __syncwarp();
    for (int e = lane; e < c; e += 32) atomicAdd(&sb.cnt[bucket(keys[e])], 1u);
    __syncwarp();
    const uint32_t c0 = sb.cnt[2 * lane], c1 = sb.cnt[2 * lane + 1];
    if (__reduce_max_sync(0xFFFFFFFFu, max(c0, c1)) > BUCK_MAX) return -1;
    const uint32_t ex = warp_scan_add(c0 + c1, lane) - c0 - c1;
    sb.cnt[2 * lane] = ex;
    sb.cnt[2 * lane + 1] = ex + c0;
    __syncwarp();
    for (int e = lane; e < c; e += 32)
        sb.part[atomicAdd(&sb.cnt[bucket(keys[e])], 1u)] = (uint16_t)e;
    __syncwarp();
    bool ties = false;
    for (int p = lane; p < c; p += 32) {
        const int e = sb.part[p];
        const K k = keys[e];
        const int b = bucket(k);
        const int q0 = b ? (int)sb.cnt[b - 1] : 0, q1 = (int)sb.cnt[b];
        int r = q0;
        for (int q = q0; q < q1; ++q) {
            const int f = sb.part[q];
            const K kf = keys[f];
            r += kf < k || (kf == k && f < e) ? 1 : 0;
            ties |= kf == k && f != e;
        }
        sb.ord[r] = (uint16_t)e;
    }
    __syncwarp();
    return __any_sync(0xFFFFFFFFu, ties) ? 1 : 0;
}

// Warp bitonic sort of (key, row) over P (power of two) entries of a list;
// entries c..P-1 are first filled with NONE.
template <typename K>
__device__ void warp_list_sort(K *keys, uint32_t *rows, int c, int P, int lane) {
    for (int i = c + lane; i < P; i += 32) {
        keys[i] = (K)~(K)0;
        rows[i] = 0;
    }
    __syncwarp();
    for (int size = 2; size <= P; size <<= 1) {
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            for (int t = lane; t < P / 2; t += 32) {
                const int i = 2 * t - (t & (stride - 1));
                const int jx = i + stride;
                const bool up = (i & size) == 0;
                const K ki = keys[i], kj = keys[jx];
                if ((ki > kj) == up) {
                    keys[i] = kj;
                    keys[jx] = ki;
                    const uint32_t r = rows[i];
                    rows[i] = rows[jx];
                    rows[jx] = r;
                }
            }
            __syncwarp();
        }
    }
}

// D 2^-sigma rounded to double, |D| < 2^63.  Normalised, rounded (to nearest,
// ties to even) and scaled in integer instructions: the conversion and the
// scaling on the double pipe (2 results per SM and cycle) cost twice as much.
__device__ __forceinline__ double fix_to_double(int64_t D, int sigma) {
    if (sigma < -900 || sigma > 900) return scalbn((double)D, -sigma);
    const uint64_t u = (uint64_t)(D < 0 ? -D : D);
    const int lz = __clzll((long long)u);
    const uint64_t f = u << (lz & 63);
    uint64_t m = f >> 11;  // 53 bits, the leading one at bit 52
    const uint32_t rest = (uint32_t)f & 0x7FFu;
    m += rest > 0x400u || (rest == 0x400u && (m & 1u)) ? 1u : 0u;
    // the leading bit adds the last 1 to the exponent
    const uint64_t r = ((uint64_t)(1085 - lz - sigma) << 52) + m;
    const uint64_t sg = (uint64_t)D & 0x8000000000000000ull;
    return __longlong_as_double((long long)(u == 0 ? 0ull : (r | sg)));
}

// sum_i |x_i| of a column (rem: of a double column's fixed-point total).
__device__ __forceinline__ double column_total(const ColInfo &c, float rem) {
    const double t = fix_to_double(c.Q, c.sigma);
    return rem == 0.0f ? t : t + scalbn((double)rem, -c.sigma);
}

// Entries of one pair from its in-range list (c > 0 rows); ord: its order, or
// null for a sorted list; ties: whether keys may be equal.
template <typename T, bool REM>
__device__ void emit_path(const PathArgs<T> &a, int64_t p, T v0, bool pos,
                          const typename Traits<T>::K *keys, const uint32_t *rows,
                          const uint16_t *ord, bool ties, int c, const Column<T> &col, const ColInfo &cj, const ColInfo &ck,
                          const ListSums &ls, bool rem_, const T *xk, int lane) {
    using Tr = Traits<T>;
    using K = typename Tr::K;
    // corrections of a run: double input's lie below the fixed point's units
    using QC = typename std::conditional<sizeof(T) == 4, int64_t, float>::type;
    const unsigned FULL = 0xFFFFFFFFu;
    const int64_t Q = cj.Q;
    const bool rem = REM && rem_;
    const float remj = rem ? a.crem[p / a.m] : 0.0f, remk = rem ? a.crem[p % a.m] : 0.0f;
    const int64_t o = a.off[p];
    const int64_t room = a.off[p + 1] - o;  // entries the count pass reserved
    auto at = [&](int i) -> int { return ord ? (int)ord[i] : i; };
    // whether run ends (starts) lie at place i, whose key is ki
    auto ends = [&](int i, K ki) { return i == c - 1 || !ties || ki != keys[at(i + 1)]; };
    auto starts = [&](int i, K ki) { return i == 0 || !ties || ki != keys[at(i - 1)]; };
    // number of runs of equal keys
    int groups = c;
    if (ties) {
        groups = 0;
        for (int i0 = 0; i0 < c; i0 += 32) {
            const int i = i0 + lane;
            groups += __popc(__ballot_sync(FULL, i < c && ends(i, keys[at(i)])));
        }
    }
    // the entries 0 .. groups lie inside the room the count pass reserved
    L1L_CHK((int64_t)groups, room);
    int64_t carry = ls.Sbelow;  // S at the end of the previous chunk
    int64_t cB = 0;          // B of the list up to there
    float cSr = ls.Srem, cBr = 0.0f;  // remainders of both
    QC crun = 0;             // corrections of the run open at the chunk's end
    int gbase = 0;           // runs ended before this chunk
    for (int i0 = 0; i0 < c; i0 += 32) {
        const int i = i0 + lane;
        const int e0 = i < c ? at(i) : 0;
        const uint32_t row = i < c ? rows[e0] : 0u;
        const K ki = keys[e0];
        const int64_t q = i < c ? col.q[row] : 0;
        const int64_t S = carry + warp_scan_add(q, lane);  // S(key_i) at a run end
        const bool end = i < c && ends(i, ki);
        const unsigned em = __ballot_sync(FULL, end);
        const int g = gbase + __popc(em & ((1u << lane) - 1u));  // run index (ascending)
        const int64_t D = 2 * S - Q;
        const double Dd = fix_to_double(D, cj.sigma);
        if (a.res) {
            // The formula counts the rows of t's own run as "ratio <= t"; a
            // row whose exact ratio lies above its rounded value t then enters
            // with the wrong sign, so each row of the run adds the correction
            // |x - t b| - (t |b| - sgn(b) x) = 2 max(sgn(b) x - t |b|, 0).
            int64_t xq = 0;
            QC qc = 0;
            T t = T(0);
            float wr = 0.0f, xr = 0.0f;
            if (i < c) {
                const T b = col.x[row], x = xk[row];
                const T sx = b < T(0) ? -x : x;
                t = Tr::value(ki);
                int e = 0;
                xq = fixq(fabs(x), ck.sigma, e);
                // the remainder of a correctly rounded division is exact in
                // its operands' precision unless it underflows: float rows
                // that small take it in double
                if constexpr (sizeof(T) == 8) {
                    const T d = fma(-t, fabs(b), sx);
                    if (d > T(0)) qc = (float)scalbn(2.0 * d, ck.sigma);
                } else if (fabs(x) >= T(0x1p-100)) {
                    const T d = fma(-t, fabs(b), sx);
                    if (d > T(0)) qc = fixq(T(2) * d, ck.sigma, e);
                } else {
                    const double d = fma(-(double)t, fabs((double)b), (double)sx);
                    if (d > 0.0) qc = fixq(2.0 * d, ck.sigma, e);
                }
                if (rem) {
                    wr = col.rem_of(row);
                    xr = fix_rem(x, ck.sigma);
                }
            }
            float Sr = 0.0f, Br = 0.0f;
            if (rem) {
                Sr = cSr + warp_scan_add(wr, lane);
                Br = cBr + warp_scan_add(xr, lane);
                cSr = __shfl_sync(FULL, Sr, 31);
                cBr = __shfl_sync(FULL, Br, 31);
            }
            const int64_t B = cB + warp_scan_add(xq, lane);
            QC run_q = 0;
            if (!ties) {  // every row is a run
                run_q = qc;
            } else if (__any_sync(FULL, qc != 0) || crun != 0) {
                const QC Qi = warp_scan_add(qc, lane);  // inclusive, this chunk only
                // run sums of qc: the run's start holds the prefix before it
                const bool start = i < c && starts(i, ki);
                const unsigned smk = __ballot_sync(FULL, start);
                const unsigned upto = smk & (lane == 31 ? FULL : ((2u << lane) - 1u));
                const int hs = upto ? 31 - __clz(upto) : -1;
                const QC Qstart = __shfl_sync(FULL, Qi - qc, hs < 0 ? 0 : hs);
                // the run began in an earlier chunk: its corrections are in crun
                run_q = hs >= 0 ? Qi - Qstart : crun + Qi;
            }
            if (end) {  // each run writes the residual of its own entry
                const int slot = pos ? groups - 1 - g : g;
                int64_t F = ck.Q - 2 * (pos ? B : ls.Ball - B);
                if constexpr (sizeof(T) == 4) F += run_q;
                double Ft = fix_to_double(F, ck.sigma), Dt = Dd;
                if (rem) {
                    float fr = remk - 2.0f * (pos ? Br : ls.Brem - Br);
                    if constexpr (sizeof(T) == 8) fr += run_q;
                    Ft += scalbn((double)fr, -ck.sigma);
                    Dt += scalbn((double)(2.0f * Sr - remj), -cj.sigma);
                }
                a.res[o + slot] = fma((double)t, Dt, Ft);
            }
            // the run still open at the end of this chunk carries its partial sum
            crun = __shfl_sync(FULL, run_q, 31);
            cB = __shfl_sync(FULL, B, 31);
        }
        if (end) {
            if (pos) {
                // run g (not the top one) starts at Q - 2 S(t_g), slot groups-1-g
                if (g < groups - 1) {
                    a.lam[o + groups - 1 - g] = D < 0 ? -Dd : 0.0;
                    a.val[o + groups - 1 - g] = Tr::value(ki);
                }
            } else {
                // the run after g starts at 2 S(t_g) - Q; after the last, 0
                a.lam[o + g + 1] = D > 0 ? Dd : 0.0;
                if (g > 0) a.val[o + g] = Tr::value(ki);
            }
        }
        carry = __shfl_sync(FULL, S, 31);
        gbase += __popc(em);
    }
    if (lane == 0) {
        a.lam[o] = 0.0;
        a.val[o] = v0;
        if (pos) {
            const int64_t D = Q - 2 * ls.Sbelow;
            a.lam[o + groups] = D > 0 ? fix_to_double(D, cj.sigma) : 0.0;
        }
        a.val[o + groups] = T(0);
        if (a.res) a.res[o + groups] = column_total(ck, remk);  // v = 0
        a.len[p] = groups + 1;
    }
}

// One pass over the rows of pair (j, k) by one warp; returns the number of
// rows in range.  Unless COUNT: appends them (exact key, row) to the list (at
// most cap; the total is returned either way), sums the exact weight below the
// range and, with residuals, the fixed-point |x_ik| of the range.  The column
// arrays hold a multiple of 128 rows, zero past n.
template <typename T, bool COUNT, bool REM>
__device__ int scan_rows(const PathArgs<T> &a, int64_t k, const Column<T> &col, uint16_t *pend,
                         bool wide, bool rem_, bool pos, uint32_t ck_lo, uint32_t ck_hi,
                         typename Traits<T>::K kv, int sigma_k, typename Traits<T>::K *keys,
                         uint32_t *rows, int cap, ListSums &ls, int lane) {
    using Tr = Traits<T>;
    using K = typename Tr::K;
    constexpr uint32_t G = Approx<T>::G;
    const unsigned FULL = 0xFFFFFFFFu;
    const T *xk = a.Xt + k * a.ldn;
    const float4 *xf = reinterpret_cast<const float4 *>(a.Xf + k * a.ldn);
    const int ng = ((int)a.n + 127) >> 7;
    const bool want_r = !COUNT && a.res != nullptr, rem = REM && rem_;
    // Rows with a coarse key outside [ck_lo - G, ck_hi + G] are certainly
    // below or above; [va, vb] holds the ratios of the others, and |fma(x,
    // inv, -cen)| differs from |fl(x inv) - cen| by at most 3 roundings of
    // 2^-24 of the larger end.  Every row is queued where that means nothing:
    // a wide column, or a range that reaches the infinities.
    const float va = akey_value(sat_sub(ck_lo, G)), vb = akey_value(sat_add(ck_hi, G));
    const float cen = 0.5f * va + 0.5f * vb;
    float delta = (0.5f * vb - 0.5f * va) * (1.0f + 0x1p-20f) +
                  0x1p-21f * fmaxf(fabsf(va), fabsf(vb)) + 0x1p-148f;
    const bool all = wide || !(delta < 0x1p126f) || !(fabsf(cen) < 0x1p126f);
    int c = 0, np = 0;
    int64_t sb = 0, bl = 0;
    float sr = 0.0f, br = 0.0f;  // their remainders
    // the queue's first 32 rows (fewer at the end): exact keys, list append
    auto flush = [&](int cnt) {
        int cls = 1;
        K ke = Tr::NONE;
        const int i = L1L_CHK(lane < cnt ? (int)pend[lane] : 0, ng * 128);
        const T b = col.x[i];
        T x = T(0);
        if (lane < cnt && b != T(0)) {
            x = xk[i];
            ke = Tr::key(Tr::div_rn(x, b));
            cls = classify<K>(ke, kv, Tr::KEY0, pos);
        }
        if (!COUNT && cls < 0) {
            sb += col.q[i];
            if (rem) sr += col.rem_of(i);
        }
        const unsigned im = __ballot_sync(FULL, cls == 0);
        if (!COUNT && cls == 0) {
            const int at = c + __popc(im & ((1u << lane) - 1u));
            if (at < cap) {
                keys[at] = ke;
                rows[at] = (uint32_t)i;
            }
            int e = 0;
            if (want_r && !pos) bl += fixq(fabs(x), sigma_k, e);
            if (rem && !pos) br += fix_rem(x, sigma_k);
        }
        c += __popc(im);
    };
    for (int g0 = 0; g0 < ng; g0 += 8) {  // 8 groups: one byte of flags per row of the lane
        const int ge = min(ng, g0 + 8);
        uint32_t mask = 0;  // bit 4 (g - g0) + u: row u of the lane in group g
        float4 xn = __ldg(xf + g0 * 32 + lane);
        for (int g = g0; g < ge; ++g) {
            const float4 x4 = xn;
            if (g + 1 < ge) xn = __ldg(xf + (g + 1) * 32 + lane);
            const int i = L1L_CHK(g * 128 + 4 * lane, ng * 128);
            const float4 v4 = *reinterpret_cast<const float4 *>(col.inv + i);
            const float z[4] = {fmaf(x4.x, v4.x, -cen), fmaf(x4.y, v4.y, -cen),
                                fmaf(x4.z, v4.z, -cen), fmaf(x4.w, v4.w, -cen)};
            uint32_t f = 0;
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (fabsf(z[u]) < delta) f |= 1u << u;
            if (!COUNT && !all) {
                const longlong2 qa = *reinterpret_cast<const longlong2 *>(col.q + i);
                const longlong2 qb = *reinterpret_cast<const longlong2 *>(col.q + i + 2);
                if (z[0] <= -delta) sb += qa.x;
                if (z[1] <= -delta) sb += qa.y;
                if (z[2] <= -delta) sb += qb.x;
                if (z[3] <= -delta) sb += qb.y;
                if (rem) {
                    if constexpr (sizeof(T) == 8) {
                        const float4 r4 = *reinterpret_cast<const float4 *>(col.rem + i);
                        if (z[0] <= -delta) sr += r4.x;
                        if (z[1] <= -delta) sr += r4.y;
                        if (z[2] <= -delta) sr += r4.z;
                        if (z[3] <= -delta) sr += r4.w;
                    } else {
#pragma unroll 1
                        for (int u = 0; u < 4; ++u)
                            if (fmaf(a.Xf[k * a.ldn + i + u], col.inv[i + u], -cen) <= -delta)
                                sr += col.rem_of(i + u);
                    }
                }
            }
            mask |= f << (4 * (g - g0));
        }
        if (all) mask = ge - g0 == 8 ? FULL : (1u << (4 * (ge - g0))) - 1u;
        unsigned m;
        while ((m = __ballot_sync(FULL, mask != 0)) != 0) {
            if (mask != 0) {
                const int bit = __ffs(mask) - 1;
                mask &= mask - 1;
                const int at = L1L_CHK(np + __popc(m & ((1u << lane) - 1u)), PEND);
                pend[at] = (uint16_t)((g0 + (bit >> 2)) * 128 + 4 * lane + (bit & 3));
            }
            np += __popc(m);
            __syncwarp();
            if (np >= 32) {
                flush(32);
                const uint16_t up = pend[32 + lane];
                __syncwarp();
                pend[lane] = up;
                np -= 32;
                __syncwarp();
            }
        }
    }
    if (np > 0) flush(np);
    if (!COUNT) {
        ls.Sbelow = warp_sum_i64(sb);
        ls.Ball = want_r ? warp_sum_i64(bl) : 0;
        ls.Srem = rem ? warp_sum_f32(sr) : 0.0f;
        ls.Brem = rem ? warp_sum_f32(br) : 0.0f;
    }
    __syncwarp();
    return c;
}

template <typename T>
__device__ __forceinline__ bool pair_is_wide(const PathArgs<T> &a, const ColInfo &cj, int64_t k) {
    return (cj.flags & COL_WIDE) != 0 || (sizeof(T) == 8 && (a.ci[k].flags & COL_WIDE));
}

// REM: with remainders.  They cost a fifth of the write pass in registers even
// where there are none, so with residuals of float input both are launched and
// `inexact` says which of them has the work (USE_FLAG).
template <typename T, bool COUNT, bool REM, bool USE_FLAG>
__global__ void __launch_bounds__(PW * 32, 4) k_path_pass(PathArgs<T> a, int kchunk, int cap) {
    if (USE_FLAG && (*a.inexact != 0) != REM) return;
    using Tr = Traits<T>;
    using K = typename Tr::K;
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int npad = ((int)a.n + ROW_PAD - 1) & ~(ROW_PAD - 1);
    float *own = reinterpret_cast<float *>(smem);
    size_t o = (size_t)npad * 4;
    float *inv = reinterpret_cast<float *>(smem + o);
    o += (size_t)npad * 4;
    int64_t *colq = reinterpret_cast<int64_t *>(smem + o);
    o += (size_t)npad * 8;
    K *keys = reinterpret_cast<K *>(smem + o + (size_t)warp * cap * (sizeof(K) + 4));
    uint32_t *rows = reinterpret_cast<uint32_t *>(keys + cap);
    o += (size_t)PW * cap * (sizeof(K) + 4) + (size_t)warp * sort_bytes(cap);
    SortBuf sb;
    sb.cnt = reinterpret_cast<uint32_t *>(smem + o);
    sb.part = reinterpret_cast<uint16_t *>(smem + o + PBUCK * 4);
    sb.ord = sb.part + cap;
    static_assert(PEND <= PATH_CAP_MIN, "the queue lies in the first index array");
    const int64_t j = blockIdx.x;
    const Column<T> col = stage_column<T>(a, j, own, inv, colq, npad, threadIdx.x, PW * 32);
    __syncthreads();
    const ColInfo cj = a.ci[j];
    const int64_t k0 = (int64_t)blockIdx.y * kchunk, k1 = min(a.m, k0 + kchunk);
    for (int64_t k = k0 + warp; k < k1; k += PW) {
        const int64_t p = j * a.m + k;
        const T v0 = a.v0[p];
        if (k == j || v0 == T(0) || cj.n_valid == 0) {  // constant path
            if (lane == 0) {
                if (COUNT) {
                    a.bound[p] = 1;
                } else {
                    const int64_t off = a.off[p];
                    a.lam[off] = 0.0;
                    a.val[off] = k == j ? T(1) : T(0);
                    // v = 1 for k == jhat: zero residual; v = 0: sum |x_ik|
                    if (a.res)
                        a.res[off] = k == j ? 0.0
                                            : column_total(a.ci[k], a.crem[k]);
                    a.len[p] = 1;
                }
            }
            continue;
        }
        bool pos;
        uint32_t ck_lo, ck_hi;
        K kv;
        range_of<T>(v0, pos, ck_lo, ck_hi, kv);
        const bool wide = pair_is_wide<T>(a, cj, k);
        const ColInfo ck = a.ci[k];
        const bool rem = REM && with_rem(a, cj, ck);
        ListSums ls{};
        const int c = scan_rows<T, COUNT, REM>(a, k, col, sb.part, wide, rem, pos, ck_lo, ck_hi, kv,
                                          ck.sigma, keys, rows, cap, ls, lane);
        if (COUNT) {
            if (lane == 0) a.bound[p] = (int64_t)c + 1;
            continue;
        }
        if (c > cap) {  // the big-pair kernel takes it
            if (lane == 0) a.big[atomicAdd(a.big_count, 1u)] = (int32_t)(p);
            continue;
        }
        const int ties = warp_bucket_sort<T>(keys, c, v0, sb, lane);
        if (ties < 0) {
            int P = 32;
            while (P < c) P <<= 1;  // at most cap, a power of two
            warp_list_sort<K>(keys, rows, c, P, lane);
        }
        emit_path<T, REM>(a, p, v0, pos, keys, rows, ties < 0 ? nullptr : sb.ord, ties != 0, c,
                          col, cj, ck, ls, rem, a.Xt + k * a.ldn, lane);
        __syncwarp();
    }
}

// Pairs with more rows in range than a warp's shared list: one warp per pair,
// the list in a global scratch slice (a pair's rows never exceed n).
template <typename T>
__global__ void __launch_bounds__(128) k_path_big(PathArgs<T> a) {
    using Tr = Traits<T>;
    using K = typename Tr::K;
    __shared__ uint16_t s_pend[4][PEND];
    const int lane = threadIdx.x & 31;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;  // worker warp
    const int npad = ((int)a.n + ROW_PAD - 1) & ~(ROW_PAD - 1);
    unsigned char *sl = a.scratch + (size_t)gw * (size_t)a.slice * (sizeof(K) + 20);
    K *keys = reinterpret_cast<K *>(sl);
    uint32_t *rows = reinterpret_cast<uint32_t *>(keys + a.slice);
    // the column arrays of jhat live in the slice too (each warp may hold a different jhat)
    float *own = reinterpret_cast<float *>(rows + a.slice);
    float *ci_inv = own + a.slice;
    int64_t *cq = reinterpret_cast<int64_t *>(ci_inv + a.slice);
    const uint32_t total = *a.big_count;  // rows > PATH_CAP_MIN, so a slice holds npad rows
    for (;;) {
        uint32_t w = 0;
        if (lane == 0) w = atomicAdd(a.big_next, 1u);
        w = __shfl_sync(0xFFFFFFFFu, w, 0);
        if (w >= total) break;
        const int64_t p = a.big[w];
        const int64_t j = p / a.m, k = p - j * a.m;
        const ColInfo cj = a.ci[j], ck = a.ci[k];
        const Column<T> col = stage_column<T>(a, j, own, ci_inv, cq, npad, lane, 32);
        __syncwarp();
        const T v0 = a.v0[p];
        bool pos;
        uint32_t ck_lo, ck_hi;
        K kv;
        range_of<T>(v0, pos, ck_lo, ck_hi, kv);
        const bool rem = with_rem(a, cj, ck);
        ListSums ls{};
        const int c = scan_rows<T, false, true>(a, k, col, s_pend[threadIdx.x >> 5],
                                          pair_is_wide<T>(a, cj, k), rem, pos, ck_lo, ck_hi, kv,
                                          ck.sigma, keys, rows, (int)a.slice, ls, lane);
        int P = 32;
        while (P < c) P <<= 1;
        warp_list_sort<K>(keys, rows, c, P, lane);
        emit_path<T, true>(a, p, v0, pos, keys, rows, nullptr, true, c, col, cj, ck, ls, rem,
                     a.Xt + k * a.ldn, lane);
        __syncwarp();
    }
}

// Exclusive scan of bound[0..N) into off[0..N] (off[N] = total), three steps.
constexpr int SCAN_B = 1024;
__global__ void __launch_bounds__(SCAN_B) k_scan_blocks(const int64_t *in, int64_t *out,
                                                        int64_t *bsum, int64_t N) {
    __shared__ int64_t ws[32];
    const int64_t i = (int64_t)blockIdx.x * SCAN_B + threadIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t x = i < N ? in[i] : 0;
    const int64_t incl = warp_scan_add(x, lane);
    if (lane == 31) ws[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const int64_t v = ws[lane];
        ws[lane] = warp_scan_add(v, lane) - v;
    }
    __syncthreads();
    const int64_t e = ws[warp] + incl - x;
    if (i < N) out[i] = e;
    if (threadIdx.x == SCAN_B - 1) bsum[blockIdx.x] = e + x;
}

__global__ void __launch_bounds__(SCAN_B) k_scan_tops(int64_t *bsum, int64_t nb, int64_t *total) {
    __shared__ int64_t ws[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t carry = 0;
    for (int64_t b0 = 0; b0 < nb; b0 += SCAN_B) {
        const int64_t b = b0 + threadIdx.x;
        const int64_t x = b < nb ? bsum[b] : 0;
        const int64_t incl = warp_scan_add(x, lane);
        if (lane == 31) ws[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            const int64_t v = ws[lane];
            ws[lane] = warp_scan_add(v, lane) - v;
        }
        __syncthreads();
        const int64_t e = carry + ws[warp] + incl - x;
        if (b < nb) bsum[b] = e;
        __syncthreads();
        if (threadIdx.x == SCAN_B - 1) ws[0] = e + x;
        __syncthreads();
        carry = ws[0];
        __syncthreads();
    }
    if (threadIdx.x == 0) *total = carry;
}

__global__ void k_scan_add(int64_t *out, const int64_t *bsum, int64_t N) {
    const int64_t i = (int64_t)blockIdx.x * SCAN_B + threadIdx.x;
    if (i < N) out[i] += bsum[blockIdx.x];
}

}  // namespace

size_t path_scan_scratch(int64_t N) { return (size_t)((N + SCAN_B - 1) / SCAN_B) * 8; }

cudaError_t launch_scan_i64(int64_t *a, int64_t N, int64_t *tmp, cudaStream_t st, int &launches) {
    const int64_t nb = (N + SCAN_B - 1) / SCAN_B;
    k_scan_blocks<<<(unsigned)nb, SCAN_B, 0, st>>>(a, a, tmp, N);
    k_scan_tops<<<1, SCAN_B, 0, st>>>(tmp, nb, a + N);
    k_scan_add<<<(unsigned)nb, SCAN_B, 0, st>>>(a, tmp, N);
    launches += 3;
    return cudaGetLastError();
}
int path_big_workers() { return 64; }

template <typename T> size_t path_slice_bytes(int64_t n) {
    int64_t P = 32;
    while (P < n) P <<= 1;
    return (size_t)P * (sizeof(typename Traits<T>::K) + 20);
}

// Shared memory of a CTA with lists of `cap` entries.
template <typename T> size_t path_smem_bytes(int64_t n, int cap) {
    const size_t npad = (size_t)((n + ROW_PAD - 1) & ~int64_t(ROW_PAD - 1));
    return npad * 16 + (size_t)PW * (cap * (sizeof(typename Traits<T>::K) + 4) + sort_bytes(cap));
}

// The limit on n is a fixed one (13,504 float, 10,368 double): the rows, in
// steps of 32, whose x, reciprocal and weight, with full lists, fit 227 KB (and
// that the fit, which solves lambda = 0, accepts).  Float rows next to it, with
// their padding to 128 and the queues, get lists of PATH_CAP_MIN.
template <typename T> int64_t path_max_rows() {
    const int64_t room = 227 * 1024 - (int64_t)PW * PATH_CAP * (sizeof(typename Traits<T>::K) + 4);
    const int64_t n = room / (int64_t)(sizeof(T) + 12) & ~int64_t(31);
    return std::min<int64_t>(n, max_rows_pairs<T>() & ~int64_t(31));
}

template <typename T>
cudaError_t launch_path(bool count, const T *Xt, const float *Xf, const ColInfo *ci, int64_t n,
                        int64_t m, int64_t ldn, const T *v0, int64_t *bound_or_off,
                        int64_t *scan_tmp, double *lam, T *val, double *res, float *crem,
                        int32_t *len, int32_t *big, uint32_t *big_count, unsigned char *scratch,
                        uint32_t *status, int num_sms, cudaStream_t st, int &launches) {
    PathArgs<T> a{};
    a.Xt = Xt;
    a.Xf = Xf;
    a.ci = ci;
    a.n = n;
    a.m = m;
    a.ldn = ldn;
    a.v0 = v0;
    a.status = status;
    // the count pass keeps no list, only the queue
    const int cap = count ? PEND : path_smem_bytes<T>(n, PATH_CAP) <= 227 * 1024 ? PATH_CAP : PATH_CAP_MIN;
    const size_t smem = path_smem_bytes<T>(n, cap);
    const int64_t chunks = std::max<int64_t>(1, std::min<int64_t>((m + PW - 1) / PW,
                                                                  (num_sms * 8 + m - 1) / m));
    const int kchunk = (int)((m + chunks - 1) / chunks);
    dim3 grid((unsigned)m, (unsigned)((m + kchunk - 1) / kchunk));
    cudaError_t e;
    if (count) {
        a.bound = bound_or_off;
        auto kern = k_path_pass<T, true, false, false>;
        if ((e = ensure_smem(reinterpret_cast<const void *>(kern), smem)) != cudaSuccess) return e;
        kern<<<grid, PW * 32, smem, st>>>(a, kchunk, cap);
        launches++;
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        // exclusive scan of the m*m bounds, in place, total at [m*m]
        return launch_scan_i64(bound_or_off, m * m, scan_tmp, st, launches);
    }
    a.off = bound_or_off;
    a.lam = lam;
    a.val = val;
    a.res = res;
    a.crem = crem;
    a.len = len;
    a.big = big;
    a.big_count = big_count;
    a.big_next = big_count + 1;
    a.inexact = big_count + 2;
    a.scratch = scratch;
    int64_t P = 32;
    while (P < n) P <<= 1;
    a.slice = P;
    if ((e = cudaMemsetAsync(big_count, 0, 3 * sizeof(uint32_t), st)) != cudaSuccess) return e;
    auto pass = [&](auto kern) -> cudaError_t {
        cudaError_t r = ensure_smem(reinterpret_cast<const void *>(kern), smem);
        if (r != cudaSuccess) return r;
        kern<<<grid, PW * 32, smem, st>>>(a, kchunk, cap);
        launches++;
        return cudaGetLastError();
    };
    if (!res) {
        e = pass(k_path_pass<T, false, false, false>);
    } else {
        k_colrem<T><<<(unsigned)m, 256, 0, st>>>(a);
        launches++;
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        if constexpr (sizeof(T) == 8) {
            e = pass(k_path_pass<T, false, true, false>);
        } else {
            e = pass(k_path_pass<T, false, false, true>);
            if (e == cudaSuccess) e = pass(k_path_pass<T, false, true, true>);
        }
    }
    if (e != cudaSuccess) return e;
    k_path_big<T><<<path_big_workers() / 4, 128, 0, st>>>(a);
    launches++;
    return cudaGetLastError();
}

template size_t path_slice_bytes<float>(int64_t);
template size_t path_slice_bytes<double>(int64_t);
template int64_t path_max_rows<float>();
template int64_t path_max_rows<double>();
template cudaError_t launch_path<float>(bool, const float *, const float *, const ColInfo *,
                                        int64_t, int64_t, int64_t, const float *, int64_t *,
                                        int64_t *, double *, float *, double *, float *,
                                        int32_t *, int32_t *, uint32_t *, unsigned char *,
                                        uint32_t *, int,
                                        cudaStream_t, int &);
template cudaError_t launch_path<double>(bool, const double *, const float *, const ColInfo *,
                                         int64_t, int64_t, int64_t, const double *, int64_t *,
                                         int64_t *, double *, double *, double *, float *,
                                         int32_t *, int32_t *, uint32_t *, unsigned char *,
                                        uint32_t *, int,
                                         cudaStream_t, int &);

L1L_CHECKS_READER(l1l_checks_path)

}  // namespace l1l
