// k_solpath.cu -- Algorithm 3: the solution path over all lambda >= 0.
//
// From the pair paths of Algorithm 2 (with each entry's residual R), the
// objective of preserved coordinate jhat is z_jhat(lambda) = sum_k (R + lambda
// |v|) of the entry of pair (jhat, k) holding at lambda: piecewise linear and
// concave in lambda.  Algorithm 3 finds, interval by interval, which jhat's
// line is lowest and where two lines cross (beta_L, beta_U).  Here:
//   1. every z_jhat is evaluated, with its slope, at NG lambdas, and a jhat is
//      dropped from every interval between two of them where it cannot be
//      lowest: z_jhat lies on or above its chord there, the minimum on or below
//      the tangents of the best functions at either end;
//   2. per interval and remaining jhat (a CTA each), the changes of its m pairs
//      inside the interval are sorted by lambda (a two-level bucket sort) and
//      prefix-summed into the pieces (lambda_start, I, s) of z_jhat;
//   3. in an interval with several, their lower envelope by a tree of pairwise
//      minimum merges (each piece of either function contributes at most one
//      interval to their minimum, so a merge never outgrows its inputs): the
//      second of two siblings to be finished merges them and goes on up, no
//      CTA waits for another.
// The intervals' pieces in order, less the seams that are no change of line,
// are the solution path: from lambda_start on, jhat* and z* = I + s lambda; v*
// is read from the pair paths of jhat*.
//
// Usually 1.0 to 1.1 functions remain per interval (planted data, 20 to 500
// columns), so sorting and merging, whose double arithmetic and 32-byte pieces
// the GPU is slow at (2 double operations per SM and cycle), is done for one
// function in all, spread over the intervals.  1000 points, 500 columns, 9.4
// million entries: 0.23 ms in all (evaluation 0.08, pieces 0.06), against
// 12.3 ms for building and merging all 500 functions whole.
#include <cmath>

#include "checks.cuh"
#include "common.cuh"
#include "launch.h"
#include "pairs.cuh"

namespace l1l {

namespace {

struct alignas(16) Piece {
    double lam;    // start of the piece (for changes: where the change happens)
    double I, s;   // intercept and slope (for changes: theirs, in fixed point)
    int32_t owner; // jhat
    int32_t pad;
};
static_assert(sizeof(Piece) == 32, "piece layout");

constexpr int NG = 32;        // lambdas of the pruning grid, one per lane
constexpr int ZT = 512;       // threads of the build and merge kernel
constexpr int NB1 = 512;      // buckets of the first level
constexpr int NB2 = 4096;     // buckets of the second, shared out by occupancy
constexpr int SORT_SMEM = 2048;  // changes sorted in shared memory, more in global
constexpr int RANK_MAX = 1024;  // larger buckets are sorted by the whole CTA

// Counters of one call, zeroed with the status word (l1line_status reads that).
struct SolHead {
    uint32_t status;
    uint32_t pad;
    unsigned long long lmax;     // largest breakpoint, as bits (all are >= 0)
    double g[NG + 1];            // the grid, then infinity
    int32_t best[NG];            // lowest function at each grid point
    int64_t unit0[NG + 1];       // first unit of each interval
};
static_assert(sizeof(SolHead) <= 1024, "head of the workspace");

// Everything the kernels share, in the workspace.  A unit is one function in
// one interval [g_i, g_(i+1)]; units are numbered interval by interval.
struct SolWs {
    SolHead *h;
    double *Z, *S;    // [NG][m] value and slope on the grid
    int64_t *C;       // [NG][m] changes at or below the grid point
    int32_t *shI, *shs;  // [m] fixed-point scales of its intercepts and slopes
    uint32_t *mask;   // [m] grid intervals in which jhat may be lowest
    int32_t *ujhat;   // [units] jhat
    int64_t *ubase;   // [units + 1] first piece of each unit's region
    int64_t *ucount;  // [units] pieces of the function at a region
    int32_t *ubuf;    // [units] the buffer it lies in
    int32_t *arrive;  // [2 units] children finished, per node of the merge trees
    Piece *buf[3];    // entries + NG m pieces each
};

// The largest sh with b 2^(e + sh) < 2^61 (b >= 0; as for 2^-1022 where b is less: the
// mantissa of a double is shifted by 9 bits at most).
__device__ __forceinline__ int fix_shift(double b, int e) {
    if (!(b > 0.0) || isinf(b)) return 0;
    return 60 - e - max(ilog2_pos(b), -1022);
}

// The largest breakpoint of all, and the fixed-point scales of jhat: a pair's
// residual and |v| run monotonically from its first entry to its last.
template <typename T>
__global__ void __launch_bounds__(256) k_zrange(int64_t m, const int64_t *__restrict__ off,
                                                const int32_t *__restrict__ len,
                                                const double *__restrict__ lam,
                                                const T *__restrict__ val,
                                                const double *__restrict__ res, SolWs w) {
    const int64_t j = blockIdx.x;
    __shared__ double sm[2][8];
    unsigned long long mx = 0;
    // both bounds; scaled down where they overflow, which the values need not
    for (int e = 0;; e = 64) {
        auto term = [&](double x) { return e != 0 ? fabs(x) * 0x1p-64 : fabs(x); };
        double bI = 0.0, bs = 0.0;
        for (int64_t k = threadIdx.x; k < m; k += blockDim.x) {
            const int64_t o = off[j * m + k], l = o + len[j * m + k] - 1;
            bI += term(res[o]) + term(res[l]);
            bs += term((double)val[o]) + term((double)val[l]);
            mx = max(mx, (unsigned long long)__double_as_longlong(lam[l]));
        }
        bI = warp_sum_f64(bI);
        bs = warp_sum_f64(bs);
        __syncthreads();
        if ((threadIdx.x & 31) == 0) {
            sm[0][threadIdx.x >> 5] = bI;
            sm[1][threadIdx.x >> 5] = bs;
        }
        __syncthreads();
        bI = bs = 0.0;
        for (int q = 0; q < 8; ++q) {
            bI += sm[0][q];
            bs += sm[1][q];
        }
        const bool finite = bI < INFINITY && bs < INFINITY;  // NaN: not
        if (!finite && e == 0) continue;
        if (threadIdx.x == 0) {
            if (!finite) atomicOr(&w.h->status, (uint32_t)ST_NONFINITE);
            w.shI[j] = fix_shift(bI, e);
            w.shs[j] = fix_shift(bs, e);
        }
        break;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, o));
    if ((threadIdx.x & 31) == 0 && mx != 0) atomicMax(&w.h->lmax, mx);
}

// The grid: squares, since most breakpoints lie near 0 (a pair's last one is
// about |x_jhat|_1 times its correlation), ending at the largest breakpoint,
// beyond which every function is linear.
__device__ __forceinline__ double grid_lambda(double lmax, int i) {
    const double u = (double)i * (1.0 / (NG - 1));
    return i == NG - 1 ? lmax : lmax * (u * u);
}

// |x| as a double; a normal float by integer instructions, which leaves the
// double pipe to the sums.
__device__ __forceinline__ double abs64(float x) {
    const uint32_t u = __float_as_uint(x) & 0x7FFFFFFFu;
    if (u - 0x00800000u >= 0x7F000000u) return (double)__uint_as_float(u);  // 0, subnormal, inf, NaN
    return __hiloint2double((int)((u >> 3) + (896u << 20)), (int)(u << 29));
}
__device__ __forceinline__ double abs64(double x) { return fabs(x); }

// z_jhat, its right slope and the changes passed, on the grid: warps over k, a
// lane per grid point, the entry holding there by binary search; sums in a
// fixed order.  Bound by the two double additions per pair and point.
constexpr int EVT = 512;
template <typename T>
__global__ void __launch_bounds__(EVT) k_zeval(int64_t m, const int64_t *__restrict__ off,
                                               const int32_t *__restrict__ len,
                                               const double *__restrict__ lam,
                                               const T *__restrict__ val,
                                               const double *__restrict__ res, SolWs w) {
    __shared__ double sz[EVT / 32][NG], ss[EVT / 32][NG];
    __shared__ int64_t sc[EVT / 32][NG];
    const int64_t j = blockIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double g = grid_lambda(__longlong_as_double((long long)w.h->lmax), lane);
    const long long gb = __double_as_longlong(g);
    double z = 0.0, s = 0.0;
    int64_t c = 0;
    for (int64_t k = warp; k < m; k += EVT / 32) {
        const int64_t o = off[j * m + k];
        int lo = 1, hi = len[j * m + k];  // first entry with lambda > g; entry 0 starts at 0
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (__double_as_longlong(lam[o + mid]) <= gb)
                lo = mid + 1;
            else
                hi = mid;
        }
        z += res[o + lo - 1];
        s += abs64(val[o + lo - 1]);
        c += lo - 1;
    }
    sz[warp][lane] = z;
    ss[warp][lane] = s;
    sc[warp][lane] = c;
    __syncthreads();
    if (warp == 0) {
        for (int q = 1; q < EVT / 32; ++q) {
            z += sz[q][lane];
            s += ss[q][lane];
            c += sc[q][lane];
        }
        w.Z[(int64_t)lane * m + j] = fma(g, s, z);
        w.S[(int64_t)lane * m + j] = s;
        w.C[(int64_t)lane * m + j] = c;
        if (j == 0) {
            w.h->g[lane] = g;
            if (lane == 0) w.h->g[NG] = INFINITY;
        }
    }
}

// The lowest function at grid point blockIdx.x (ties to the smaller jhat).
__global__ void __launch_bounds__(256) k_zbest(int64_t m, SolWs w) {
    const double *z = w.Z + (int64_t)blockIdx.x * m;
    double b = INFINITY;
    int32_t bj = 0x7FFFFFFF;
    auto take = [&](double x, int32_t j) {
        if (x < b || (x == b && j < bj)) {
            b = x;
            bj = j;
        }
    };
    for (int64_t j = threadIdx.x; j < m; j += 256) take(z[j], (int32_t)j);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        take(__shfl_xor_sync(0xFFFFFFFFu, b, o), __shfl_xor_sync(0xFFFFFFFFu, bj, o));
    __shared__ double sb[8];
    __shared__ int32_t sj[8];
    if ((threadIdx.x & 31) == 0) {
        sb[threadIdx.x >> 5] = b;
        sj[threadIdx.x >> 5] = bj;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int q = 1; q < 8; ++q) take(sb[q], sj[q]);
        w.h->best[blockIdx.x] = bj == 0x7FFFFFFF ? 0 : bj;
    }
}

// The grid intervals in which jhat may be lowest: a warp per jhat, lane i for
// [g_i, g_(i+1)], the last lane for [g_31, inf).  z_jhat is on or above its
// chord, the minimum on or below four tangents (of the lowest function at
// either end, at both ends); jhat stays where some lambda has the chord below
// all four lines plus the margin.  The margin, 2^-20 (float) or 2^-30
// (double) of the largest value, is far above what departs from that: the
// rounding of the values v (a pair's objective is concave only up to
// 2^-23 sum_i |x_ik|, respectively 2^-52), and every sum's rounding.  A NaN
// keeps the jhat.
template <typename T> __global__ void __launch_bounds__(256) k_zsurvive(int64_t m, SolWs w) {
    const int lane = threadIdx.x & 31;
    const int64_t j = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (j >= m) return;
    const int q0 = w.h->best[lane], q1 = w.h->best[min(lane + 1, NG - 1)];
    const double g = w.h->g[lane];
    const bool last = lane == NG - 1;
    const double h = last ? INFINITY : w.h->g[lane + 1] - g;
    const double *Z0 = w.Z + (int64_t)lane * m, *S0 = w.S + (int64_t)lane * m;
    double zs = fabs(Z0[q0]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) zs = fmax(zs, __shfl_xor_sync(0xFFFFFFFFu, zs, o));
    const double mg = (sizeof(T) == 4 ? 0x1p-20 : 0x1p-30) * zs;
    const double a = Z0[j];
    double lo = 0.0, hi = h;
    bool out = false;
    double sl;
    auto line = [&](double y, double s) {  // y + s x against a + sl x, x = lambda - g_i
        const double c = a - y, d = sl - s;
        if (d > 0.0)
            hi = fmin(hi, (mg - c) / d);
        else if (d < 0.0)
            lo = fmax(lo, (mg - c) / d);
        else if (d == 0.0 && c > mg)
            out = true;
    };
    if (last) {
        sl = S0[j];
        line(Z0[q0], S0[q0]);
    } else {
        const double *Z1 = Z0 + m, *S1 = S0 + m;
        sl = (Z1[j] - a) / h;
        line(Z0[q0], S0[q0]);
        line(Z1[q0] - S1[q0] * h, S1[q0]);
        line(Z0[q1], S0[q1]);
        line(Z1[q1] - S1[q1] * h, S1[q1]);
        out |= h == 0.0;  // no breakpoints at all: only the last interval
    }
    const unsigned keep = __ballot_sync(0xFFFFFFFFu, !out && !(lo > hi));
    if (lane == 0) w.mask[j] = keep;
}

// Block-wide exclusive scan of one int64 per thread.
__device__ int64_t block_excl_scan(int64_t x, int64_t *sm, int64_t &total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t incl = warp_scan_add(x, lane);
    __syncthreads();
    if (lane == 31) sm[warp] = incl;
    __syncthreads();
    int64_t t = lane < (int)(blockDim.x >> 5) ? sm[lane] : 0;
    t = warp_scan_add(t, lane);
    total = __shfl_sync(0xFFFFFFFFu, t, 31);
    const int64_t before = __shfl_sync(0xFFFFFFFFu, t, max(warp - 1, 0));
    return (warp ? before : 0) + incl - x;
}

// The units: warp i lists the functions of interval i in ascending order, with
// their regions (one piece per change, and the one holding at the start).
constexpr int ZL = 1024;
__global__ void __launch_bounds__(ZL) k_zlist(int64_t m, SolWs w) {
    static_assert(ZL == 32 * NG, "a warp per interval");
    __shared__ int64_t s_n[NG], s_c[NG];
    const unsigned FULL = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31, i = threadIdx.x >> 5;
    const int64_t *C0 = w.C + (int64_t)i * m, *C1 = C0 + m;
    auto room = [&](int64_t j) -> int64_t { return i == NG - 1 ? 1 : C1[j] - C0[j] + 1; };
    int64_t n = 0, c = 0;
    for (int64_t j = lane; j < m; j += 32)
        if ((w.mask[j] >> i) & 1u) {
            n += 1;
            c += room(j);
        }
    n = warp_sum_i64(n);
    c = warp_sum_i64(c);
    if (lane == 0) {
        s_n[i] = n;
        s_c[i] = c;
    }
    __syncthreads();
    int64_t u = 0, base = 0;
    for (int q = 0; q < i; ++q) {
        u += s_n[q];
        base += s_c[q];
    }
    if (lane == 0) {
        w.h->unit0[i] = u;
        if (i == NG - 1) {
            w.h->unit0[NG] = u + n;
            w.ubase[u + n] = base + c;
        }
    }
    for (int64_t j0 = 0; j0 < m; j0 += 32) {
        const int64_t j = j0 + lane;
        const bool on = j < m && ((w.mask[j] >> i) & 1u);
        const unsigned b = __ballot_sync(FULL, on);
        const int64_t r = on ? room(j) : 0;
        const int64_t incl = warp_scan_add(r, lane);
        if (on) {
            const int64_t at = u + __popc(b & ((1u << lane) - 1u));
            w.ujhat[at] = (int32_t)j;
            w.ubase[at] = base + incl - r;
            w.arrive[2 * at] = 0;
            w.arrive[2 * at + 1] = 0;
        }
        u += __popc(b);
        base += __shfl_sync(FULL, incl, 31);
    }
}

// x 2^sh rounded to an integer (half up), |x| 2^sh < 2^62.  Sums of these are
// exact, so a function's intercept at any piece is the rounded sum of its
// pairs' current entries, whatever the order, to within m 2^-62 of the bound.
// bad: x is above the bound or not finite (not a path of l1line_path_write).
__device__ __forceinline__ int64_t fix_rn(double x, int sh, bool &bad) {
    const uint64_t u = (uint64_t)__double_as_longlong(x);
    const int be = (int)((u >> 52) & 0x7FF);
    uint64_t f = u & 0xFFFFFFFFFFFFFull;
    if (be) f |= 0x10000000000000ull;
    const int s = (be ? be : 1) - 1075 + sh;
    bad |= s > 9 && f != 0;
    if (s >= 0)
        f = s > 9 ? 0 : f << s;
    else if (s > -60)
        f = (f + (1ull << (-s - 1))) >> -s;
    else
        f = 0;
    return (u >> 63) ? -(int64_t)f : (int64_t)f;
}
__device__ __forceinline__ double unfix(int64_t x, int sh) { return scalbn((double)x, -sh); }

// One change in the bucket sort: its lambda as bits and the entry it leads to
// (-1: the base), which also orders equal lambdas.
struct alignas(16) KeySrc {
    long long key, src;
};
__device__ __forceinline__ bool before(const KeySrc &a, const KeySrc &b) {
    return a.key < b.key || (a.key == b.key && a.src < b.src);
}

struct BuildSmem {
    KeySrc a[SORT_SMEM], b[SORT_SMEM];
    uint32_t fine[NB2];        // counts, then ends, of the second-level buckets
    uint32_t coarse[NB1];      // counts of the first-level ones
    uint32_t fbase[NB1 + 1];   // first second-level bucket of each
};

// Bitonic sort of x[0..c) by the whole CTA (a bucket too large to rank).
__device__ void cta_sort(KeySrc *x, int64_t c) {
    int64_t P = 1;
    while (P < c) P <<= 1;
    for (int64_t size = 2; size <= P; size <<= 1)
        for (int64_t stride = size >> 1; stride > 0; stride >>= 1) {
            for (int64_t t = threadIdx.x; t < P / 2; t += ZT) {
                // ascending throughout: the first step of a size mirrors, so
                // that slots past c stay behind every element
                const int64_t i = 2 * t - (t & (stride - 1));
                const int64_t o = stride == size >> 1 ? (i ^ (size - 1)) : i + stride;
                if (i < c && o < c) {
                    const KeySrc a = x[i], b = x[o];
                    if (before(b, a)) {
                        x[i] = b;
                        x[o] = a;
                    }
                }
            }
            __syncthreads();
        }
}

// The pieces of unit u, function j in interval i, into buf[0]; more than
// SORT_SMEM changes are sorted in its region of buf[1] and buf[2].
template <typename T>
__device__ void build_unit(int64_t m, int64_t u, int i, const int64_t *__restrict__ off,
                           const int32_t *__restrict__ len, const double *__restrict__ lam,
                           const T *__restrict__ val, const double *__restrict__ res,
                           const SolWs &w, BuildSmem &sm) {
    __shared__ int64_t smi[ZT / 32];
    __shared__ uint32_t s_big;
    const int tid = threadIdx.x;
    const int64_t j = w.ujhat[u], base = w.ubase[u], room = w.ubase[u + 1] - base;
    const int shI = w.shI[j], shs = w.shs[j];
    const double g0 = w.h->g[i];
    const long long k0 = __double_as_longlong(g0), k1 = __double_as_longlong(w.h->g[i + 1]);
    KeySrc *fill = room <= SORT_SMEM ? sm.a : reinterpret_cast<KeySrc *>(w.buf[1] + base);
    KeySrc *part = room <= SORT_SMEM ? sm.b : reinterpret_cast<KeySrc *>(w.buf[2] + base);
    Piece *sorted = w.buf[1] + base, *out = w.buf[0] + base;
    for (int b = tid; b < NB2; b += ZT) sm.fine[b] = 0;
    for (int b = tid; b < NB1; b += ZT) sm.coarse[b] = 0;
    if (tid == 0) s_big = 0;
    // buckets: equal steps of the lambda as float, monotone in lambda
    const float f0 = (float)g0, width = (float)w.h->g[i + 1] - f0;
    const float sc = width > 0x1p-100f && width < 0x1p100f ? (float)NB1 / width : 0.0f;
    auto spot = [&](long long key, float &x) -> int {
        x = ((float)__longlong_as_double(key) - f0) * sc;
        x = fminf(fmaxf(x, 0.0f), (float)NB1);
        return min(NB1 - 1, (int)x);
    };
    __syncthreads();
    // the entry of each pair holding at g_i, and the changes inside the interval
    bool bad = false;
    int64_t I0 = 0, s0 = 0, cnt = 1;  // element 0: the piece holding at g_i
    for (int64_t kb = 0; kb < m; kb += ZT) {
        const int64_t k = kb + tid;
        int64_t o = 0;
        int lo = 1, hi = 0;
        if (k < m) {
            o = off[j * m + k];
            const int L = len[j * m + k];
            hi = L;
            while (lo < hi) {  // first entry past g_i
                const int mid = (lo + hi) >> 1;
                if (__double_as_longlong(lam[o + mid]) <= k0)
                    lo = mid + 1;
                else
                    hi = mid;
            }
            int top = L;
            hi = lo;
            while (hi < top) {  // first entry from g_(i+1) on
                const int mid = (hi + top) >> 1;
                if (__double_as_longlong(lam[o + mid]) < k1)
                    hi = mid + 1;
                else
                    top = mid;
            }
            I0 += fix_rn(res[o + lo - 1], shI, bad);
            s0 += fix_rn(fabs((double)val[o + lo - 1]), shs, bad);
        }
        int64_t tot;
        const int64_t dst = cnt + block_excl_scan((int64_t)max(hi - lo, 0), smi, tot);
        auto put = [&](int64_t at, int64_t src) {
            const long long key = __double_as_longlong(lam[src]);
            fill[L1L_CHK(at, room)] = KeySrc{key, src};
            float x;
            atomicAdd(&sm.coarse[spot(key, x)], 1u);
        };
        constexpr int FEW = 8;  // a pair with more changes here is filled by the warp
        if (hi - lo <= FEW)
            for (int g = lo; g < hi; ++g) put(dst + (g - lo), o + g);
        for (unsigned b = __ballot_sync(0xFFFFFFFFu, hi - lo > FEW); b; b &= b - 1) {
            const int ln = __ffs(b) - 1;
            const int64_t d = __shfl_sync(0xFFFFFFFFu, dst, ln);
            const int64_t e = __shfl_sync(0xFFFFFFFFu, o + lo, ln);
            const int c = __shfl_sync(0xFFFFFFFFu, hi - lo, ln);
            for (int g = tid & 31; g < c; g += 32) put(d + g, e + g);
        }
        cnt += tot;
    }
    if (tid == 0) {
        fill[0] = KeySrc{k0, -1};
        float x;
        atomicAdd(&sm.coarse[spot(k0, x)], 1u);
    }
    {
        int64_t t;
        block_excl_scan(I0, smi, t);
        I0 = t;
        block_excl_scan(s0, smi, t);
        s0 = t;
    }
    __syncthreads();
    // second level: every first-level bucket is cut evenly, into as many as its
    // share of the elements asks for
    {
        static_assert(NB1 == ZT, "a thread per first-level bucket");
        const uint32_t c = sm.coarse[tid];
        const int64_t want = (int64_t)c * (NB2 - NB1) / cnt + 1;
        int64_t t;
        const int64_t ex = block_excl_scan(want, smi, t);
        sm.fbase[tid] = (uint32_t)ex;
        if (tid == 0) sm.fbase[NB1] = (uint32_t)t;  // <= NB2
    }
    __syncthreads();
    auto bucket = [&](long long key) -> int {
        float x;
        const int b = spot(key, x);
        const uint32_t b0 = sm.fbase[b], nf = sm.fbase[b + 1] - b0;
        return (int)(b0 + min(nf - 1, (uint32_t)((x - (float)b) * (float)nf)));
    };
    for (int64_t e = tid; e < cnt; e += ZT) atomicAdd(&sm.fine[bucket(fill[e].key)], 1u);
    __syncthreads();
    {  // starts of the second-level buckets, eight to a thread
        constexpr int Q = NB2 / ZT;
        uint32_t c[Q], sum = 0, big = 0;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            c[q] = sm.fine[Q * tid + q];
            sum += c[q];
            big = max(big, c[q]);
        }
        if (big > RANK_MAX) atomicMax(&s_big, big);
        int64_t t;
        uint32_t ex = (uint32_t)block_excl_scan((int64_t)sum, smi, t);
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            sm.fine[Q * tid + q] = ex;
            ex += c[q];
        }
    }
    __syncthreads();
    for (int64_t e = tid; e < cnt; e += ZT) {
        const KeySrc x = fill[e];
        part[L1L_CHK((int64_t)atomicAdd(&sm.fine[bucket(x.key)], 1u), room)] = x;
    }
    __syncthreads();
    if (s_big > RANK_MAX) {  // sm.fine now holds the ends
        for (int b = 0; b < NB2; ++b) {
            const uint32_t b0 = b ? sm.fine[b - 1] : 0u, b1 = sm.fine[b];
            if (b1 - b0 > RANK_MAX) cta_sort(part + b0, b1 - b0);
        }
    }
    // each change to its place in its bucket, with its steps of I and s
    for (int64_t e = tid; e < cnt; e += ZT) {
        const KeySrc x = part[e];
        const int b = bucket(x.key);
        const uint32_t b0 = b ? sm.fine[b - 1] : 0u, b1 = sm.fine[b];
        int64_t pos = e;
        if (b1 - b0 <= RANK_MAX) {
            uint32_t r = 0;
            for (uint32_t q = b0; q < b1; ++q) r += before(part[q], x) ? 1u : 0u;
            pos = b0 + r;
        }
        int64_t dI = I0, ds = s0;
        if (x.src >= 0) {
            dI = fix_rn(res[x.src], shI, bad) - fix_rn(res[x.src - 1], shI, bad);
            ds = fix_rn(fabs((double)val[x.src]), shs, bad) -
                 fix_rn(fabs((double)val[x.src - 1]), shs, bad);
        }
        Piece p;
        p.lam = __longlong_as_double(x.key);
        p.I = __longlong_as_double(dI);
        p.s = __longlong_as_double(ds);
        p.owner = (int32_t)j;
        p.pad = 0;
        sorted[L1L_CHK(pos, room)] = p;
    }
    if (bad) atomicOr(&w.h->status, (uint32_t)ST_NONFINITE);
    __syncthreads();
    // prefix sums, one piece per distinct lambda (the last change at that
    // lambda closes it) that is another line than the piece before: a step between
    // values that differ in the last place can leave intercept and slope as they are
    struct Line {
        double I, s;
    };
    Line *line = reinterpret_cast<Line *>(sm.a);  // the chunk's, in order
    static_assert(sizeof(sm.a) >= ZT * sizeof(Line), "a line per thread");
    int64_t cI = 0, cs = 0, cw = 0;
    Line held{0.0, 0.0};  // of the last piece of the chunks before
    for (int64_t e0 = 0; e0 < cnt; e0 += ZT) {
        const int64_t e = e0 + tid;
        Piece p{};
        bool end = false;
        if (e < cnt) {
            p = sorted[e];
            end = e == cnt - 1 || __double_as_longlong(sorted[e + 1].lam) !=
                                      __double_as_longlong(p.lam);
        }
        const int64_t x = __double_as_longlong(p.I), y = __double_as_longlong(p.s);
        int64_t tI, ts, tl, tw;
        const int64_t eI = block_excl_scan(x, smi, tI);
        const int64_t es = block_excl_scan(y, smi, ts);
        const int64_t el = block_excl_scan(end ? 1 : 0, smi, tl);
        if (end) {
            p.I = unfix(cI + eI + x, shI);
            p.s = unfix(cs + es + y, shs);
            line[el] = Line{p.I, p.s};
        }
        __syncthreads();
        bool keep = end;
        if (end && (cw != 0 || el != 0)) {
            const Line q = el != 0 ? line[el - 1] : held;
            keep = q.I != p.I || q.s != p.s;
        }
        if (tl != 0) held = line[tl - 1];
        const int64_t ew = block_excl_scan(keep ? 1 : 0, smi, tw);
        if (keep) out[cw + ew] = p;
        __syncthreads();
        cI += tI;
        cs += ts;
        cw += tw;
    }
    if (tid == 0) {
        w.ucount[u] = cw;
        w.ubuf[u] = 0;
    }
    __syncthreads();
}

// Minimum of two concave piecewise-linear functions F, G (pieces ordered by
// start, both starting at 0).
// Intercepts and slopes are double sums of many terms, so values and slopes
// that agree to a relative 1e-12 are taken as equal: equal lines go to the
// smaller owner, and lines of equal slope never cross (far beyond the last
// breakpoint every slope is exactly 1 and rounding would otherwise invent a
// crossing).
constexpr double SOL_RTOL = 1e-12;
// The winner(s) on one elementary interval [cur, end) where F is the line f
// and G the line g: calls emit(line, start) once or twice (a crossing).
template <typename E>
__device__ __forceinline__ void interval_min(const Piece &f, const Piece &g, double cur,
                                             double end, E &&emit) {
    double dI = f.I - g.I, ds = f.s - g.s;  // (f - g)(lambda) = dI + ds lambda
    if (fabs(ds) <= SOL_RTOL * fmax(fabs(f.s), fabs(g.s))) ds = 0.0;
    double d0 = dI + ds * cur;
    if (fabs(d0) <= SOL_RTOL * (fabs(f.I) + fabs(g.I) + (fabs(f.s) + fabs(g.s)) * cur)) d0 = 0.0;
    const bool f_first =
        d0 < 0.0 || (d0 == 0.0 && (ds < 0.0 || (ds == 0.0 && f.owner <= g.owner)));
    emit(f_first ? f : g, cur);
    if (ds != 0.0) {
        const double x = -dI / ds;  // the lines cross at x
        if (x > cur && x < end) {
            // past the crossing, f is lower exactly when f - g decreases
            const bool f_after = ds < 0.0;
            if (f_after != f_first) emit(f_after ? f : g, x);
        }
    }
}

__device__ __forceinline__ bool same_line(const Piece &a, const Piece &b) {
    return a.owner == b.owner && a.I == b.I && a.s == b.s;
}

struct MergeSmem {
    Piece lastp[ZT], firstp[ZT];
    int64_t cnt[ZT / 32];
    int last[ZT];
};

// Minimum of two concave piecewise-linear functions F (a pieces) and G (b
// pieces), starting at the same lambda, by one CTA.  The merged sequence of piece
// starts is split evenly (merge path); each thread handles the elementary
// intervals that end at its consumed starts: a counting pass, a block scan of
// the counts (dropping a thread's first piece when it repeats the previous
// thread's last one), then the writing pass.  stop: the lambda where the
// interval ends.  Returns the piece count, or -1 when it would exceed cap.
__device__ int64_t block_min_merge(const Piece *F, int64_t a, const Piece *G, int64_t b,
                                   Piece *out, int64_t cap, double stop, MergeSmem &sm) {
    const int t = threadIdx.x;
    const int64_t L = a + b;
    const int64_t p0 = L * t / ZT, p1 = L * (t + 1) / ZT;
    auto bits = [](double x) { return __double_as_longlong(x); };  // lambdas are >= 0
    // merge-path split: i starts of F among the first p0 consumed
    int64_t lo = p0 > b ? p0 - b : 0, hi = p0 < a ? p0 : a;
    while (lo < hi) {
        const int64_t i = (lo + hi) >> 1;
        if (bits(F[i].lam) <= bits(G[p0 - 1 - i].lam))
            lo = i + 1;
        else
            hi = i;
    }
    const int64_t i_start = lo, j_start = p0 - lo;
    // one walk, run twice: count (write == false) or write at base
    auto walk = [&](bool write, int64_t base, bool drop_first, Piece &first, Piece &last,
                    int64_t &count) {
        int64_t i = i_start, j = j_start, w = 0;
        bool have = false;
        Piece prev;
        auto emit = [&](const Piece &ln, double start) {
            if (have && same_line(prev, ln)) return;
            if (!have) first = ln;
            const bool skip = !have && drop_first;
            have = true;
            prev = ln;
            if (skip) return;
            if (write && base + w < cap) {
                Piece q = ln;
                q.lam = start;
                out[base + w] = q;
            }
            ++w;
        };
        // the pieces holding and the starts to come
        Piece f{}, g{};
        if (i > 0) f = F[i - 1];
        if (j > 0) g = G[j - 1];
        Piece fn{}, gn{};
        fn.lam = gn.lam = stop;
        if (i < a) fn = F[i];
        if (j < b) gn = G[j];
        for (int64_t p = p0; p < p1; ++p) {
            if (j >= b || (i < a && bits(fn.lam) <= bits(gn.lam))) {
                f = fn;
                ++i;
                if (i < a) fn = F[i];
                else fn.lam = stop;
            } else {
                g = gn;
                ++j;
                if (j < b) gn = G[j];
                else gn.lam = stop;
            }
            if (i < 1 || j < 1) continue;
            const double cur = bits(f.lam) > bits(g.lam) ? f.lam : g.lam;
            const double end = bits(fn.lam) < bits(gn.lam) ? fn.lam : gn.lam;
            if (bits(cur) >= bits(end)) continue;
            interval_min(f, g, cur, end, emit);
        }
        if (have) last = prev;
        count = w;
        return have;
    };
    Piece first{}, last{};
    int64_t c = 0;
    const bool have = walk(false, 0, false, first, last, c);
    sm.last[t] = have ? t : -1;
    sm.lastp[t] = last;
    sm.firstp[t] = first;
    __syncthreads();
    // nearest earlier thread that produced a piece (its last line)
    int prev_t = -1;
    for (int u = t - 1; u >= 0; --u)
        if (sm.last[u] >= 0) {
            prev_t = u;
            break;
        }
    const bool drop = have && prev_t >= 0 && same_line(sm.lastp[prev_t], sm.firstp[t]);
    int64_t total;
    const int64_t base = block_excl_scan(c - (drop ? 1 : 0), sm.cnt, total);
    int64_t c2 = 0;
    walk(true, base, drop, first, last, c2);
    __syncthreads();
    return total > cap ? -1 : total;
}

// Units in turn over the CTAs: a unit's pieces, then up its interval's merge
// tree.  At every node the first sibling to arrive leaves; the second, which
// sees both, merges them into the buffer that holds neither.  A piece count
// beyond the region sets status bit ST_INTERNAL.
template <typename T>
__global__ void __launch_bounds__(ZT, 2) k_zbuild(int64_t m, const int64_t *off, const int32_t *len,
                                                const double *lam, const T *val,
                                                const double *res, SolWs w) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_old;
    const int64_t units = w.h->unit0[NG];
    for (int64_t u = blockIdx.x; u < units; u += gridDim.x) {
        int i = 0;
        while (w.h->unit0[i + 1] <= u) ++i;
        const int64_t u0 = w.h->unit0[i], ns = w.h->unit0[i + 1] - u0;
        build_unit<T>(m, u, i, off, len, lam, val, res, w, *reinterpret_cast<BuildSmem *>(smem));
        int64_t s = u - u0;
        int64_t node0 = 2 * u0;  // first counter of the level
        for (int64_t half = 1; half < ns; half *= 2) {
            const int64_t left = s & ~(2 * half - 1), right = left + half;
            const int64_t node = node0 + left / (2 * half);
            node0 += (ns + 2 * half - 1) / (2 * half);
            s = left;
            if (right >= ns) continue;  // no sibling
            __threadfence();
            __syncthreads();
            if (threadIdx.x == 0) s_old = atomicAdd(&w.arrive[node], 1);
            __syncthreads();
            if (s_old == 0) break;
            __threadfence();
            const int bf = w.ubuf[u0 + left], bg = w.ubuf[u0 + right];
            const int bo = bf != 0 && bg != 0 ? 0 : (bf != 1 && bg != 1 ? 1 : 2);
            const int64_t fb = w.ubase[u0 + left], gb = w.ubase[u0 + right];
            const int64_t cap = w.ubase[u0 + min(ns, left + 2 * half)] - fb;
            const int64_t r = block_min_merge(
                w.buf[bf] + fb, w.ucount[u0 + left], w.buf[bg] + gb, w.ucount[u0 + right],
                w.buf[bo] + fb, cap, w.h->g[i + 1], *reinterpret_cast<MergeSmem *>(smem));
            if (threadIdx.x == 0) {
                if (r < 0) atomicOr(&w.h->status, (uint32_t)ST_INTERNAL);
                w.ucount[u0 + left] = r < 0 ? cap : r;
                w.ubuf[u0 + left] = bo;
            }
        }
        __syncthreads();
    }
}

// The solution's pieces: the intervals' in order, without an interval's first
// piece where it is the line that holds already.  Built by a CTA's first warp.
struct SolView {
    int64_t first[NG + 1];   // first solution piece of each interval
    const Piece *src[NG];    // its pieces, the dropped one left out
    __device__ void init(const SolWs &w) {
        static_assert(NG == 32, "a lane per interval");
        const unsigned FULL = 0xFFFFFFFFu;
        const int i = threadIdx.x & 31;
        const int64_t u = w.h->unit0[i];
        const bool any = u < w.h->unit0[i + 1];
        const Piece *p = any ? w.buf[w.ubuf[u]] + w.ubase[u] : nullptr;
        int64_t c = any ? w.ucount[u] : 0;
        const unsigned before = __ballot_sync(FULL, any) & ((1u << i) - 1u);
        const Piece *last = reinterpret_cast<const Piece *>(__shfl_sync(
            FULL, (unsigned long long)(any ? p + c - 1 : p), before ? 31 - __clz(before) : 0));
        if (any && before && same_line(*last, *p)) {
            ++p;
            --c;
        }
        const int64_t incl = warp_scan_add(c, i);
        first[i] = incl - c;
        src[i] = p;
        if (i == 31) first[NG] = incl;
    }
    __device__ const Piece &operator[](int64_t e) const {
        int i = 0;
        while (first[i + 1] <= e) ++i;
        return src[i][e - first[i]];
    }
};

// v* of each solution piece: for pair (jhat*, k), the value holding just after
// the piece's start (last entry whose lambda is <= the start).  A CTA takes
// VB consecutive pieces, a thread one k at a time: it searches the pair's path
// for the first piece and steps forward from there (again for a new owner).
constexpr int VB = 32, VT = 256;
template <typename T>
__global__ void __launch_bounds__(VT) k_solution_v(int64_t m, int64_t cap, SolWs w,
                                                    const int64_t *__restrict__ off,
                                                    const int32_t *__restrict__ len,
                                                    const double *__restrict__ lam,
                                                    const T *__restrict__ val,
                                                    T *__restrict__ out_v) {
    __shared__ long long s_lam[VB];
    __shared__ int32_t s_own[VB];
    __shared__ SolView env;
    if (threadIdx.x < 32) env.init(w);
    __syncthreads();
    const int64_t count = min(env.first[NG], cap);
    for (int64_t e0 = (int64_t)blockIdx.x * VB; e0 < count; e0 += (int64_t)gridDim.x * VB) {
        const int c = (int)min((int64_t)VB, count - e0);
        __syncthreads();
        if (threadIdx.x < c) {
            s_lam[threadIdx.x] = __double_as_longlong(env[e0 + threadIdx.x].lam);
            s_own[threadIdx.x] = env[e0 + threadIdx.x].owner;
        }
        __syncthreads();
        for (int64_t k = threadIdx.x; k < m; k += VT) {
            int own = -1, at = 0, L = 0;
            int64_t o = 0;
            long long next = 0;
            T v = T(0);
            for (int e = 0; e < c; ++e) {
                const long long x = s_lam[e];
                if (s_own[e] != own) {
                    own = s_own[e];
                    o = off[(int64_t)own * m + k];
                    L = len[(int64_t)own * m + k];
                    int lo = 0, hi = L;  // first entry with lam > start
                    while (lo < hi) {
                        const int mid = (lo + hi) >> 1;
                        if (__double_as_longlong(lam[o + mid]) <= x)
                            lo = mid + 1;
                        else
                            hi = mid;
                    }
                    at = lo > 0 ? lo - 1 : 0;
                    v = val[o + at];
                    next = at + 1 < L ? __double_as_longlong(lam[o + at + 1]) : 0x7FFFFFFFFFFFFFFFll;
                } else if (next <= x) {
                    do {
                        ++at;
                        next = at + 1 < L ? __double_as_longlong(lam[o + at + 1])
                                          : 0x7FFFFFFFFFFFFFFFll;
                    } while (next <= x);
                    v = val[o + at];
                }
                out_v[(e0 + e) * m + k] = v;
            }
        }
    }
}

__global__ void k_solution_out(SolWs w, int64_t cap, double *start, int32_t *jhat, double *I,
                               double *s, int64_t *count) {
    __shared__ SolView env;
    if (threadIdx.x < 32) env.init(w);
    __syncthreads();
    const int64_t c = env.first[NG];
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < min(c, cap);
         e += (int64_t)gridDim.x * blockDim.x) {
        start[e] = env[e].lam;
        jhat[e] = env[e].owner;
        I[e] = env[e].I;
        s[e] = env[e].s;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *count = c;
}

size_t sol_layout(int64_t m, int64_t entries, unsigned char *ws, SolWs &w) {
    size_t o = 0;
    auto take = [&](size_t bytes) -> unsigned char * {
        unsigned char *p = ws ? ws + o : nullptr;
        o += (bytes + 255) & ~size_t(255);
        return p;
    };
    const size_t um = (size_t)m;
    w.h = reinterpret_cast<SolHead *>(take(sizeof(SolHead)));
    w.Z = reinterpret_cast<double *>(take(um * NG * 8));
    w.S = reinterpret_cast<double *>(take(um * NG * 8));
    w.C = reinterpret_cast<int64_t *>(take(um * NG * 8));
    w.shI = reinterpret_cast<int32_t *>(take(um * 4));
    w.shs = reinterpret_cast<int32_t *>(take(um * 4));
    w.mask = reinterpret_cast<uint32_t *>(take(um * 4));
    w.ujhat = reinterpret_cast<int32_t *>(take(um * NG * 4));
    w.ubase = reinterpret_cast<int64_t *>(take((um * NG + 1) * 8));
    w.ucount = reinterpret_cast<int64_t *>(take(um * NG * 8));
    w.ubuf = reinterpret_cast<int32_t *>(take(um * NG * 4));
    w.arrive = reinterpret_cast<int32_t *>(take(2 * um * NG * 4));
    for (int b = 0; b < 3; ++b)
        w.buf[b] = reinterpret_cast<Piece *>(take((size_t)(entries + NG * m) * sizeof(Piece)));
    return o;
}

}  // namespace

size_t solpath_bytes(int64_t m, int64_t entries) {
    SolWs w;
    return sol_layout(m, entries, nullptr, w);
}

template <typename T>
cudaError_t launch_solpath(int64_t m, const int64_t *off, const int32_t *len, const double *lam,
                           const T *val, const double *res, unsigned char *ws, int64_t entries,
                           double *out_start, int32_t *out_jhat, double *out_I, double *out_s,
                           T *out_v, int64_t *out_count, int64_t cap, cudaStream_t st,
                           int &launches) {
    SolWs w;
    sol_layout(m, entries, ws, w);
    cudaError_t e;
    if ((e = cudaMemsetAsync(w.h, 0, sizeof(SolHead), st)) != cudaSuccess) return e;
    k_zrange<T><<<(unsigned)m, 256, 0, st>>>(m, off, len, lam, val, res, w);
    k_zeval<T><<<(unsigned)m, EVT, 0, st>>>(m, off, len, lam, val, res, w);
    k_zbest<<<NG, 256, 0, st>>>(m, w);
    k_zsurvive<T><<<(unsigned)((m + 7) / 8), 256, 0, st>>>(m, w);
    k_zlist<<<1, ZL, 0, st>>>(m, w);
    launches += 5;
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    constexpr size_t smem = std::max(sizeof(BuildSmem), sizeof(MergeSmem));
    auto kern = k_zbuild<T>;
    if ((e = ensure_smem(reinterpret_cast<const void *>(kern), smem)) != cudaSuccess) return e;
    int dev = 0, sms = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
        return e;
    // two CTAs fit an SM; more units than that take turns
    const int64_t units = std::min<int64_t>(NG * m, 2 * (int64_t)sms);
    kern<<<(unsigned)units, ZT, smem, st>>>(m, off, len, lam, val, res, w);
    k_solution_out<<<64, 256, 0, st>>>(w, cap, out_start, out_jhat, out_I, out_s, out_count);
    launches += 2;
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (out_v) {
        const int64_t blocks = std::min<int64_t>((cap + VB - 1) / VB, 4096);
        k_solution_v<T><<<(unsigned)blocks, VT, 0, st>>>(m, cap, w, off, len, lam, val, out_v);
        launches++;
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template cudaError_t launch_solpath<float>(int64_t, const int64_t *, const int32_t *,
                                           const double *, const float *, const double *,
                                           unsigned char *, int64_t, double *, int32_t *,
                                           double *, double *, float *, int64_t *, int64_t,
                                           cudaStream_t, int &);
template cudaError_t launch_solpath<double>(int64_t, const int64_t *, const int32_t *,
                                            const double *, const double *, const double *,
                                            unsigned char *, int64_t, double *, int32_t *,
                                            double *, double *, double *, int64_t *, int64_t,
                                            cudaStream_t, int &);

L1L_CHECKS_READER(l1l_checks_solpath)

}  // namespace l1l
