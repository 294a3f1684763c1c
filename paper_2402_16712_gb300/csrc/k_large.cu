// k_large.cu -- steps A2-A4 (ratios, exact weighted median of Lemma 1,
// per-pair residual of Algorithm 1) for n beyond what the pair kernel holds
// in shared memory.
//
// The pair kernel stages column jhat in shared memory, which bounds n.  Here
// every (lambda, jhat, k) is solved by a cluster of C CTAs that stream the two
// columns from the staged column-major copy in global memory (L2-resident for
// moderate m), each CTA over its own slice of the rows:
//
//   sample   the ratios of 1024 rows, sorted with their weights, bracket the
//            median (12% of the weight either side);
//   bins     one pass: the exact fixed-point weight (the pair kernel's q_i) of
//            the rows below the bracket and, for those inside, of each of 1024
//            equal steps of the approximate ratio x_ik * (1 / x_ijhat).  The
//            CTAs of the cluster read each other's sums through distributed
//            shared memory and every CTA finds the same crossing bin;
//   rows     one pass: the rows whose approximate ratio lies within the guard
//            band of that bin (a few hundred) are divided exactly, and the
//            smallest exact key that passes the Decide test is the median.  As
//            in the pair kernel's selection no step before has to be trusted:
//            the rows' weights must add up to the bin's, and the weight below
//            must fail the test.
//   keys     more rows there than the list holds (from some 5 million rows on), or a
//            sample that is dense around the median (ties, nearly collinear columns;
//            in place of bins and rows): the smallest and largest exact key of the
//            rows next to it, and if these differ passes that histogram the weights
//            of the rows between by 2048 equal steps of the key, one or two for float.
//   descent  what that cannot settle (a wide column, few valid rows): a
//            radix descent over the order-preserving key of the correctly
//            rounded ratio r_i = x_ik / x_ijhat, 11 key bits per pass (float:
//            3 passes, double: 6).  A pass histograms the weights of the rows
//            whose key lies in the surviving range by its next digit; every CTA
//            takes the same decision from the cluster's totals, and the first
//            bin at which "weight at or below t exceeds W/2" (penalty point (0,
//            lambda) included) becomes true is kept.  After the last digit the
//            surviving key is the median itself.
//   residual sum_i |x_ik - v x_ijhat| over the rows (float input: runs of 32
//            terms in float, the runs in double; double input: double), a
//            fixed reduction order per CTA, then rank order over the cluster;
//            C depends on n only, so results do not depend on m or on the
//            number of lambdas.
//
// A row costs the bins pass a reciprocal and ~20 further instructions, the rows
// pass ~8, against a division, a 64-bit weight and a key compare in each pass of
// the descent (~60): 1,000,000 x 16 float 2.48 -> 1.14 ms.
// A decision the truncated weights cannot settle lists the pair for the exact
// wide-accumulator path, as in the pair kernel.  Control flow depends only on
// the pair index and on values every CTA of a cluster computes identically,
// so all CTAs meet every cluster barrier.
#include <cooperative_groups.h>

#include <algorithm>

#include "checks.cuh"
#include "common.cuh"
#include "launch.h"
#include "pairs.cuh"

namespace cg = cooperative_groups;

namespace l1l {

constexpr int LG_NT = 512;                // threads per CTA
constexpr int LG_BITS = 11;               // key bits per pass (at most)
constexpr int LG_NB = 1 << LG_BITS;       // histogram bins
constexpr int LG_BPT = LG_NB / LG_NT;     // bins per thread in the scan
constexpr int LG_COPIES = 4;              // privatised histogram copies per CTA
constexpr int LG_MAXC = 8;                // CTAs per cluster (portable limit)
constexpr int64_t LG_ROWS_PER_CTA = 65536;  // rows of one CTA before the cluster grows

// Shift of the lowest key bit of pass l (digits of 11 bits from the top, the
// last two of 10 bits for double keys, the last one for float keys).
template <typename T> struct LgDigits;
template <> struct LgDigits<float> {
    static constexpr int levels = 3;
    static __device__ __forceinline__ int shift(int l) { return l == 0 ? 21 : (l == 1 ? 10 : 0); }
};
template <> struct LgDigits<double> {
    static constexpr int levels = 6;
    static __device__ __forceinline__ int shift(int l) {
        return l < 4 ? 53 - 11 * l : (l == 4 ? 10 : 0);
    }
};

// Two rows per 8-byte word / four per 16-byte word: the vector of one load.
template <typename T> struct LgVec;
template <> struct LgVec<float> {
    using V = float4;
    static constexpr int W = 4;
    static __device__ __forceinline__ void get(const V &v, float *o) {
        o[0] = v.x;
        o[1] = v.y;
        o[2] = v.z;
        o[3] = v.w;
    }
};
template <> struct LgVec<double> {
    using V = double2;
    static constexpr int W = 2;
    static __device__ __forceinline__ void get(const V &v, double *o) {
        o[0] = v.x;
        o[1] = v.y;
    }
};

enum : int { LG_SEARCH = 0, LG_FOUND = 1, LG_EXACT = 2, LG_NONE = 3, LG_INTERNAL = 4 };

template <typename K> struct LgDecision {
    K prefix;        // key bits decided so far
    int64_t sbelow;  // weight of valid rows whose key lies below the surviving range
    int state;
    int first;       // first bin whose test is not "false" (LG_NB: none)
};

constexpr int LG_NS = 1024;    // sampled rows
constexpr int LG_BINS = 1024;  // bins of the bracket
constexpr int LG_SIDE = 8;     // bins kept free either side of it
constexpr int LG_ROWS = 1024;  // rows divided exactly, at most
constexpr float LG_HALF = 0.12f;  // sampled weight either side of the crossing
// Weights of up to 46 bits are summed as two halves of at most 23 bits, 512
// rows at a time in 32 bits.
constexpr int LG_QBITS = 46;
constexpr int LG_FLUSH = 128;  // vectors of four rows

// The bracket search's arrays, in the space of the descent's histograms.
template <typename T> struct LgPick {
    using K = typename Traits<T>::K;
    float key[LG_NS], w[LG_NS];            // the sample
    uint32_t hi[LG_BINS], lo[LG_BINS];     // this CTA's bins, upper and lower halves
    K akey[LG_ROWS + 1];                   // the cluster's rows
    long long aq[LG_ROWS + 1];
    K lkey[LG_ROWS];                       // this CTA's rows, read by the cluster
    long long lq[LG_ROWS];
    int lcnt;                              // their number (read by the cluster)
    long long lsum[3];                     // in the bin, under it, below the range
    int gcnt[LG_MAXC];                     // every CTA's lcnt and sums, copied here
    long long gsum[3][LG_MAXC];
    int j1, ia, ib, first;
    long long fl, fw;                      // weight before the crossing bin, its own
    float wsumf[LG_NT / 32];
    long long wsum[3][LG_NT / 32];
    K kmin;
    int und;
    K kmn[3], kmx[3];                      // large_keys: of each part (read by the cluster);
    uint32_t klo, khi, clo, chi;           // their range, and the middle one's
};

template <typename T> struct LgSmem {
    using K = typename Traits<T>::K;
    unsigned long long copies[LG_COPIES][LG_NB];  // this CTA's histogram copies
    unsigned long long tot[2][LG_NB];             // their sum, read by the cluster
    double part[2];                               // residual partial, read by rank 0
    long long wsum[LG_NT / 32];                   // scan: warp totals
    double wres[LG_NT / 32];                      // residual: warp partials
    LgDecision<K> dec;
};

// floor(w 2^sigma) as hi 2^b + lo.  Float: w 2^(sigma - b) < 2^23, so adding
// 2^23 rounding down leaves its floor in the mantissa, and the remainder, exact,
// the same way.  up: 2^(sigma - b), dn: 2^b.
__device__ __forceinline__ void split_q(float w, int, int, float up, float dn, uint32_t &hi,
                                        uint32_t &lo) {
    const float t = w * up;
    const float m1 = __fadd_rz(t, Z32);
    const float m2 = __fmaf_rz(t - (m1 - Z32), dn, Z32);
    hi = __float_as_uint(m1) - Z32_BITS;
    lo = __float_as_uint(m2) - Z32_BITS;
}
__device__ __forceinline__ void split_q(double w, int sigma, int b, float, float, uint32_t &hi,
                                        uint32_t &lo) {
    int e = 0;
    const uint64_t q = (uint64_t)fixq(w, sigma, e);
    hi = (uint32_t)(q >> b);
    lo = (uint32_t)q & ((1u << b) - 1u);
}

// One row of the bins pass: its weight to the sum below (z < 2^23) or to the sum
// inside and to bin z - 2^23 (z < 2^23 + LG_BINS), whose upper half lies at
// shared address hb + 4 (bits of z), its lower half LG_BINS words further; NaN is
// neither.  Predicated throughout: as branches the row cost twice as much.
__device__ __forceinline__ void lg_bin(float z, uint32_t qh, uint32_t ql, uint32_t hb,
                                       uint32_t &bh, uint32_t &bl, uint32_t &ih, uint32_t &il) {
    static_assert(LG_BINS == 1024, "the PTX below holds 2^23 + LG_BINS and 4 LG_BINS");
#if L1L_CHECKS
    if (z < Z32) {
        bh += qh;
        bl += ql;
    } else if (z < Z32 + (float)LG_BINS) {
        (void)L1L_CHK((int)(__float_as_uint(z) - Z32_BITS), LG_BINS);
#else
    {
#endif
        asm volatile(
            "{\n\t"
            ".reg .pred pb, pc;\n\t"
            ".reg .b32 a, zb;\n\t"
            "setp.lt.f32 pb, %4, 0f4B000000;\n\t"
            "setp.lt.and.f32 pc, %4, 0f4B000400, !pb;\n\t"
            "@pb add.u32 %0, %0, %5;\n\t"
            "@pb add.u32 %1, %1, %6;\n\t"
            "@pc add.u32 %2, %2, %5;\n\t"
            "@pc add.u32 %3, %3, %6;\n\t"
            "mov.b32 zb, %4;\n\t"
            "shl.b32 a, zb, 2;\n\t"
            "add.u32 a, a, %7;\n\t"
            "@pc red.shared.add.u32 [a], %5;\n\t"
            "@pc red.shared.add.u32 [a + 4096], %6;\n\t"
            "}"
            : "+r"(bh), "+r"(bl), "+r"(ih), "+r"(il)
            : "f"(z), "r"(qh), "r"(ql), "r"(hb)
            : "memory");
    }
}

// U vectors of four rows of the two columns, LG_NT apart, loaded together (the
// passes are bound by the latency of these loads from L2); rows from `end` on
// are 0.  w: the weights, in the input's type.
template <typename T, int U> struct LgRows {
    float4 vb[U], va[U];
    double2 d0[sizeof(T) == 8 ? U : 1], d1[sizeof(T) == 8 ? U : 1];
    __device__ __forceinline__ void get(int g, const float *fj, const float *fk, const T *xj,
                                        int64_t p) {
        vb[g] = __ldg(reinterpret_cast<const float4 *>(fj) + p);
        va[g] = __ldg(reinterpret_cast<const float4 *>(fk) + p);
        if constexpr (sizeof(T) == 8) {
            d0[g] = __ldg(reinterpret_cast<const double2 *>(xj) + 2 * p);
            d1[g] = __ldg(reinterpret_cast<const double2 *>(xj) + 2 * p + 1);
        }
    }
    __device__ __forceinline__ void load(const float *fj, const float *fk, const T *xj, int64_t v,
                                         int64_t end) {
        if (v + (U - 1) * LG_NT < end) {  // all but the last step
#pragma unroll
            for (int g = 0; g < U; ++g) get(g, fj, fk, xj, v + g * LG_NT);
            return;
        }
#pragma unroll
        for (int g = 0; g < U; ++g) {
            vb[g] = va[g] = make_float4(0.f, 0.f, 0.f, 0.f);
            if constexpr (sizeof(T) == 8) d0[g] = d1[g] = make_double2(0.0, 0.0);
            if (v + g * LG_NT < end) get(g, fj, fk, xj, v + g * LG_NT);
        }
    }
    static __device__ __forceinline__ float at(const float4 &v, int u) {
        return u == 0 ? v.x : (u == 1 ? v.y : (u == 2 ? v.z : v.w));
    }
    __device__ __forceinline__ float b(int g, int u) const { return at(vb[g], u); }
    __device__ __forceinline__ float a(int g, int u) const { return at(va[g], u); }
    __device__ __forceinline__ T w(int g, int u) const {
        if constexpr (sizeof(T) == 4)
            return b(g, u);
        else
            return u == 0 ? d0[g].x : (u == 1 ? d0[g].y : (u == 2 ? d1[g].x : d1[g].y));
    }
};
constexpr int LG_UB = 2;  // vectors in flight per thread: bins pass (4 spill),
constexpr int LG_UR = 4;  // rows pass and residual

// The block's sum of one value per thread, for every thread.
__device__ __forceinline__ long long lg_sum(long long x, long long *ws) {
    x = warp_sum_i64(x);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = x;
    __syncthreads();
    long long r = 0;
    for (int w = 0; w < LG_NT / 32; ++w) r += ws[w];
    return r;
}

// A key into the CTA's smallest and largest.
template <typename T>
__device__ __forceinline__ void lg_min_max(LgPick<T> &pk, int part, typename Traits<T>::K k) {
    using K = typename Traits<T>::K;
    if (k < *(volatile K *)&pk.kmn[part]) smem_min(&pk.kmn[part], k);
    if (k > *(volatile K *)&pk.kmx[part]) smem_max(&pk.kmx[part], k);
}

// The median among the rows with a coarse key in [lo, hi] by their exact keys, LG_SEARCH
// where it lies elsewhere.  listed: as the last step of the rows pass, whose list they
// exceed: L is their exact weight below and at least `thr` lies at or below hi.  Else a
// pass sums the weights below, and of those under, in and over [pk.clo, pk.chi].
// k_large, 100,000 and 1,000,000 x 6 float: small integers 194 -> 80, 670 -> 229 us (by a
// bracket that does not serve and the descent), multiples of one column 296 -> 229, 973 ->
// 639 us; continuous, 8,000,000 x 4, 2.66 -> 0.80 ms.
template <typename T>
__device__ __noinline__ int large_keys(int sigma, const Decide &dec, const float *fj,
                                       const float *fk, const T *xj, const T *xk, int64_t c0,
                                       int64_t c1, uint32_t lo, uint32_t hi, bool listed,
                                       long long L, long long thr, LgSmem<T> &sm, int &buf,
                                       typename Traits<T>::K &key) {
    using Tr = Traits<T>;
    using K = typename Tr::K;
    constexpr uint32_t G = Approx<T>::G;
    cg::cluster_group cl = cg::this_cluster();
    const int C = (int)cl.num_blocks();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    LgPick<T> &pk = *reinterpret_cast<LgPick<T> *>(&sm.copies[0][0]);
    // rows that |fma(x, 1/b, -cen)| < delta does not flag lie outside [lo, hi]
    const float va = akey_value(sat_sub(lo, G)), vb = akey_value(sat_add(hi, G));
    const float cen = 0.5f * va + 0.5f * vb;
    const float delta = (0.5f * vb - 0.5f * va) * (1.0f + 0x1p-20f) +
                        0x1p-21f * fmaxf(fabsf(va), fabsf(vb)) + 0x1p-148f;
    if (!(delta < 0x1p126f) || !(fabsf(cen) < 0x1p126f)) return LG_SEARCH;
    K A = Tr::NONE, B = 0;
    if (listed) {
        for (int e = tid; e < min(pk.lcnt, LG_ROWS); e += LG_NT) lg_min_max(pk, 0, pk.lkey[e]);
        cl.sync();
        for (int r = 0; r < C; ++r) {
            const LgPick<T> *o = cl.map_shared_rank(&pk, r);
            A = o->kmn[0] < A ? o->kmn[0] : A;
            B = o->kmx[0] > B ? o->kmx[0] : B;
        }
        cl.sync();  // the histograms overlap what the cluster read
        if (lo <= CK0 && CK0 <= hi) {  // the penalty point
            A = Tr::KEY0 < A ? Tr::KEY0 : A;
            B = Tr::KEY0 > B ? Tr::KEY0 : B;
        }
    } else {
        const uint32_t clo = pk.clo, chi = pk.chi;
        if (tid < 3) {  // the penalty point among them
            const bool zero = lo <= CK0 && CK0 <= hi && tid == (CK0 < clo ? 0 : (CK0 <= chi ? 1 : 2));
            pk.kmn[tid] = zero ? Tr::KEY0 : Tr::NONE;
            pk.kmx[tid] = zero ? Tr::KEY0 : 0;
        }
        __syncthreads();
        long long below = 0, part[3] = {0, 0, 0};
        for (int64_t v = c0 + tid; v < c1; v += LG_UB * LG_NT) {
            LgRows<T, LG_UB> x;
            x.load(fj, fk, xj, v, c1);
#pragma unroll
            for (int g = 0; g < LG_UB; ++g)
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const T b = x.w(g, u);
                    const float z = __fmaf_rn(x.a(g, u), rcp_approx(x.b(g, u)), -cen);
                    int e = 0;
                    if (fabsf(z) < delta) {  // b != 0: else z is infinite or NaN
                        const K k = Tr::key(Tr::div_rn(xk[4 * (v + g * LG_NT) + u], b));
                        const uint32_t ck = coarse_of<T>(k);
                        const long long q = fixq(fabs(b), sigma, e);
                        if (ck < lo) below += q;
                        if (ck >= lo && ck <= hi) {
                            const int p = ck < clo ? 0 : (ck <= chi ? 1 : 2);
#pragma unroll
                            for (int r = 0; r < 3; ++r) part[r] += p == r ? q : 0;
                            lg_min_max(pk, p, k);
                        }
                    } else if (z <= -delta) {
                        below += fixq(fabs(b), sigma, e);
                    }
                }
        }
        below = lg_sum(below, pk.wsum[0]);
#pragma unroll
        for (int r = 0; r < 3; ++r) part[r] = lg_sum(part[r], pk.wsum[r]);
        if (tid == 0) {
            sm.tot[buf][0] = (unsigned long long)below;
            for (int r = 0; r < 3; ++r) sm.tot[buf][r + 1] = (unsigned long long)part[r];
        }
        cl.sync();
        long long t[4] = {0, 0, 0, 0};
        K mn[3] = {Tr::NONE, Tr::NONE, Tr::NONE}, mx[3] = {0, 0, 0};
        for (int r = 0; r < C; ++r) {
            const LgPick<T> *o = cl.map_shared_rank(&pk, r);
            const unsigned long long *ot = cl.map_shared_rank(&sm.tot[buf][0], r);
#pragma unroll
            for (int p = 0; p < 4; ++p) t[p] += (long long)ot[p];
#pragma unroll
            for (int p = 0; p < 3; ++p) {
                mn[p] = o->kmn[p] < mn[p] ? o->kmn[p] : mn[p];
                mx[p] = o->kmx[p] > mx[p] ? o->kmx[p] : mx[p];
            }
        }
        buf ^= 1;
        cl.sync();  // the histograms overlap what the cluster read
        thr = t[0];
        int res = dec.cond(thr, lo > CK0);
        if (res != 0) return LG_SEARCH;
#pragma unroll
        for (int p = 0; p < 3; ++p)
            if (res == 0 && mn[p] <= mx[p]) {  // the first part whose last key passes
                L = thr;
                thr += t[p + 1];
                A = mn[p];
                B = mx[p];
                res = dec.cond(thr, B >= Tr::KEY0);
            }
        if (res == 0) return LG_SEARCH;
        if (res < 0) return LG_EXACT;
    }
    if (!(A <= B) || (listed && dec.cond(L, lo > CK0) != 0)) return LG_SEARCH;
    if (A == B && dec.cond(thr, A >= Tr::KEY0) == 1) {  // a tie, the only key there
        key = A;
        return LG_FOUND;
    }
    for (int pass = 0; pass < 6; ++pass) {
        const K span = B - A;
        int sh = 0;
        if (span >= (K)LG_NB)
            sh = (sizeof(K) == 4 ? 32 - __clz((int)span) : 64 - __clzll((long long)span)) - LG_BITS;
        for (int b = tid; b < LG_COPIES * LG_NB; b += LG_NT) (&sm.copies[0][0])[b] = 0ull;
        if (tid == 0) sm.dec.first = LG_NB;
        __syncthreads();
        unsigned long long *cp = sm.copies[warp % LG_COPIES];
        int cur = -1;
        unsigned long long csum = 0;
        for (int64_t v = c0 + tid; v < c1; v += LG_UR * LG_NT) {
            LgRows<float, LG_UR> x;
            x.load(fj, fk, fj, v, c1);
            uint32_t hit = 0;
#pragma unroll
            for (int g = 0; g < LG_UR; ++g)
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (fabsf(__fmaf_rn(x.a(g, u), rcp_approx(x.b(g, u)), -cen)) < delta)
                        hit |= 1u << (4 * g + u);
            for (; hit; hit &= hit - 1) {
                const int bit = __ffs(hit) - 1;
                const int64_t i = 4 * (v + (bit >> 2) * LG_NT) + (bit & 3);
                const T b = xj[i];
                if (b == T(0)) continue;
                const K k = Tr::key(Tr::div_rn(xk[i], b));
                if (k < A || k > B) continue;
                int e = 0;
                const unsigned long long q = (unsigned long long)fixq(fabs(b), sigma, e);
                const int bin = L1L_CHK((int)((k - A) >> sh), LG_NB);
                if (bin != cur) {
                    if (cur >= 0) atomicAdd(&cp[cur], csum);
                    cur = bin;
                    csum = 0;
                }
                csum += q;
            }
        }
        if (cur >= 0) atomicAdd(&cp[cur], csum);
        __syncthreads();
        for (int b = tid; b < LG_NB; b += LG_NT) {
            unsigned long long t = 0;
#pragma unroll
            for (int c = 0; c < LG_COPIES; ++c) t += sm.copies[c][b];
            sm.tot[buf][b] = t;
        }
        cl.sync();  // every CTA's totals are complete and visible
        long long h[LG_BPT], run = 0;
#pragma unroll
        for (int u = 0; u < LG_BPT; ++u) {
            unsigned long long t = 0;
            for (int r = 0; r < C; ++r)
                t += cl.map_shared_rank(&sm.tot[buf][0], r)[tid * LG_BPT + u];
            h[u] = (long long)t;
            run += h[u];
        }
        buf ^= 1;
        const long long incl = warp_scan_add(run, lane);
        if (lane == 31) sm.wsum[warp] = incl;
        __syncthreads();
        long long acc = L + incl - run;
        for (int w = 0; w < warp; ++w) acc += sm.wsum[w];
        // first bin whose test at its last key is true or undecidable
        int mine = LG_NB, mine_res = 0;
        long long mine_below = 0;
#pragma unroll
        for (int u = 0; u < LG_BPT; ++u) {
            const int b = tid * LG_BPT + u;
            const long long below = acc;
            acc += h[u];
            if (mine == LG_NB && (K)b <= span >> sh) {
                const K first = A + ((K)b << sh), in = ((K)1 << sh) - 1;
                const K last = B - first < in ? B : first + in;
                const int res = dec.cond(acc, last >= Tr::KEY0);
                if (res != 0) {
                    mine = b;
                    mine_res = res;
                    mine_below = below;
                }
            }
        }
        if (mine < LG_NB) atomicMin(&sm.dec.first, mine);
        __syncthreads();
        if (mine < LG_NB && mine == sm.dec.first) {
            sm.dec.sbelow = mine_below;
            sm.dec.state = mine_res;
        }
        __syncthreads();
        const int first = sm.dec.first;
        if (first == LG_NB) return LG_SEARCH;
        const int res = sm.dec.state;
        L = sm.dec.sbelow;
        __syncthreads();  // sm.dec is rewritten by the next pass
        if (res < 0) return LG_EXACT;
        A += (K)first << sh;
        if (sh == 0) {
            key = A;
            return LG_FOUND;
        }
        const K in = ((K)1 << sh) - 1;
        B = B - A < in ? B : A + in;
    }
    return LG_SEARCH;
}

// The weighted median of a pair by the cluster: LG_FOUND with its key, LG_EXACT
// where the weights cannot settle it, LG_SEARCH where the descent has to look.
// Every CTA returns the same.  c0, c1: this CTA's rows in vectors of four.
template <typename T>
__device__ int large_pick(const ScanArgs<T> &a, const ColInfo &ci, int64_t j, int64_t k,
                          const Decide &dec, int64_t c0, int64_t c1, LgSmem<T> &sm, int &buf,
                          typename Traits<T>::K &key) {
    using Tr = Traits<T>;
    using K = typename Tr::K;
    constexpr uint32_t G = Approx<T>::G;
    cg::cluster_group cl = cg::this_cluster();
    const int C = (int)cl.num_blocks();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t n = a.n, ldn = a.ldn;
    // what the split and the approximate ratio need (else: the descent)
    const int qbits = 61 - (32 - __clz(ci.n_valid));
    const int qb = (qbits + 1) / 2, es = ci.sigma - qb;
    if (qbits > LG_QBITS || (ci.flags & COL_WIDE) || es < -120 || es > 120 ||
        (sizeof(T) == 8 && (a.ci[k].flags & COL_WIDE)))
        return LG_SEARCH;
    const float up = __int_as_float((127 + es) << 23), dn = __int_as_float((127 + qb) << 23);
    static_assert(sizeof(LgPick<T>) <= sizeof(sm.copies), "the descent's histograms hold it");
    LgPick<T> &pk = *reinterpret_cast<LgPick<T> *>(&sm.copies[0][0]);
    const T *xj = a.Xt + j * ldn, *xk = a.Xt + k * ldn;
    const float *fj = a.Xf + j * ldn, *fk = a.Xf + k * ldn;

    // ---- sample: the same rows and the same arithmetic in every CTA ----
    for (int s = tid; s < LG_NS; s += LG_NT) {
        const int64_t i = (int64_t)(2 * s + 1) * n / (2 * LG_NS);
        const float xb = fj[i];
        const float r = fk[i] * rcp_approx(xb);
        pk.key[s] = xb != 0.0f ? r : INFINITY;
        pk.w[s] = fabsf(xb);
    }
    if (tid == 0) pk.j1 = pk.ia = pk.ib = LG_NS - 1;
    for (int size = 2; size <= LG_NS; size <<= 1)
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            __syncthreads();
            for (int t = tid; t < LG_NS / 2; t += LG_NT) {
                const int i = 2 * t - (t & (stride - 1)), o = i + stride;
                const float x = pk.key[i], y = pk.key[o];
                if ((x > y) == ((i & size) == 0)) {
                    pk.key[i] = y;
                    pk.key[o] = x;
                    const float u = pk.w[i];
                    pk.w[i] = pk.w[o];
                    pk.w[o] = u;
                }
            }
        }
    __syncthreads();
    float a0, b0;
    {
        static_assert(LG_NS == 2 * LG_NT, "two samples per thread");
        const float w0 = pk.w[2 * tid], w1 = pk.w[2 * tid + 1];
        const float incl = warp_scan_add(w0 + w1, lane);
        if (lane == 31) pk.wsumf[warp] = incl;
        __syncthreads();
        float before = 0.0f, total = 0.0f;
        for (int w = 0; w < LG_NT / 32; ++w) {
            if (w == warp) before = total;
            total += pk.wsumf[w];
        }
        const float cum1 = before + incl, cum0 = cum1 - w1;
        const float per = total / (float)dec.Q;
        const float tpos = 0.5f * per * (float)(dec.Q - dec.Lc);
        const float tneg = 0.5f * per * (float)(dec.Q + dec.Lf);
        auto passes = [&](float cum, float x) { return cum >= (x >= 0.0f ? tpos : tneg); };
        if (passes(cum0, pk.key[2 * tid]))
            atomicMin(&pk.j1, 2 * tid);
        else if (passes(cum1, pk.key[2 * tid + 1]))
            atomicMin(&pk.j1, 2 * tid + 1);
        __syncthreads();
        if (pk.j1 == 2 * tid) pk.wsumf[0] = cum0;
        if (pk.j1 == 2 * tid + 1) pk.wsumf[0] = cum1;
        __syncthreads();
        const float mid = pk.wsumf[0];
        const float ta = mid - LG_HALF * total, tb = mid + LG_HALF * total;
        if (cum0 >= ta)
            atomicMin(&pk.ia, 2 * tid);
        else if (cum1 >= ta)
            atomicMin(&pk.ia, 2 * tid + 1);
        if (cum0 >= tb)
            atomicMin(&pk.ib, 2 * tid);
        else if (cum1 >= tb)
            atomicMin(&pk.ib, 2 * tid + 1);
        __syncthreads();
        a0 = pk.key[max(pk.ia - 1, 0)];
        b0 = pk.key[pk.ib];
    }
    auto keys = [&](uint32_t klo, uint32_t khi, bool listed, long long L, long long thr) -> int {
        const Decide dk = dec;  // in memory from here on, as the others
        int bk = buf;
        K kk = 0;
        const int st = large_keys<T>(ci.sigma, dk, fj, fk, xj, xk, c0, c1, klo, khi, listed, L,
                                     thr, sm, bk, kk);
        buf = bk;
        key = kk;
        return st;
    };
    // Five of the samples up to 48 (three deviations of the crossing) either side within
    // 64 coarse keys: ties or nearly collinear columns, of which the bins below would
    // hold more rows than their halves sum (512).  Looked at by exact keys instead, those
    // at the crossing apart from those under and over them.
    {
        const int j0 = max(max(pk.ia - 1, pk.j1 - 48), 0), j2 = min(pk.ib, pk.j1 + 48);
        const int t = j0 + tid;
        const bool run = t + 4 <= j2 && pk.key[t + 4] < INFINITY &&
                         akey(pk.key[t + 4]) - akey(pk.key[t]) <= 64u;
        if (__syncthreads_or(run)) {
            if (tid == 0) {
                auto at = [&](int i) { return akey(pk.key[i]); };
                int e = j2, p = pk.j1, q = pk.j1;
                while (e > pk.j1 && pk.key[e] == INFINITY) --e;  // x_ijhat = 0
                while (p > j0 && at(p) - at(p - 1) <= 64u) --p;
                while (q < e && at(q + 1) - at(q) <= 64u) ++q;
                pk.klo = sat_sub(at(j0), G + 4);
                pk.khi = sat_add(at(e), G + 4);
                pk.clo = max(pk.klo, sat_sub(at(p), G + 4));
                pk.chi = min(pk.khi, sat_add(at(q), G + 4));
            }
            __syncthreads();
            const int st = keys(pk.klo, pk.khi, false, 0, 0);
            if (st != LG_SEARCH) return st;
            __syncthreads();
        }
    }

    for (int attempt = 0; attempt < 3; ++attempt) {
        // ---- bins: steps of w1, no finer than 16 keys of the largest ratio ----
        // (or 2^-99, where the whole bracket is 0: sparse columns)
        const float w1 = fmaxf((b0 - a0) * (1.0f / (LG_BINS - 2 * LG_SIDE)),
                               fmaxf(fmaxf(fabsf(a0), fabsf(b0)) * 0x1p-19f, 0x1p-99f));
        if (!(w1 < 0x1p100f)) return LG_SEARCH;
        const float sc = __frcp_rn(w1);
        const float bm = __fmaf_rn(-a0, sc, Z32 + (float)LG_SIDE);
        constexpr float ZT = Z32 + (float)LG_BINS;
        for (int b = tid; b < LG_BINS; b += LG_NT) pk.hi[b] = pk.lo[b] = 0;
        if (tid == 0) pk.first = LG_BINS;
        __syncthreads();
        long long Sb = 0, Sa = 0;  // below the bracket; inside it, then below its end
        const uint32_t hb = smem_addr(pk.hi) - 4u * Z32_BITS;
        for (int64_t v0 = c0 + tid; v0 < c1; v0 += (int64_t)LG_FLUSH * LG_NT) {
            const int64_t ve = std::min<int64_t>(c1, v0 + (int64_t)LG_FLUSH * LG_NT);
            uint32_t bh = 0, bl = 0, ih = 0, il = 0;
            for (int64_t v = v0; v < ve; v += LG_UB * LG_NT) {
                LgRows<T, LG_UB> x;
                x.load(fj, fk, xj, v, ve);
#pragma unroll
                for (int g = 0; g < LG_UB; ++g)
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        // x_ijhat = 0: the weight is 0, wherever the ratio falls
                        const float z = __fmaf_rn(__fmul_rn(x.a(g, u), rcp_approx(x.b(g, u))), sc, bm);
                        uint32_t qh, ql;
                        split_q(fabs(x.w(g, u)), ci.sigma, qb, up, dn, qh, ql);
                        lg_bin(z, qh, ql, hb, bh, bl, ih, il);
                    }
            }
            Sb += ((long long)bh << qb) + (long long)bl;
            Sa += ((long long)ih << qb) + (long long)il;
        }
        Sa += Sb;
        Sb = lg_sum(Sb, pk.wsum[0]);
        Sa = lg_sum(Sa, pk.wsum[1]);  // also: the bins are complete
        for (int b = tid; b < LG_BINS; b += LG_NT)
            sm.tot[buf][b] = ((unsigned long long)pk.hi[b] << qb) + pk.lo[b];
        if (tid == 0) {
            sm.tot[buf][LG_BINS] = (unsigned long long)Sb;
            sm.tot[buf][LG_BINS + 1] = (unsigned long long)Sa;
        }
        cl.sync();
        // ---- the crossing bin of the cluster's totals ----
        constexpr int Q = LG_BINS / LG_NT;
        long long h[Q], run = 0;
#pragma unroll
        for (int u = 0; u < Q; ++u) {
            unsigned long long x = 0;
            for (int r = 0; r < C; ++r) x += cl.map_shared_rank(&sm.tot[buf][0], r)[Q * tid + u];
            h[u] = (long long)x;
            run += h[u];
        }
        if (tid < C) {
            const unsigned long long *o = cl.map_shared_rank(&sm.tot[buf][0], tid);
            pk.gsum[0][tid] = (long long)o[LG_BINS];
            pk.gsum[1][tid] = (long long)o[LG_BINS + 1];
        }
        buf ^= 1;
        const long long incl = warp_scan_add(run, lane);
        if (lane == 31) pk.wsum[2][warp] = incl;
        __syncthreads();
        Sb = Sa = 0;
        for (int r = 0; r < C; ++r) {
            Sb += pk.gsum[0][r];
            Sa += pk.gsum[1][r];
        }
        long long cum = Sb + incl - run, all = 0;
        for (int w = 0; w < LG_NT / 32; ++w) {
            if (w < warp) cum += pk.wsum[2][w];
            all += pk.wsum[2][w];
        }
        if (all != Sa - Sb) return LG_SEARCH;  // a bin of one CTA left 32 bits
        const int zb = bm < Z32 ? 0 : (bm < ZT ? (int)(bm - Z32) : LG_BINS);
        const int64_t tneg = ((dec.Q + dec.Lf) >> 1) + 1, tpos = ((dec.Q - dec.Lc) >> 1) + 1;
        int mine = LG_BINS;
        long long ml = 0, mw = 0;
#pragma unroll
        for (int u = 0; u < Q; ++u) {
            const int b = Q * tid + u;
            if (mine == LG_BINS && cum + h[u] >= (b >= zb ? tpos : tneg)) {
                mine = b;
                ml = cum;
                mw = h[u];
            }
            cum += h[u];
        }
        if (mine < LG_BINS) atomicMin(&pk.first, mine);
        __syncthreads();
        const int ca = pk.first;
        if (mine == ca && mine < LG_BINS) {
            pk.fl = ml;
            pk.fw = mw;
        }
        if (tid == 0) {
            pk.lcnt = 0;
            pk.kmin = Tr::NONE;
            pk.und = 0;
            pk.kmn[0] = Tr::NONE;
            pk.kmx[0] = 0;
        }
        __syncthreads();
        if (ca < 1 || ca >= LG_BINS) {  // missed: further out on that side
            const float span = b0 - a0;
            if (ca < 1) {
                b0 = a0 + 2.0f * w1;
                a0 = a0 - 4.0f * fmaxf(span, 2.0f * w1);
            } else {
                a0 = b0 - 2.0f * w1;
                b0 = b0 + 4.0f * fmaxf(span, 2.0f * w1);
            }
            if (!(a0 < b0)) return LG_SEARCH;
            continue;
        }
        // ---- the coarse keys [lo, hi] around it (pair kernel's selection) ----
        const float ra = ((Z32 + (float)ca - bm) - 0.5f) * w1;
        const float rb = ((Z32 + (float)ca - bm) + 0.5f) * w1;
        const uint32_t ka = sat_sub(akey(ra), 2 * G + 4), kb = sat_add(akey(rb), 2 * G + 4);
        const float va = akey_value(ka), vb = akey_value(kb);
        if (!(va < vb)) return LG_SEARCH;
        const uint32_t lo = ka + G, hi = kb - G;
        const float cen = 0.5f * (va + vb);
        const float delta =
            0.5f * (vb - va) * (1.0f + 0x1p-20f) + 0x1p-21f * fmaxf(fabsf(va), fabsf(vb));
        long long in_w = 0, under_w = 0, below_w = 0;
        for (int64_t v = c0 + tid; v < c1; v += LG_UR * LG_NT) {
            LgRows<float, LG_UR> x;
            x.load(fj, fk, fj, v, c1);
            uint32_t hit = 0;
#pragma unroll
            for (int g = 0; g < LG_UR; ++g)
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (fabsf(__fmaf_rn(x.a(g, u), rcp_approx(x.b(g, u)), -cen)) < delta)
                        hit |= 1u << (4 * g + u);
            for (; hit; hit &= hit - 1) {
                const int bit = __ffs(hit) - 1;
                const int64_t i = 4 * (v + (bit >> 2) * LG_NT) + (bit & 3);
                const float b = fj[i], r = __fmul_rn(fk[i], rcp_approx(b));
                if (!(r >= va && r <= vb) || b == 0.0f) continue;
                int e = 0;
                const long long q = fixq(fabs(xj[i]), ci.sigma, e);
                const float z = __fmaf_rn(r, sc, bm);
                if (z < Z32 + (float)ca)
                    under_w += q;
                else if (z <= Z32 + (float)ca)
                    in_w += q;
                const K fkey = Tr::key(Tr::div_rn(xk[i], xj[i]));
                const uint32_t ck = coarse_of<T>(fkey);
                if (ck < lo) {
                    below_w += q;
                } else if (ck <= hi) {
                    // not counted on once the list is full: ties would queue for the count
                    const int at = *(volatile int *)&pk.lcnt > LG_ROWS ? LG_ROWS
                                                                       : atomicAdd(&pk.lcnt, 1);
                    if (at < LG_ROWS) {
                        pk.lkey[at] = fkey;
                        pk.lq[at] = q;
                    } else {
                        lg_min_max(pk, 0, fkey);
                    }
                }
            }
        }
        in_w = lg_sum(in_w, pk.wsum[0]);
        under_w = lg_sum(under_w, pk.wsum[1]);
        below_w = lg_sum(below_w, pk.wsum[2]);
        if (tid == 0) {
            pk.lsum[0] = in_w;
            pk.lsum[1] = under_w;
            pk.lsum[2] = below_w;
        }
        cl.sync();
        // ---- every CTA gathers the cluster's rows ----
        if (tid < C) {
            const LgPick<T> *o = cl.map_shared_rank(&pk, tid);
            pk.gcnt[tid] = o->lcnt;
            for (int q = 0; q < 3; ++q) pk.gsum[q][tid] = o->lsum[q];
        }
        __syncthreads();
        int c = 0;
        in_w = 0;
        long long L = pk.fl;
        for (int r = 0; r < C; ++r) {
            const LgPick<T> *o = cl.map_shared_rank(&pk, r);
            const int cr = pk.gcnt[r];
            in_w += pk.gsum[0][r];
            L += pk.gsum[2][r] - pk.gsum[1][r];
            for (int e = tid; e < cr && c + e < LG_ROWS; e += LG_NT) {
                pk.akey[c + e] = o->lkey[e];
                pk.aq[c + e] = o->lq[e];
            }
            c += cr;
        }
        const long long W = pk.fw, thr = pk.fl + W;
        cl.sync();  // the lists are free again
        if (in_w != W || dec.cond(L, lo > CK0) != 0) return LG_SEARCH;
        if (c > LG_ROWS) return keys(lo, hi, true, L, thr);
        if (lo <= CK0 && CK0 <= hi) {  // the penalty point; lambda sits in the test
            if (tid == 0) {
                pk.akey[c] = Tr::KEY0;
                pk.aq[c] = 0;
            }
            c += 1;
            __syncthreads();
        }
        for (int e = tid; e < c; e += LG_NT) {
            const K x = pk.akey[e];
            long long S = L;
            for (int q = 0; q < c; ++q) S += pk.akey[q] <= x ? pk.aq[q] : 0;
            const int res = dec.cond(S, x >= Tr::KEY0);
            if (res != 0) {
                if constexpr (sizeof(K) == 4)
                    atomicMin(&pk.kmin, x);
                else
                    atomicMin(reinterpret_cast<unsigned long long *>(&pk.kmin),
                              (unsigned long long)x);
            }
        }
        __syncthreads();
        key = pk.kmin;
        if (key == Tr::NONE) return LG_SEARCH;
        // equal keys have equal sums: any of them tells whether it was certain
        for (int e = tid; e < c; e += LG_NT)
            if (pk.akey[e] == key) {
                long long S = L;
                for (int q = 0; q < c; ++q) S += pk.akey[q] <= key ? pk.aq[q] : 0;
                if (dec.cond(S, key >= Tr::KEY0) < 0) pk.und = 1;
            }
        __syncthreads();
        return pk.und ? LG_EXACT : LG_FOUND;
    }
    return LG_SEARCH;
}

template <typename T>
__global__ void __launch_bounds__(LG_NT, 2)
    k_large(ScanArgs<T> a, const __grid_constant__ LambdaPack lp, int t0, int nlc,
            int64_t rows_per_cta) {
    using Tr = Traits<T>;
    using K = typename Tr::K;
    using VT = LgVec<T>;
    using V = typename VT::V;
    constexpr int VW = VT::W;
    constexpr int KB = Tr::KEY_BITS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LgSmem<T> &sm = *reinterpret_cast<LgSmem<T> *>(smem_raw);

    cg::cluster_group cl = cg::this_cluster();
    const int C = (int)cl.num_blocks();
    const int rank = (int)cl.block_rank();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t cid = blockIdx.x / C, ncl = gridDim.x / C;
    const int64_t m = a.m, nj = a.nj, ldn = a.ldn;
    const int64_t P = (int64_t)nlc * nj * m;
    // this CTA's rows [r0, r1), whole vectors (ldn and rows_per_cta are multiples of 128)
    const int64_t r0 = std::min<int64_t>(ldn, (int64_t)rank * rows_per_cta);
    const int64_t r1 = std::min<int64_t>(ldn, r0 + rows_per_cta);
    const int64_t v0 = r0 / VW, v1 = r1 / VW;
    int buf = 0;

    for (int64_t p = cid; p < P; p += ncl) {
        const int tl = (int)(p / (nj * m));
        const int64_t rem = p - (int64_t)tl * nj * m;
        const int64_t q = rem / m, k = rem - q * m;
        const int64_t j = a.jlist ? (int64_t)a.jlist[q] : q;
        const bool leader = rank == 0 && tid == 0;
        if (j < 0 || j >= m) {
            if (leader) atomicOr(a.status, ST_BADINDEX);
            continue;
        }
        const int t = t0 + tl;
        const double lam = lp.lam[tl];
        const int64_t o = L1L_CHK(((int64_t)t * m + j) * m + k, (int64_t)a.n_lambda * m * m);
        if (k == j) {  // v_jhat = 1: zero residual, penalty lambda * 1
            if (leader) {
                a.v_all[o] = T(1);
                a.s_all[o] = lam;
            }
            continue;
        }
        const ColInfo ci = a.ci[j];
        if (a.force_exact) {
            if (leader) {
                const uint32_t slot = atomicAdd(a.slow_count, 1u);
                a.slow[slot] = SlowEntry{t, (int32_t)j, (int32_t)k, (int16_t)a.inst,
                                         (int16_t)SEL_SLOW};
            }
            continue;
        }
        const V *xjv = reinterpret_cast<const V *>(a.Xt + j * ldn);
        const V *xkv = reinterpret_cast<const V *>(a.Xt + k * ldn);
        Decide dec;
        dec.init(ci, lam);

        K prefix = 0;
        int64_t sbelow = 0;
        int state = ci.n_valid > 0 ? LG_SEARCH : LG_NONE;  // no valid row: v = 0
        if (state == LG_SEARCH) {
            state = large_pick<T>(a, ci, j, k, dec, r0 / 4, r1 / 4, sm, buf, prefix);
            if (state == LG_SEARCH) {
                prefix = 0;
                cl.sync();  // the descent's histograms overlap what the cluster read
            }
            __syncthreads();
        }
        for (int l = 0; state == LG_SEARCH && l < LgDigits<T>::levels; ++l) {
            const int sh = LgDigits<T>::shift(l);
            const int top = l == 0 ? KB : LgDigits<T>::shift(l - 1);
            const int nbl = 1 << (top - sh);
            const K bmask = (K)(nbl - 1);
            const K pmask = top == KB ? (K)0 : ~(((K)1 << top) - 1);
            // ---- one pass: histogram of the surviving rows by this digit ----
            for (int b = tid; b < LG_COPIES * LG_NB; b += LG_NT) (&sm.copies[0][0])[b] = 0ull;
            if (tid == 0) sm.dec.first = LG_NB;
            __syncthreads();
            unsigned long long *cp = sm.copies[warp % LG_COPIES];
            int cur = -1;
            unsigned long long csum = 0;
            // the next vectors are loaded while the current ones are processed
            V nj{}, nk{};
            if (v0 + tid < v1) {
                nj = xjv[v0 + tid];
                nk = xkv[v0 + tid];
            }
            for (int64_t v = v0 + tid; v < v1; v += LG_NT) {
                T xb[VW], xa[VW];
                VT::get(nj, xb);
                VT::get(nk, xa);
                if (v + LG_NT < v1) {
                    nj = xjv[v + LG_NT];
                    nk = xkv[v + LG_NT];
                }
#pragma unroll
                for (int u = 0; u < VW; ++u) {
                    if (xb[u] == T(0)) continue;
                    const K kk = Tr::key(Tr::div_rn(xa[u], xb[u]));
                    if ((kk & pmask) != prefix) continue;
                    const int bin = (int)((kk >> sh) & bmask);
                    int inx = 0;
                    const unsigned long long w =
                        (unsigned long long)fixq(fabs(xb[u]), ci.sigma, inx);
                    if (bin == cur) {
                        csum += w;
                    } else {
                        if (cur >= 0 && csum) atomicAdd(&cp[cur], csum);
                        cur = bin;
                        csum = w;
                    }
                }
            }
            if (cur >= 0 && csum) atomicAdd(&cp[cur], csum);
            __syncthreads();
            for (int b = tid; b < LG_NB; b += LG_NT) {
                unsigned long long s = 0;
#pragma unroll
                for (int c = 0; c < LG_COPIES; ++c) s += sm.copies[c][b];
                sm.tot[buf][b] = s;
            }
            cl.sync();  // every CTA's totals are complete and visible
            // ---- the cluster's totals, scanned in bin order ----
            long long h[LG_BPT];
            long long run = 0;
#pragma unroll
            for (int u = 0; u < LG_BPT; ++u) {
                const int b = tid * LG_BPT + u;
                unsigned long long s = 0;
                for (int r = 0; r < C; ++r) s += cl.map_shared_rank(&sm.tot[buf][0], r)[b];
                h[u] = (long long)s;
                run += h[u];
            }
            long long incl = run;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const long long y = __shfl_up_sync(0xFFFFFFFFu, incl, off);
                if (lane >= off) incl += y;
            }
            if (lane == 31) sm.wsum[warp] = incl;
            __syncthreads();
            long long before = incl - run;  // weight of this CTA's earlier bins
            for (int w = 0; w < warp; ++w) before += sm.wsum[w];
            // first bin whose test is true or undecidable
            int mine = LG_NB, mine_res = 0;
            long long mine_below = 0;
            long long acc = before;
#pragma unroll
            for (int u = 0; u < LG_BPT; ++u) {
                const int b = tid * LG_BPT + u;
                const long long below = acc;
                acc += h[u];
                if (mine == LG_NB && b < nbl) {
                    const K full = prefix | ((K)b << sh);
                    const bool nonneg = ((full >> (KB - 1)) & 1) != 0;
                    const int res = dec.cond(sbelow + acc, nonneg);
                    if (res != 0) {
                        mine = b;
                        mine_res = res;
                        mine_below = below;
                    }
                }
            }
            if (mine < LG_NB) atomicMin(&sm.dec.first, mine);
            __syncthreads();
            if (mine < LG_NB && mine == sm.dec.first) {
                LgDecision<K> d;
                d.first = mine;
                d.prefix = prefix | ((K)mine << sh);
                d.sbelow = sbelow + mine_below;
                d.state = mine_res == 1 ? (l + 1 == LgDigits<T>::levels ? LG_FOUND : LG_SEARCH)
                                        : LG_EXACT;
                sm.dec = d;
            }
            __syncthreads();
            if (sm.dec.first == LG_NB) {
                // "true" at no key: W = 0 at the top level; below it the parent
                // bin's test was true at its last key, so this cannot happen
                state = l == 0 ? LG_NONE : LG_INTERNAL;
            } else {
                prefix = sm.dec.prefix;
                sbelow = sm.dec.sbelow;
                state = sm.dec.state;
            }
            buf ^= 1;
            __syncthreads();  // sm.dec is rewritten by the next pass
        }
        if (state == LG_EXACT) {
            if (leader) {
                const uint32_t slot = atomicAdd(a.slow_count, 1u);
                a.slow[slot] = SlowEntry{t, (int32_t)j, (int32_t)k, (int16_t)a.inst,
                                         (int16_t)SEL_SLOW_BAND};
            }
            continue;
        }
        if (state == LG_INTERNAL) {
            if (leader) {
                atomicOr(a.status, ST_INTERNAL);
                a.v_all[o] = T(NAN);
                a.s_all[o] = NAN;
            }
            continue;
        }
        const T vv = state == LG_FOUND ? Tr::value(prefix) : T(0);
        // ---- residual: sum_i |x_ik - v x_ijhat| ----
        // float input: terms summed in float over runs of 32 rows (a relative
        // error below 2^-19 of the run's sum), runs in double; double input:
        // every term in double
        double racc = 0.0;
        T run = T(0);
        int nrun = 0;
        for (int64_t v = v0 + tid; v < v1; v += LG_UR * LG_NT) {
            V vb[LG_UR], va[LG_UR];
            if (v + (LG_UR - 1) * LG_NT < v1) {
#pragma unroll
                for (int g = 0; g < LG_UR; ++g) {
                    vb[g] = xjv[v + g * LG_NT];
                    va[g] = xkv[v + g * LG_NT];
                }
            } else {
#pragma unroll
                for (int g = 0; g < LG_UR; ++g) {
                    vb[g] = va[g] = V{};
                    if (v + g * LG_NT < v1) {
                        vb[g] = xjv[v + g * LG_NT];
                        va[g] = xkv[v + g * LG_NT];
                    }
                }
            }
#pragma unroll
            for (int g = 0; g < LG_UR; ++g) {
                T xb[VW], xa[VW];
                VT::get(vb[g], xb);
                VT::get(va[g], xa);
                T t4 = T(0);
#pragma unroll
                for (int u = 0; u < VW; ++u) t4 += fabs(fma(-vv, xb[u], xa[u]));
                run += t4;
                if (++nrun == 32 / VW || sizeof(T) == 8) {
                    racc += (double)run;
                    run = T(0);
                    nrun = 0;
                }
            }
        }
        racc += (double)run;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) racc += __shfl_xor_sync(0xFFFFFFFFu, racc, off);
        if (lane == 0) sm.wres[warp] = racc;
        __syncthreads();
        if (tid == 0) {
            double s = 0.0;
            for (int w = 0; w < LG_NT / 32; ++w) s += sm.wres[w];
            sm.part[buf] = s;
        }
        cl.sync();  // every CTA's partial is visible
        if (rank == 0 && warp == 0) {  // read together, added in rank order
            const double x = cl.map_shared_rank(&sm.part[0], min(lane, C - 1))[buf];
            double s = 0.0;
            for (int r = 0; r < C; ++r) s += __shfl_sync(0xFFFFFFFFu, x, r);
            if (leader) {
                a.v_all[o] = vv;
                a.s_all[o] = s + lam * (double)fabs(vv);
            }
        }
        buf ^= 1;
    }
    cl.sync();  // no CTA leaves while another may still read its shared memory
}

int large_cluster_size(int64_t ldn) {
    const int64_t c = (ldn + LG_ROWS_PER_CTA - 1) / LG_ROWS_PER_CTA;
    return (int)std::max<int64_t>(1, std::min<int64_t>(LG_MAXC, c));
}

template <typename T>
cudaError_t launch_large(const ScanArgs<T> &a, const double *lambdas, int t0, int nlc,
                         cudaStream_t st, int &launches) {
    const int C = large_cluster_size(a.ldn);
    const int64_t rpc = ((a.ldn + C - 1) / C + ROW_PAD - 1) & ~int64_t(ROW_PAD - 1);
    const size_t smem = sizeof(LgSmem<T>);
    auto kern = k_large<T>;
    cudaError_t e = ensure_smem(reinterpret_cast<const void *>(kern), smem);
    if (e != cudaSuccess) return e;
    LambdaPack lp;
    lp.tl_min = lp.tl_max = 0;
    for (int q = 0; q < nlc; ++q) lp.lam[q] = lambdas[t0 + q];
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(LG_NT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cfg.gridDim = dim3((unsigned)C);
    int clusters = 0;
    e = cudaOccupancyMaxActiveClusters(&clusters, reinterpret_cast<const void *>(kern), &cfg);
    if (e != cudaSuccess) return e;
    if (clusters < 1) return cudaErrorInvalidConfiguration;
    const int64_t P = (int64_t)nlc * a.nj * a.m;
    const int64_t ncl = std::max<int64_t>(1, std::min<int64_t>(P, clusters));
    cfg.gridDim = dim3((unsigned)(ncl * C));
    e = cudaLaunchKernelEx(&cfg, kern, a, lp, t0, nlc, rpc);
    launches++;
    return e;
}

template cudaError_t launch_large<float>(const ScanArgs<float> &, const double *, int, int,
                                         cudaStream_t, int &);
template cudaError_t launch_large<double>(const ScanArgs<double> &, const double *, int, int,
                                          cudaStream_t, int &);

L1L_CHECKS_READER(l1l_checks_large)

}  // namespace l1l
