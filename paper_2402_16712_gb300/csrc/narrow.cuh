// narrow.cuh -- the weighted median of a pair among rows whose ratios lie too
// close together for the selection's bins: ties (rounded or count data, sparse
// columns), columns that are nearly multiples of one another, or a decision that
// needs the 64-bit weights.
//
// The median's coarse key is expected in [lo, hi].  One warp bins the rows there
// by their exact keys, 32 equal steps of the range and a bin per lane: weight,
// number of rows, smallest and largest key of each.  A bin whose two keys are equal
// is settled, however many rows it holds.  Where the crossing bin is not, it becomes
// the next range, cut to its keys, or is listed row by row when it has at most 31.
// A tie takes one pass, rows that a float cannot tell apart two or three.  What comes
// out are the rows listed, or the settled bins around the crossing: distinct keys
// with the weight of each.
//
// Nothing is taken on trust: the weight below lo is summed in the first pass and
// must fail the test of Lemma 1, and a key in the range must pass it.
//
// Bound by instructions, ~12 per row outside the range and a division (queued, so
// that all lanes divide) and three shared-memory words per row inside.  2000 x 64 of
// small integers, double, where such a pair went to the exact kernel (64 bisection
// steps with all rows): 47 -> 0.15 ms; near-multiples (spread 1e-5): 49 -> 0.24 ms.
// A few listed pairs cost the latency of one warp (at 1/4 instruction per cycle, those
// fetched for the first time more): 2000 rows 13 us, 22 with a rounded reciprocal, the
// weight's bits taken apart for every row and x_ijhat loaded where it is used.  Double:
// all four x_ijhat of a lane loaded at once and their weights without a branch, where each
// had a load and a wait of its own for the rows below: 701 x 103, one pair listed, 106.6 ->
// 102.2 us; 5000 x 32 of small integers 219 -> 190.
#pragma once

namespace l1l {

// Column jhat for narrow(), from the column copies: x_ijhat as float and as it is, and
// its 64-bit weight, floor(|b| 2^sigma).  Float: the scaling by a power of two, in two
// steps, is exact where the weight is not 0.  Double: fixq's value by shifts alone, which
// the FP64 pipe would slow where many pairs are listed.
template <typename T> struct ReadCol {
    const float *xf;
    const T *x;
    int sigma;
    float s0, s1;  // 2^sigma in two factors
    __device__ __forceinline__ ReadCol(const float *xf_, const T *x_, int sigma_)
        : xf(xf_), x(x_), sigma(sigma_) {
        s0 = __int_as_float((127 + sigma / 2) << 23);
        s1 = __int_as_float((127 + sigma - sigma / 2) << 23);
    }
    __device__ __forceinline__ T at(int i) const { return __ldg(x + i); }
    // rows i .. i + 3 (i a multiple of 4, padded rows included)
    __device__ __forceinline__ void rows(int i, double2 &a, double2 &b) const {
        a = __ldg(reinterpret_cast<const double2 *>(x + i));
        b = __ldg(reinterpret_cast<const double2 *>(x + i) + 1);
    }
    __device__ __forceinline__ unsigned long long weight(T b) const {
        if constexpr (sizeof(T) == 4) {
            return __float2ull_rz(fabsf(b) * s0 * s1);
        } else {
            const uint64_t u = (uint64_t)__double_as_longlong(b) & 0x7FFFFFFFFFFFFFFFull;
            const int be = (int)(u >> 52), s = max(be, 1) - 1075 + sigma;
            const uint64_t m = (u & 0xFFFFFFFFFFFFFull) | (be ? 0x10000000000000ull : 0);
            return s >= 0 ? m << s : m >> min(-s, 63);
        }
    }
};
__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

constexpr int NARROW_PEND = 64;  // rows queued for the division

// In the histogram's space; the list takes mn and w.
template <typename T> struct NarrowBins {
    typename Traits<T>::K mn[32], mx[32];
    unsigned long long w[32];
    uint32_t cnt[32];
    uint16_t pend[NARROW_PEND];
};

__device__ __forceinline__ void smem_min(uint32_t *p, uint32_t k) { atomicMin(p, k); }
__device__ __forceinline__ void smem_max(uint32_t *p, uint32_t k) { atomicMax(p, k); }
__device__ __forceinline__ void smem_min(uint64_t *p, uint64_t k) {
    atomicMin(reinterpret_cast<unsigned long long *>(p), (unsigned long long)k);
}
__device__ __forceinline__ void smem_max(uint64_t *p, uint64_t k) {
    atomicMax(reinterpret_cast<unsigned long long *>(p), (unsigned long long)k);
}

// Lane l's candidate: exact key fk (NONE: none) of weight fq.  L: the exact weight below
// all of them, after_zero: the penalty point lies there too.
template <typename T> struct NarrowCand {
    typename Traits<T>::K fk;
    int64_t fq, L;
    bool after_zero;
};

// Candidates around the median by the test d, on col's weights; few: at most 32 rows are
// expected in [lo, hi].  SEL_OK, SEL_SLOW_BAND
// where those weights cannot settle it, SEL_BELOW or SEL_ABOVE where it lies outside
// [lo, hi], or SEL_W64 (a range with infinities).
template <typename T>
__device__ int narrow(const float *__restrict__ xf, const T *__restrict__ xk,
                      const ReadCol<T> &col, uint32_t *mem, int n, uint32_t lo, uint32_t hi,
                      const Decide &d, bool few, NarrowCand<T> &out, int lane) {
    using Tr = Traits<T>;
    using K = typename Tr::K;
    constexpr uint32_t G = Approx<T>::G;
    const unsigned FULL = 0xFFFFFFFFu;
    using W = unsigned long long;
    static_assert(sizeof(NarrowBins<T>) <= HIST_WORDS * 4, "the histogram's space holds them");
    NarrowBins<T> &bins = *reinterpret_cast<NarrowBins<T> *>(mem);
    const int ng = (n + 127) >> 7;
    K A = Tr::key((T)akey_value(lo)), B = Tr::key((T)akey_value(hi));
    int64_t L = 0;
    bool list = few;  // the rows of [A, B] are listed in this pass
    for (int pass = 0; pass < 16; ++pass) {
        // rows that |fma(x, inv, -cen)| < delta does not flag have a coarse key
        // certainly outside [lo, hi] (as in the selection's second pass)
        const float va = akey_value(sat_sub(lo, G)), vb = akey_value(sat_add(hi, G));
        const float cen = 0.5f * va + 0.5f * vb;
        const float delta = (0.5f * vb - 0.5f * va) * (1.0f + 0x1p-20f) +
                            0x1p-21f * fmaxf(fabsf(va), fabsf(vb)) + 0x1p-148f;
        if (!(delta < 0x1p126f) || !(fabsf(cen) < 0x1p126f) || !(A <= B)) return SEL_W64;
        int c = 0;  // rows listed
        const K span = B - A;
        int sh = 0;
        if (span >= 32) {
            if constexpr (sizeof(K) == 4)
                sh = 27 - __clz((int)span);
            else
                sh = 59 - __clzll((long long)span);
        }
        // little more than 32 keys: one to a bin in the middle, where the median is
        // expected, the others in the outermost two
        K base = A;
        if (sh == 1) {
            sh = 0;
            base = A + ((span - 31) >> 1);
        }
        {
            // the penalty point is there from the start
            const bool zero = A <= Tr::KEY0 && Tr::KEY0 <= B;
            const int at =
                list || Tr::KEY0 <= base ? 0 : (int)min((Tr::KEY0 - base) >> sh, (K)31);
            bins.mn[lane] = zero && lane == at ? Tr::KEY0 : Tr::NONE;
            bins.mx[lane] = zero && lane == at ? Tr::KEY0 : 0;
            bins.w[lane] = 0;
            bins.cnt[lane] = zero && lane == at ? 1 : 0;
            c = zero ? 1 : 0;
        }
        __syncwarp();
        int64_t below = 0;
        int np = 0;  // rows queued
        // a lane holds back the sums of the bin it met last: ties meet one bin
        int cur = -1;
        W csum = 0;
        uint32_t ccnt = 0;
        K cmn = Tr::NONE, cmx = 0;
        auto add = [&](int b, W sum, uint32_t cnt, K kmin, K kmax) {
            b = L1L_CHK(b, 32);
            atomicAdd(&bins.w[b], sum);
            atomicAdd(&bins.cnt[b], cnt);
            if (kmin < *(volatile K *)&bins.mn[b]) smem_min(&bins.mn[b], kmin);
            if (kmax > *(volatile K *)&bins.mx[b]) smem_max(&bins.mx[b], kmax);
        };
        auto put = [&](bool in, K key, W q) {  // by all lanes
            if (list) {
                const unsigned m = __ballot_sync(FULL, in);
                const int at = c + __popc(m & ((1u << lane) - 1u));
                if (in && at < 32) {
                    bins.mn[at] = key;
                    bins.w[at] = q;
                }
                c += __popc(m);
            } else if (in) {
                const int b = key <= base ? 0 : (int)min((key - base) >> sh, (K)31);
                if (b != cur) {
                    if (cur >= 0) add(cur, csum, ccnt, cmn, cmx);
                    cur = b;
                    csum = 0;
                    ccnt = 0;
                    cmn = cmx = key;
                }
                csum += q;
                ccnt += 1;
                cmn = key < cmn ? key : cmn;
                cmx = key > cmx ? key : cmx;
            }
        };
        auto take = [&](bool on, int i) {  // row i by its exact key
            K key = Tr::NONE;
            W q = 0;
            if (on) {
                const T x = __ldg(xk + i);
                const T b = col.at(i);
                key = x == T(0) ? Tr::KEY0 : Tr::key(Tr::div_rn(x, b));
                q = col.weight(b);
            }
            if (pass == 0 && key < A) below += (int64_t)q;
            put(on && key >= A && key <= B, key, q);
        };
        float4 an = __ldg(reinterpret_cast<const float4 *>(xf) + lane);
        float4 bn = __ldg(reinterpret_cast<const float4 *>(col.xf) + lane);
        uint32_t mask = 0;  // 8 groups: a bit per row of the lane
        for (int g = 0; g < ng; ++g) {
            const float4 a4 = an, b4 = bn;
            const int i0 = L1L_CHK(g * 128 + 4 * lane, ng * 128);
            double2 c2 = {}, d2 = {};  // the weights' rows (double)
            if constexpr (sizeof(T) == 8) {
                if (pass == 0) col.rows(i0, c2, d2);
            }
            if (g + 1 < ng) {
                an = __ldg(reinterpret_cast<const float4 *>(xf + 128 + i0));
                bn = __ldg(reinterpret_cast<const float4 *>(col.xf + 128 + i0));
            }
            const float b[4] = {b4.x, b4.y, b4.z, b4.w};
            // x_ijhat = 0 (a padding row): infinite or NaN; neither inside nor, with its
            // weight of 0, of account below
            const float z[4] = {fmaf(a4.x, rcp_approx(b4.x), -cen), fmaf(a4.y, rcp_approx(b4.y), -cen),
                                fmaf(a4.z, rcp_approx(b4.z), -cen), fmaf(a4.w, rcp_approx(b4.w), -cen)};
            T e[4];
            if constexpr (sizeof(T) == 4) {
                e[0] = b[0], e[1] = b[1], e[2] = b[2], e[3] = b[3];
            } else {
                e[0] = c2.x, e[1] = c2.y, e[2] = d2.x, e[3] = d2.y;
            }
            uint32_t f = 0;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (fabsf(z[u]) < delta) f |= 1u << u;
                if (pass == 0) {
                    const int64_t q = (int64_t)col.weight(e[u]);
                    below += z[u] <= -delta ? q : 0;
                }
            }
            if (__popc(__ballot_sync(FULL, f == 15u)) >= 24) {  // most rows: as they lie
#pragma unroll 1
                for (int u = 0; u < 4; ++u) take((f >> u) & 1u, i0 + u);
                f = 0;
            }
            mask |= f << (4 * (g & 7));
            const bool end = g == ng - 1;
            if ((g & 7) != 7 && !end) continue;
            // the others by way of the queue, 32 at a time
            for (;;) {
                const unsigned m = __ballot_sync(FULL, mask != 0);
                if (mask != 0) {
                    const int bit = __ffs(mask) - 1;
                    mask &= mask - 1;
                    bins.pend[L1L_CHK(np + __popc(m & ((1u << lane) - 1u)), NARROW_PEND)] =
                        (uint16_t)(((g & ~7) + (bit >> 2)) * 128 + 4 * lane + (bit & 3));
                }
                np += __popc(m);
                __syncwarp();
                if (np >= 32 || (end && m == 0 && np > 0)) {
                    const bool on = lane < np;
                    take(on, L1L_CHK(on ? (int)bins.pend[lane] : 0, ng * 128));
                    __syncwarp();
                    const uint16_t up = bins.pend[32 + lane];
                    __syncwarp();
                    bins.pend[lane] = up;
                    np = max(np - 32, 0);
                    __syncwarp();
                }
                if (m == 0) break;
            }
        }
        __syncwarp();
        // what the lanes hold: a bin of many lanes is summed across them first (64-bit
        // atomics in shared memory take their turns)
        if (const unsigned on = __ballot_sync(FULL, cur >= 0)) {
            const int b = __shfl_sync(FULL, cur, __ffs(on) - 1);
            if (__popc(__ballot_sync(FULL, cur == b)) >= 4) {
                const bool in = cur == b;
                W sum = in ? csum : 0;
                const uint32_t cnt = __reduce_add_sync(FULL, in ? ccnt : 0u);
                K kmin = in ? cmn : Tr::NONE, kmax = in ? cmx : 0;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    sum += __shfl_xor_sync(FULL, sum, o);
                    const K x = __shfl_xor_sync(FULL, kmin, o), y = __shfl_xor_sync(FULL, kmax, o);
                    kmin = x < kmin ? x : kmin;
                    kmax = y > kmax ? y : kmax;
                }
                if (lane == 0) add(b, sum, cnt, kmin, kmax);
                if (in) cur = -1;
            }
            if (cur >= 0) add(cur, csum, ccnt, cmn, cmx);
        }
        __syncwarp();
        if (pass == 0) {
            L = warp_sum_i64(below);
            const int r = d.cond(L, A > Tr::KEY0);
            if (r != 0) return r > 0 ? SEL_BELOW : SEL_SLOW_BAND;
        }
        if (list && c > 32) {
            list = false;
            continue;
        }
        if (list) {
            out.fk = lane < c ? bins.mn[lane] : Tr::NONE;
            out.fq = lane < c ? (int64_t)bins.w[lane] : 0;
            out.L = L;
            out.after_zero = __all_sync(FULL, out.fk > Tr::KEY0);
            return SEL_OK;
        }
        const K mn = bins.mn[lane], mx = bins.mx[lane];
        const int64_t w = (int64_t)bins.w[lane];
        const int rows = (int)bins.cnt[lane];
        __syncwarp();
        const bool has = rows != 0;
        const int64_t P = L + warp_scan_add(w, lane);  // weight up to this bin's last key
        const int r = has ? d.cond(P, mx >= Tr::KEY0) : 0;
        const unsigned any = __ballot_sync(FULL, r != 0);
        if (any == 0) return SEL_ABOVE;
        const int ca = __ffs(any) - 1;  // the crossing bin
        if (__shfl_sync(FULL, r, ca) < 0) return SEL_SLOW_BAND;
        const unsigned open = __ballot_sync(FULL, has && mn != mx);
        if (((open >> ca) & 1u) == 0) {
            // the settled bins from the first such below it to the last above
            const unsigned under = open & ((1u << ca) - 1u), over = open & ~(FULL >> (31 - ca));
            const int a = under ? 32 - __clz((int)under) : 0, b = over ? __ffs(over) - 2 : 31;
            const bool in = has && lane >= a && lane <= b;
            out.fk = in ? mn : Tr::NONE;
            out.fq = in ? w : 0;
            out.L = __shfl_sync(FULL, P - w, a);
            const unsigned ins = __ballot_sync(FULL, in);  // ca is among them
            out.after_zero = __shfl_sync(FULL, mn, __ffs(ins) - 1) > Tr::KEY0;
            return SEL_OK;
        }
        // the next range: that bin, or for the list as many around it as fit
        int a = ca, b = ca;
        const int R = warp_scan_add(rows, lane), Rc = __shfl_sync(FULL, R, ca);
        const int rc = __shfl_sync(FULL, rows, ca);
        list = rc <= 31;
        if (list) {
            a = __ffs(__ballot_sync(FULL, has && Rc - R + rows <= max(16, rc))) - 1;
            const int Ra = __shfl_sync(FULL, R - rows, a);
            b = 31 - __clz((int)__ballot_sync(FULL, has && R - Ra <= 31));
        }
        L = __shfl_sync(FULL, P - w, a);
        A = __shfl_sync(FULL, mn, a);
        B = __shfl_sync(FULL, mx, b);
        lo = coarse_of<T>(A);
        hi = coarse_of<T>(B);
    }
    return SEL_W64;
}

// One penalty, by every lane: the smallest key that passes.  The sums by rank, in a loop
// (as everything here that runs once per pair: what a few listed pairs cost is mostly
// the fetch of instructions).
template <typename T>
__device__ __forceinline__ int narrow_pick(const NarrowCand<T> &f, const Decide &d,
                                           typename Traits<T>::K &tstar, int lane) {
    const unsigned FULL = 0xFFFFFFFFu;
    using K = typename Traits<T>::K;
    const unsigned on = __ballot_sync(FULL, f.fk != Traits<T>::NONE);
    int64_t S = f.L;
#pragma unroll 1
    for (unsigned c = on; c; c &= c - 1) {
        const int u = __ffs(c) - 1;
        const K ku = __shfl_sync(FULL, f.fk, u);
        const int64_t qu = __shfl_sync(FULL, f.fq, u);
        S += ku <= f.fk ? qu : 0;
    }
    const int r = f.fk != Traits<T>::NONE ? d.cond(S, f.fk >= Traits<T>::KEY0) : 0;
    K best = Traits<T>::NONE;  // equal keys have equal sums
    int rb = 0;
#pragma unroll 1
    for (unsigned c = __ballot_sync(FULL, r != 0); c; c &= c - 1) {
        const int u = __ffs(c) - 1;
        const K ku = __shfl_sync(FULL, f.fk, u);
        const int ru = __shfl_sync(FULL, r, u);
        if (ku < best) {
            best = ku;
            rb = ru;
        }
    }
    if (rb == 0) return SEL_ABOVE;
    tstar = best;
    return rb < 0 ? SEL_SLOW_BAND : SEL_OK;
}

// How far the range above (or below) [lo, hi] has to reach to hold the next row
// outside it: the coarse key of the nearest approximate ratio beyond the guard band,
// and the band again.
template <typename T>
__device__ uint32_t next_coarse(const float *__restrict__ xf, const ReadCol<T> &col, int n,
                                uint32_t lo, uint32_t hi, bool above, int lane) {
    constexpr uint32_t G = Approx<T>::G;
    const uint32_t ka = sat_sub(lo, G), kb = sat_add(hi, G);
    uint32_t near = above ? CKNONE : 0u;
    for (int i = lane; i < n; i += 32) {
        const float b = __ldg(col.xf + i);
        if (b == 0.0f) continue;
        const uint32_t k = akey(__fmul_rn(__ldg(xf + i), __frcp_rn(b)));
        if (above && k > kb) near = min(near, k);
        if (!above && k < ka) near = max(near, k);
    }
    if (above) return sat_add(max(__reduce_min_sync(0xFFFFFFFFu, near), kb), G);
    return sat_sub(min(__reduce_max_sync(0xFFFFFFFFu, near), ka), G);
}

// The median on 64-bit weights, within [lo, hi] or next to it: where the 32-bit
// weights could not settle whether a key passes, it may be the next key above or
// below.
template <typename T>
__device__ __noinline__ int narrow64(const float *xf, const T *xk, const ReadCol<T> &col,
                                     uint32_t *hist, int n, uint32_t lo, uint32_t hi,
                                     const Decide &d, bool few, typename Traits<T>::K &tstar,
                                     int lane) {
    int st = SEL_W64;
    for (int tries = 0; tries < 3; ++tries) {
        NarrowCand<T> f;
        st = narrow<T>(xf, xk, col, hist, n, lo, hi, d, few, f, lane);
        __syncwarp();
        if (st == SEL_OK) st = narrow_pick<T>(f, d, tstar, lane);
        if (st != SEL_BELOW && st != SEL_ABOVE) return st;
        // from the value of hi (lo) on: an exact key beyond it may round to it
        const uint32_t at = next_coarse<T>(xf, col, n, lo, hi, st == SEL_ABOVE, lane);
        if (st == SEL_ABOVE) {
            lo = hi;
            hi = at;
        } else {
            hi = lo;
            lo = at;
        }
    }
    return st;
}

}  // namespace l1l
