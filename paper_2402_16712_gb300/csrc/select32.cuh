// select32.cuh -- the weighted median of one (jhat, k) pair on 32-bit
// fixed-point weights (Lemma 1, decided exactly).
//
// The weights are q32_i = floor(|x_ijhat| 2^s32) with the column total below
// 2^32 (ColInfo::Q32), so every partial sum is one 32-bit add.  A row's ratio
// is approximated by one multiply, r' = fl(x_ik * fl(1/x_ijhat)), within G
// coarse keys of the correctly rounded one; r' decides which few rows are
// looked at, and those are divided exactly.  Two passes over the rows, and
// nothing is stored per row:
//
//   bracket  32 sampled rows (weight-proportional) are sorted across the warp;
//            the sample keys d0 positions either side of the estimated
//            crossing of half the weight bracket the median;
//   pass 1   the weight of every row by the bin of r': bins are equal steps
//            of the ratio itself, bin = round(fma(r', 1/w, bm)), read off the
//            low mantissa bits of the sum with 2^23 in bm -- one multiply-add,
//            no branch at 0, monotone in r'; rows below the bracket add to a
//            register, rows inside to a 256-bin shared histogram;
//   crossing a warp scan finds the bin where half the weight is passed under
//            the order of r'.  Moving every ratio by at most G keys moves the
//            weighted median by at most G keys, so the exact median lies
//            within G keys of that bin: [lo, hi].  Rows whose bin lies below
//            that range (widened by G once more) have exact keys below lo,
//            rows above it have exact keys above hi, and the histogram's
//            prefix sum is the exact weight of the former;
//   pass 2   flags the rows whose r' may fall in the range (one multiply-add
//            and one compare per row, slightly too wide); their bins are
//            computed again, and those in the range are the candidates;
//   final    the candidates (at most 31) are divided exactly, and the
//            smallest exact key that passes half the weight is the median.
//
// None of the steps before the last has to be trusted: the candidates'
// weights must add up to the histogram's (no weighted row of the range is
// missing), the weight below lo must fail the test of Lemma 1, and a key in
// [lo, hi] must pass it.  A pair that does not meet this, more than 31 rows
// in the range (ties), a decision inside the certainty band of the truncated
// weights (Dec32), or a bracket too wide for float steps is listed for the
// kernel behind, with the range where it is known (exact.cuh, narrow.cuh).
//
// Bound (2000 x 2000 float, 32 resident warps): the L1/shared data pipe, ~690
// wavefronts of 128 bytes per pair at 85% of its rate (pass 1: x, 1/x_ijhat,
// q and ~2.5 per histogram atomic; pass 2: x and 1/x_ijhat; residual: x and
// x_ijhat), and ~2200 instructions per pair at 69% of the issue slots.  Against the
// selection that kept every row of the bracket in a per-lane list: 13.66 -> 11.14 ms
// there; 1000 x 500 with 32 lambdas 5.62 -> 2.61 ms (one selection instead of two and a
// pass); and without the lists 5000 rows keep 32 warps resident instead of 16, 5000 x
// 1000 10.23 -> 7.61 ms.
// Finding the crossing lane before the bin in it, instead of every bin's prefix
// sum and test: 11.14 -> 11.06 ms, double 19.36 -> 19.19 ms.  Pairs that are not
// settled here listed, not taken through a fallback in the same kernel: 11.06 ->
// 10.52 ms, double 19.19 -> 18.35, 5000 x 1000 7.58 -> 6.24.
#pragma once
#include <cstdint>

#include "checks.cuh"
#include "common.cuh"

namespace l1l {

constexpr int NB32 = 256;     // bins of the bracket histogram
constexpr int BPL = NB32 / 32;  // bins per lane of its scan
constexpr int NB32_SIDE = 8;  // bins kept free either side of the bracket
constexpr float Z32 = 8388608.0f;  // 2^23: a float at or above it has integer steps
constexpr uint32_t Z32_BITS = 0x4B000000u;

// Float value of a key of akey's order (-0 just below +0).
__device__ __forceinline__ float akey_value(uint32_t k) {
    const uint32_t u = (k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k;
    return __uint_as_float(u);
}

// Shared-memory accesses by 32-bit shared-window address, so that they stay
// shared-memory instructions (not generic ones) whatever the inlining.
__device__ __forceinline__ uint32_t smem_addr(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ float4 ld_shared_v4f(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(addr)
                 : "memory");
    return v;
}

// Read-only global loads (the column copies do not change during a launch).
__device__ __forceinline__ float4 ldg_f4(const float *p) {
    return __ldg(reinterpret_cast<const float4 *>(p));
}

// Pass 1 for this lane's four consecutive rows of a 128-row group (x: their
// x_ik; ainv, aq: shared addresses of their 1/x_ijhat and q32): per row
// z = fma(x * inv, 1/w, bm); z < 2^23: below the bracket, add q to Sb;
// z < 2^23 + NB32: bin z - 2^23 of the histogram, hb being its shared address
// less 4 * Z32_BITS.  NaN (x_ijhat = 0, a padding row) is neither.  The
// multiplies go two rows to an instruction (rn in each half, so the bins are
// those of the scalar form).
__device__ __forceinline__ void hist32_group(float4 x, uint32_t ainv, uint32_t aq, uint64_t sc2,
                                             uint64_t bm2, uint32_t hb, uint32_t &Sb) {
    asm volatile(
        "{\n\t"
        ".reg .pred pb, pc;\n\t"
        ".reg .b64 x01, x23, v01, v23;\n\t"
        ".reg .f32 z0, z1, z2, z3;\n\t"
        ".reg .b32 q0, q1, q2, q3, a, zb;\n\t"
        "ld.shared.v2.b64 {v01, v23}, [%1];\n\t"
        "ld.shared.v4.u32 {q0, q1, q2, q3}, [%2];\n\t"
        "mov.b64 x01, {%3, %4};\n\t"
        "mov.b64 x23, {%5, %6};\n\t"
        "mul.rn.f32x2 x01, x01, v01;\n\t"
        "mul.rn.f32x2 x23, x23, v23;\n\t"
        "fma.rn.f32x2 x01, x01, %7, %8;\n\t"
        "fma.rn.f32x2 x23, x23, %7, %8;\n\t"
        "mov.b64 {z0, z1}, x01;\n\t"
        "mov.b64 {z2, z3}, x23;\n\t"
        // row 0
        "setp.lt.f32 pb, z0, 0f4B000000;\n\t"
        "setp.lt.and.f32 pc, z0, 0f4B000100, !pb;\n\t"
        "@pb add.u32 %0, %0, q0;\n\t"
        "mov.b32 zb, z0;\n\t"
        "shl.b32 a, zb, 2;\n\t"
        "add.u32 a, a, %9;\n\t"
        "@pc red.shared.add.u32 [a], q0;\n\t"
        // row 1
        "setp.lt.f32 pb, z1, 0f4B000000;\n\t"
        "setp.lt.and.f32 pc, z1, 0f4B000100, !pb;\n\t"
        "@pb add.u32 %0, %0, q1;\n\t"
        "mov.b32 zb, z1;\n\t"
        "shl.b32 a, zb, 2;\n\t"
        "add.u32 a, a, %9;\n\t"
        "@pc red.shared.add.u32 [a], q1;\n\t"
        // row 2
        "setp.lt.f32 pb, z2, 0f4B000000;\n\t"
        "setp.lt.and.f32 pc, z2, 0f4B000100, !pb;\n\t"
        "@pb add.u32 %0, %0, q2;\n\t"
        "mov.b32 zb, z2;\n\t"
        "shl.b32 a, zb, 2;\n\t"
        "add.u32 a, a, %9;\n\t"
        "@pc red.shared.add.u32 [a], q2;\n\t"
        // row 3
        "setp.lt.f32 pb, z3, 0f4B000000;\n\t"
        "setp.lt.and.f32 pc, z3, 0f4B000100, !pb;\n\t"
        "@pb add.u32 %0, %0, q3;\n\t"
        "mov.b32 zb, z3;\n\t"
        "shl.b32 a, zb, 2;\n\t"
        "add.u32 a, a, %9;\n\t"
        "@pc red.shared.add.u32 [a], q3;\n\t"
        "}"
        : "+r"(Sb)
        : "r"(ainv), "r"(aq), "f"(x.x), "f"(x.y), "f"(x.z), "f"(x.w), "l"(sc2), "l"(bm2), "r"(hb)
        : "memory");
}
static_assert(NB32 == 256, "the PTX above holds 2^23 + NB32 as 0f4B000100");

// Pass 2 for the same four rows: mask |= 1 when some |fma(x, inv, -c)| <
// delta (NaN: never).
__device__ __forceinline__ void flag32_group(float4 x, uint32_t ainv, float nc, float delta,
                                             uint32_t &mask) {
    asm volatile(
        "{\n\t"
        ".reg .pred p;\n\t"
        ".reg .f32 v0, v1, v2, v3;\n\t"
        "ld.shared.v4.f32 {v0, v1, v2, v3}, [%1];\n\t"
        "fma.rn.f32 v0, %2, v0, %6;\n\t"
        "fma.rn.f32 v1, %3, v1, %6;\n\t"
        "fma.rn.f32 v2, %4, v2, %6;\n\t"
        "fma.rn.f32 v3, %5, v3, %6;\n\t"
        "abs.f32 v0, v0;\n\t"
        "abs.f32 v1, v1;\n\t"
        "abs.f32 v2, v2;\n\t"
        "abs.f32 v3, v3;\n\t"
        "setp.lt.f32 p, v0, %7;\n\t"
        "setp.lt.or.f32 p, v1, %7, p;\n\t"
        "setp.lt.or.f32 p, v2, %7, p;\n\t"
        "setp.lt.or.f32 p, v3, %7, p;\n\t"
        "@p or.b32 %0, %0, 1;\n\t"
        "}"
        : "+r"(mask)
        : "r"(ainv), "f"(x.x), "f"(x.y), "f"(x.z), "f"(x.w), "f"(nc), "f"(delta)
        : "memory");
}

// One key per lane, ascending in the lane index.
__device__ __forceinline__ float warp_sort32f(float k, int lane) {
#pragma unroll
    for (int size = 2; size <= 32; size <<= 1) {
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            const float o = __shfl_xor_sync(0xFFFFFFFFu, k, stride);
            const bool up = (lane & size) == 0, lower = (lane & stride) == 0;
            k = lower == up ? fminf(k, o) : fmaxf(k, o);
        }
    }
    return k;
}

// What the selection leaves for the final test: lane l < c holds candidate l
// (exact key fk, weight fq; fk = NONE, fq = 0 where its exact key falls
// outside [lo, hi]), lane c the key of 0 when 0 lies in [lo, hi]; nv lanes are
// used; L is the exact weight of the rows with a coarse key below lo.
template <typename T> struct Cand32 {
    typename Traits<T>::K fk;
    uint32_t fq, lo, hi;
    int64_t L;
    int nv;
};

// The candidates of every weighted median between that of penalty d1 and that
// of penalty d2 (the same for one penalty).  xf: column k as float (global,
// rows padded to a multiple of 128 with zeros; the column itself for float
// input, its float copy for double input); xk, w.colb: column k and x_ijhat in
// the input type, read for the exact divisions.  Returns SEL_OK, SEL_W64 or
// SEL_MANY: more than 31 rows lie in [out.lo, out.hi] (for two penalties: that no
// bins separate; `one` says that the two are equal).
template <typename T, bool TWO>
__device__ __forceinline__ int candidates32(const float *__restrict__ xf, const T *__restrict__ xk,
                                            const WarpCtx<T> &w, const Dec32 &d1, const Dec32 &d2,
                                            Cand32<T> &out, int lane, bool one = false) {
    using Tr = Traits<T>;
    using K = typename Tr::K;
    constexpr uint32_t G = Approx<T>::G;  // guard band of the approximate keys
    const unsigned FULL = 0xFFFFFFFFu;
    const int ng = (w.n + 127) >> 7;  // 128-row groups (rows are padded to them)
    uint32_t *hist = w.hist;
    const uint32_t ahist = smem_addr(hist);
    const uint32_t ainv0 = smem_addr(w.inv) + 16u * (uint32_t)lane;
    const uint32_t aq0 = smem_addr(w.q32) + 16u * (uint32_t)lane;

    // ---------------- sample bracket ------------------------------------
    // Every second of the column's 64 samples: +-6 of 32 holds ~37% of the
    // weight and misses ~0.3% of the medians.  All 64, as two sorted lists or
    // one, cost more to gather and sort than their narrower bracket saved
    // (2000 x 2000 float: 11.4 -> 11.7 ms).
    const float s = warp_sort32f(__fmul_rn(__ldg(xf + w.srow), w.sinv), lane);
    const float cum = (float)(lane + 1) * d1.Qf;
    auto crossing = [&](const Dec32 &d) -> int {
        const unsigned b = __ballot_sync(FULL, cum >= (s >= 0.0f ? d.fpos : d.fneg));
        return b ? __ffs(b) - 1 : 31;
    };
    const int j1 = crossing(d1), j2 = TWO ? crossing(d2) : j1;
    const int ja = (TWO ? min(j1, j2) : j1) - w.d0, jb = (TWO ? max(j1, j2) : j1) + w.d0;
    float a = __shfl_sync(FULL, s, max(ja, 0)), b = __shfl_sync(FULL, s, min(jb, 31));
    // past the sample's ends: as far again
    if (ja < 0) a -= b - a;
    if (jb > 31) b += b - a;

    for (int attempt = 0; attempt < 4; ++attempt) {
        // ---- bins: steps of w1, no finer than 16 keys of the largest ratio (or
        // 2^-99, where the whole bracket is 0: sparse columns)
        const float wf = fmaxf(fmaxf(fabsf(a), fabsf(b)) * 0x1p-19f, 0x1p-99f);
        const float w1 = fmaxf((b - a) * (1.0f / (NB32 - 2 * NB32_SIDE)), wf);
        if (!(w1 < 0x1p100f)) return SEL_W64;
        const float sc = __frcp_rn(w1);
        const float bm = __fmaf_rn(-a, sc, Z32 + (float)NB32_SIDE);
        // ---- pass 1 ------------------------------------------------------
        reinterpret_cast<uint4 *>(hist)[lane] = make_uint4(0, 0, 0, 0);
        reinterpret_cast<uint4 *>(hist)[lane + 32] = make_uint4(0, 0, 0, 0);
        __syncwarp();
        uint32_t Sb = 0;
        {
            const float4 *xp = reinterpret_cast<const float4 *>(xf) + lane;
#if L1L_CHECKS
            for (int g = 0; g < ng; ++g) {
                const float4 x4 = __ldg(xp);
                xp += 32;
                const float xs[4] = {x4.x, x4.y, x4.z, x4.w};
                for (int u = 0; u < 4; ++u) {
                    const int i = L1L_CHK(g * 128 + 4 * lane + u, ng * 128);
                    const float z = __fmaf_rn(__fmul_rn(xs[u], w.inv[i]), sc, bm);
                    if (z < Z32)
                        Sb += w.q32[i];
                    else if (z < Z32 + (float)NB32)
                        atomicAdd(&hist[L1L_CHK(__float_as_uint(z) - Z32_BITS, (uint32_t)NB32)],
                                  w.q32[i]);
                }
            }
#else
            uint64_t sc2, bm2;
            asm("mov.b64 %0, {%1, %1};" : "=l"(sc2) : "f"(sc));
            asm("mov.b64 %0, {%1, %1};" : "=l"(bm2) : "f"(bm));
            const uint32_t hb = ahist - 4u * Z32_BITS;
            uint32_t ainv = ainv0, aq = aq0;
            float4 xn = __ldg(xp);
#pragma unroll 2
            for (int g = 0; g < ng; ++g) {
                const float4 xc = xn;
                xp += 32;
                if (g + 1 < ng) xn = __ldg(xp);
                hist32_group(xc, ainv, aq, sc2, bm2, hb, Sb);
                ainv += 512u;
                aq += 512u;
            }
#endif
        }
        Sb = __reduce_add_sync(FULL, Sb);  // <= Q32 < 2^32
        __syncwarp();
        // ---- the crossing bin(s): first the lane (bins 8l .. 8l+7), then the
        // bin among its eight.  Whether a bin passes is monotone in the bin.
        uint32_t tot = 0;
        {
#pragma unroll
            for (int e = 0; e < BPL; e += 4) {
                const uint4 h = reinterpret_cast<const uint4 *>(hist)[(BPL / 4) * lane + e / 4];
                tot += (h.x + h.y) + (h.z + h.w);
            }
        }
        uint32_t end = tot;  // weight up to this lane's last bin
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(FULL, end, o);
            if (lane >= o) end += y;
        }
        end += Sb;
        // bins from that of 0 on end at ratios >= 0
        const int zb = bm < Z32 ? 0 : (bm < Z32 + (float)NB32 ? (int)(bm - Z32) : NB32);
        auto cross_bin = [&](const Dec32 &d, uint32_t &before, uint32_t &through) -> int {
            const unsigned any =
                __ballot_sync(FULL, end >= (BPL * lane + BPL - 1 >= zb ? d.tpos : d.tneg));
            if (!any) return NB32;
            const int ln = __ffs(any) - 1, e = lane & (BPL - 1);
            const uint32_t q = hist[BPL * ln + e];
            uint32_t c = q;
#pragma unroll
            for (int o = 1; o < BPL; o <<= 1) {
                const uint32_t y = __shfl_up_sync(FULL, c, o, BPL);
                if (e >= o) c += y;
            }
            c += __shfl_sync(FULL, end - tot, ln);
            const int at =
                __ffs(__ballot_sync(FULL, c >= (BPL * ln + e >= zb ? d.tpos : d.tneg))) - 1;
            through = __shfl_sync(FULL, c, at);
            before = through - __shfl_sync(FULL, q, at);
            return BPL * ln + at;
        };
        uint32_t L1 = 0, E1 = 0, L2 = 0, E2 = 0;
        const int c1 = cross_bin(d1, L1, E1);
        const int c2 = TWO ? cross_bin(d2, L2, E2) : c1;
        const int ca = TWO ? min(c1, c2) : c1, cb = TWO ? max(c1, c2) : c1;
        // ---- the coarse keys [lo, hi] around the crossing and their bins ----
        // r' of bin b: (2^23 + b - bm -+ 1/2) w1, up to a few keys
        const float ra = ((Z32 + (float)ca - bm) - 0.5f) * w1;
        const float rb = ((Z32 + (float)cb - bm) + 0.5f) * w1;
        const uint32_t ka = sat_sub(akey(ra), 2 * G + 4), kb = sat_add(akey(rb), 2 * G + 4);
        const float va = akey_value(ka), vb = akey_value(kb);
        const bool under = ca < 1, over = cb >= NB32;
        if (under || over) {
            // missed: once more, on the side the median lies
            if (attempt >= 2 || (under && over)) return SEL_W64;
            if (under) {
                const int jn = ja - 2 * w.d0 - 1;
                const float s0 = fminf(__shfl_sync(FULL, s, 0), 0.0f);
                b = a + 2.0f * w1;
                a = jn >= 0 ? __shfl_sync(FULL, s, jn) : s0 - 0.25f * (b - s0);
            } else {
                const int jn = jb + 2 * w.d0 + 1;
                const float s1 = fmaxf(__shfl_sync(FULL, s, 31), 0.0f);
                a = b - 2.0f * w1;
                b = jn <= 31 ? __shfl_sync(FULL, s, jn) : s1 + 0.25f * (s1 - a);
            }
            if (!(a < b)) return SEL_W64;
            __syncwarp();
            continue;
        }
        if (!(va < vb)) return SEL_W64;  // also NaN: keys past the infinities
        uint32_t L = TWO && c2 < c1 ? L2 : L1;
        const uint32_t W = (TWO && c2 > c1 ? E2 : E1) - L;  // weight of the bins ca .. cb
        __syncwarp();
        // ---- pass 2: flag the groups with a row in [va, vb], list those rows.
        // |fma(x, inv, -cen)| differs from |r' - cen| by at most 3 roundings
        // of 2^-24 of the larger end.
        const float cen = 0.5f * (va + vb);
        const float delta = 0.5f * (vb - va) * (1.0f + 0x1p-20f) + 0x1p-21f * fmaxf(fabsf(va), fabsf(vb));
        int c = 0;
        for (int g0 = 0; g0 < ng; g0 += 32) {
            const int ge = min(ng, g0 + 32);
            uint32_t mask = 0;
            const float4 *xp = reinterpret_cast<const float4 *>(xf) + g0 * 32 + lane;
            uint32_t ainv = ainv0 + 512u * (uint32_t)g0;
            float4 xn = __ldg(xp);
#pragma unroll 2
            for (int g = g0; g < ge; ++g) {
                const float4 xc = xn;
                xp += 32;
                if (g + 1 < ge) xn = __ldg(xp);
                mask <<= 1;
                flag32_group(xc, ainv, -cen, delta, mask);
                ainv += 512u;
            }
            // bit b of the mask is group ge - 1 - b
            while (__any_sync(FULL, mask != 0)) {
                const bool has = mask != 0;
                const int i0 = has ? (ge - __ffs(mask)) * 128 + 4 * lane : 4 * lane;
                mask &= mask - 1;
                const float4 x4 = ldg_f4(xf + L1L_CHK(i0, ng * 128));
                const uint32_t ro = 4u * (uint32_t)(i0 - 4 * lane);
                const float4 v4 = ld_shared_v4f(ainv0 + ro);
                const float xs[4] = {x4.x, x4.y, x4.z, x4.w}, vs[4] = {v4.x, v4.y, v4.z, v4.w};
                uint32_t in = 0;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const float r = __fmul_rn(xs[u], vs[u]);
                    in |= r >= va && r <= vb ? 1u << u : 0u;
                }
                if (!has) in = 0;
                while (__any_sync(FULL, in != 0)) {
                    const unsigned m = __ballot_sync(FULL, in != 0);
                    const int pos = c + __popc(m & ((1u << lane) - 1u));
                    if (in != 0 && pos < 31)
                        hist[L1L_CHK(pos, 31)] = (uint32_t)(i0 + __ffs(in) - 1);
                    in &= in - 1;
                    c += __popc(m);
                }
                if (c > 31) mask = 0;
            }
        }
        __syncwarp();
        if (c > 31) {
            out.lo = ka + G;
            out.hi = kb - G;
            if (!TWO || one || w1 == wf) return SEL_MANY;
            // two penalties: finer bins over the range, unless it hardly shrank
            if (!(vb - va < 0.25f * (b - a))) return SEL_W64;
            a = va;
            b = vb;
            continue;
        }
        // ---- exact keys ------------------------------------------------------
        const uint32_t lo = ka + G, hi = kb - G;
        K fk = Tr::NONE;
        uint32_t fq = 0, below = 0, under_w = 0, in_w = 0;
        if (lane < c) {
            const uint32_t row = L1L_CHK(hist[lane], (uint32_t)(ng * 128));
            fk = Tr::key(Tr::div_rn(__ldg(xk + row), w.colb[row]));
            fq = w.q32[row];
            // candidates of the bins next to ca .. cb: below, they leave L
            const float z = __fmaf_rn(__fmul_rn(__ldg(xf + row), w.inv[row]), sc, bm);
            under_w = z < Z32 + (float)ca ? fq : 0u;
            in_w = z >= Z32 + (float)ca && z <= Z32 + (float)cb ? fq : 0u;
        }
        // every weighted row of the bins is among the candidates
        if (__reduce_add_sync(FULL, in_w) != W) return SEL_W64;
        L -= __reduce_add_sync(FULL, under_w);
        if (lane < c) {
            const uint32_t ck = coarse_of<T>(fk);
            if (ck < lo || ck > hi) {
                below = ck < lo ? fq : 0u;
                fk = Tr::NONE;
                fq = 0;
            }
        }
        const bool zero_in = lo <= CK0 && CK0 <= hi;
        if (lane == c && zero_in) fk = Tr::KEY0;  // the penalty point; lambda sits in the test
        out.fk = fk;
        out.fq = fq;
        out.lo = lo;
        out.hi = hi;
        out.L = (int64_t)L + (int64_t)__reduce_add_sync(FULL, below);
        out.nv = c + (zero_in ? 1 : 0);
        __syncwarp();
        return SEL_OK;
    }
    return SEL_W64;
}

// Weighted median of pair (jhat, k) at one penalty: SEL_OK with its exact key in
// tstar, else SEL_MANY or SEL_W64 and the mark to list it with.
template <typename T>
__device__ __forceinline__ int select_w32(const float *__restrict__ xf, const T *__restrict__ xk,
                                          const WarpCtx<T> &w, const Dec32 &dc,
                                          typename Traits<T>::K &tstar, int64_t &mark,
                                          int lane) {
    using Tr = Traits<T>;
    using K = typename Tr::K;
    const unsigned FULL = 0xFFFFFFFFu;
    Cand32<T> f;
    if (const int st = candidates32<T, false>(xf, xk, w, dc, dc, f, lane); st != SEL_OK) {
        mark = st == SEL_MANY ? off_mark(OFF_MANY, f.lo, f.hi) : off_mark(OFF_NONE, 1, 0);
        return st;
    }
    // no key below lo passes
    if (dc.cond(f.L, f.lo > CK0) != 0) {
        mark = off_mark(OFF_RANGE, f.lo, f.hi);
        return SEL_W64;
    }
    // each candidate's cumulative weight: the weight of candidates with a key
    // at or below its own (equal keys alike); the smallest key that passes
    uint32_t S = 0;
    for (int u = 0; u < f.nv; ++u) {
        const K ku = __shfl_sync(FULL, f.fk, u);
        const uint32_t qu = __shfl_sync(FULL, f.fq, u);
        S += ku <= f.fk ? qu : 0u;
    }
    int r = 0;
    if (f.fk != Tr::NONE) r = dc.cond(f.L + (int64_t)S, f.fk >= Tr::KEY0);
    K kmin = r != 0 ? f.fk : Tr::NONE;
    if constexpr (sizeof(T) == 4) {
        kmin = __reduce_min_sync(FULL, kmin);
    } else {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const K y = __shfl_xor_sync(FULL, kmin, o);
            kmin = y < kmin ? y : kmin;
        }
    }
    if (kmin == Tr::NONE || __any_sync(FULL, r == -1 && f.fk == kmin)) {
        mark = off_mark(OFF_RANGE, f.lo, f.hi);
        return SEL_W64;
    }
    tstar = kmin;
    return SEL_OK;
}

// Residual sum_i |x_ik - v x_ijhat| over the padded rows (padding rows are 0
// in both columns), float input, four consecutive rows per lane per 128-row
// group and four groups per step: the step's sixteen loads are in flight
// together (column k comes from L2, so the pass is bound by load latency, not
// arithmetic); xj in shared memory when XS, else in global memory.
template <bool XS>
__device__ __forceinline__ float warp_residual_f4(const float *__restrict__ xk,
                                                  const float *__restrict__ xj, int n, float v,
                                                  int lane) {
    const int ng = (n + 127) >> 7;
    const float4 *a4 = reinterpret_cast<const float4 *>(xk) + lane;
    const float4 *b4 = reinterpret_cast<const float4 *>(xj) + lane;
    auto ldb = [&](int g) -> float4 {
        if constexpr (XS)
            return b4[g * 32];
        else
            return __ldg(b4 + g * 32);
    };
    float acc0 = 0.f, acc1 = 0.f, acc2 = 0.f, acc3 = 0.f;
    auto add4 = [&](const float4 &a, const float4 &b) {
        acc0 += fabsf(fmaf(-v, b.x, a.x));
        acc1 += fabsf(fmaf(-v, b.y, a.y));
        acc2 += fabsf(fmaf(-v, b.z, a.z));
        acc3 += fabsf(fmaf(-v, b.w, a.w));
    };
    int g = 0;
    for (; g + 3 < ng; g += 4) {
        float4 a[4], b[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) a[u] = __ldg(a4 + (g + u) * 32);
#pragma unroll
        for (int u = 0; u < 4; ++u) b[u] = ldb(g + u);
#pragma unroll
        for (int u = 0; u < 4; ++u) add4(a[u], b[u]);
    }
    for (; g < ng; ++g) add4(__ldg(a4 + g * 32), ldb(g));
    float s = (acc0 + acc1) + (acc2 + acc3);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
    return s;
}

}  // namespace l1l
