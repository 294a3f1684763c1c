// k_exact.cu -- exact slow path of step A3 for the pairs the fixed-point fast
// path could not settle (a column with weights too small for its scale, tied
// within the truncation band) or for every pair under L1L_FLAG_FORCE_EXACT.
//
// One warp per pair.  The median key is found by bisection over the key
// space: at each probe t the weight of rows with key <= t is summed EXACTLY in
// a wide fixed-point integer whose unit is 2^-1074 (every finite double, and
// so every float, is an integer multiple of it), reduced across the warp limb
// by limb, and compared with the exact total W = sum w + lambda.
//
// Bound by the double divisions of its probes and the latency of one warp's
// chain, so the listed pairs are dealt out over all SMs, CTA by CTA.  One CTA
// of 1024 threads per SM (two do not fit): placed while the pair
// kernel's last CTAs run, two CTAs of 128 per SM went 16 to an SM to the few SMs
// that were free, and all pairs waited for those.  Every pair here (FORCE_EXACT),
// double: 20,480 x 48 265 -> 61 ms, 2000 x 64 46 -> 12 ms; none here: no change
// (200 x 20 fit 27.8 us, against 28.4 us with a launch that is not placed early).
#include <algorithm>

#include "common.cuh"
#include "exact.cuh"
#include "launch.h"

namespace l1l {

constexpr int EX_NT = 1024;  // threads per CTA at most

template <typename T>
__global__ void __launch_bounds__(EX_NT) k_exact(ScanArgs<T> a,
                                                 const __grid_constant__ LambdaPack lp, int t0,
                                                 int nlc) {
    next_may_start();
    wait_for_previous();
    const int lane = threadIdx.x & 31;
    const uint32_t gw = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    const uint32_t nwarps = gridDim.x * (blockDim.x >> 5);
    const uint32_t count = *(volatile uint32_t *)a.slow_count;
    extern __shared__ __align__(16) uint32_t hist[];  // HIST_WORDS per warp
    uint32_t acc[WL];
    uint32_t S[WL], W[WL];  // used by lane 0
    for (uint32_t e = gw; e < count; e += nwarps) {
        const SlowEntry en = a.slow[e];
        listed_entry<T>(a, en, t0, lp.lam, nlc, hist + (threadIdx.x >> 5) * HIST_WORDS, acc, S, W,
                        lane);
    }
}

template <typename T>
cudaError_t launch_exact(const ScanArgs<T> &a, const double *lambdas, int t0, int nlc,
                         int num_sms, cudaStream_t st, int &launches) {
    LambdaPack lp;
    lp.tl_min = lp.tl_max = 0;
    for (int q = 0; q < nlc; ++q) lp.lam[q] = lambdas[t0 + q];
    // little work whatever is listed: four or eight warps to a CTA, as full ones, which the
    // pair kernel's leave no room beside, lengthen an empty launch (200 x 20 fit 27.7 us,
    // 28.5 with them; 1315 x 36 36.8 and 38.4, 343 x 39 29.5 and 30.8).  With more work, sizes
    // of which two or more go to an SM bring the crowding back (every pair listed: 20,480 x
    // 48, 16 warps, 111 ms; 2000 x 64, 8 warps, 0.24 ms, 0.13 with 32; up to the line 0 to 7 us)
    const int64_t most = a.nj * a.m * nlc;
    const int w = most <= 4 * (int64_t)num_sms ? 4 : most * a.n <= (1 << 21) ? 8 : EX_NT / 32;
    const size_t smem = (size_t)w * HIST_WORDS * 4;
    static_assert(EX_NT / 32 * HIST_WORDS * 4 <= 48 * 1024, "needs no opt-in");
    launches++;
    return launch_after(k_exact<T>, dim3(num_sms), dim3((unsigned)w * 32), smem, st, a, lp, t0, nlc);
}

template cudaError_t launch_exact<float>(const ScanArgs<float> &, const double *, int, int, int,
                                         cudaStream_t, int &);
template cudaError_t launch_exact<double>(const ScanArgs<double> &, const double *, int, int, int,
                                          cudaStream_t, int &);

L1L_CHECKS_READER(l1l_checks_exact)

}  // namespace l1l
