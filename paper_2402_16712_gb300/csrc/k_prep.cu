// k_prep.cu -- step A1 (staging) kernels for one instance.
#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "launch.h"
#include "prep.cuh"

namespace cg = cooperative_groups;

namespace l1l {

// grid.x: 32-column tiles; grid.y strides over the 32-row tiles (tall X
// has more of them than a grid dimension holds).
template <typename T>
__global__ void __launch_bounds__(256) k_transpose(const T *__restrict__ X, T *__restrict__ Xt,
                                                   float *__restrict__ Xf,
                                                   int64_t n, int64_t m, int64_t ldn,
                                                   uint32_t *status, int64_t tiles_r) {
    next_may_start();
    for (int64_t tr = blockIdx.y; tr < tiles_r; tr += gridDim.y) {
        transpose_tile<T>(X, Xt, Xf, n, m, ldn, status, blockIdx.x, tr);
        __syncthreads();  // the next row tile refills the shared tile
    }
}

// The same for up to NARROW columns and many rows: a CTA's NR_ROWS rows are one
// contiguous run of X, read 16 bytes a thread (where X is aligned) and written a
// column at a time.  Half or more of a 32 x 32 tile is empty there: 1,000,000 x
// 16 float 73 us (1.8 TB/s), 21 us here.
constexpr int NARROW = 16, NR_ROWS = 256;
template <typename T>
__global__ void __launch_bounds__(256) k_transpose_narrow(const T *__restrict__ X,
                                                          T *__restrict__ Xt,
                                                          float *__restrict__ Xf, int64_t n,
                                                          int m, int64_t ldn, uint32_t *status) {
    using V = typename std::conditional<sizeof(T) == 4, float4, double2>::type;
    constexpr int W = 16 / sizeof(T);
    __shared__ T tile[NR_ROWS * (NARROW + 1)];
    const int64_t r0 = (int64_t)blockIdx.x * NR_ROWS;
    const int rows = (int)std::max<int64_t>(0, std::min<int64_t>(NR_ROWS, n - r0));
    const int total = rows * m, ms = m | 1;  // odd row stride: no bank conflicts
    const T *x = X + r0 * m;
    bool bad = false;
    const bool vec = (reinterpret_cast<uintptr_t>(X) & 15) == 0;  // r0 m is a multiple of W
    for (int e = threadIdx.x * W; e < total; e += 256 * W) {
        T v[W];
        if (vec && e + W <= total) {
            const V q = __ldg(reinterpret_cast<const V *>(x + e));
            v[0] = q.x, v[1] = q.y;
            if constexpr (W == 4) v[2] = q.z, v[3] = q.w;
        } else {
#pragma unroll
            for (int u = 0; u < W; ++u) v[u] = e + u < total ? x[e + u] : T(0);
        }
        int r = e / m, c = e - r * m;
#pragma unroll
        for (int u = 0; u < W; ++u) {
            if (e + u < total) tile[r * ms + c] = v[u];
            bad |= !isfinite(v[u]);
            if (++c == m) {
                c = 0;
                ++r;
            }
        }
    }
    if (__any_sync(0xFFFFFFFFu, bad) && (threadIdx.x & 31) == 0) atomicOr(status, ST_NONFINITE);
    __syncthreads();
    const int r = threadIdx.x;
    if (r0 + r < ldn)
        for (int c = 0; c < m; ++c)
            put_column<T>(Xt, Xf, m, ldn, c, r0 + r, r < rows ? tile[r * ms + c] : T(0));
}

template <typename T>
__global__ void __launch_bounds__(256) k_colprep(const T *__restrict__ Xt, ColInfo *ci,
                                                 int64_t n, int64_t ldn) {
    next_may_start();
    wait_for_previous();
    colprep_column<T>(Xt + (int64_t)blockIdx.x * ldn, ci + blockIdx.x, n);
}

// Block-wide reductions of one value per thread; `red` holds
// the warp partials, `out` receives the result for every thread.
enum { RED_SUM, RED_MAX, RED_MIN };
template <int OP>
__device__ __forceinline__ long long block_reduce_ll(long long x, long long *red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const long long y = __shfl_xor_sync(0xFFFFFFFFu, x, o);
        x = OP == RED_SUM ? x + y : (OP == RED_MAX ? (x > y ? x : y) : (x < y ? x : y));
    }
    __syncthreads();  // red may still be read by an earlier reduction
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
    __syncthreads();
    long long r = red[0];
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
        const long long y = red[w];
        r = OP == RED_SUM ? r + y : (OP == RED_MAX ? (r > y ? r : y) : (r < y ? r : y));
    }
    return r;
}

// Column statistics of tall columns: a cluster of C CTAs per column, each over
// its slice of rows; the two dependent reductions (count and exponent range ->
// sigma; Q and truncations) are combined across the cluster through distributed
// shared memory.  Integer sums, so the result equals the one-CTA version's.  The
// 32-bit weights' totals are left out: only the pair kernel reads them, which
// ends far below these heights.  16 columns of 1,000,000 floats are 128 CTAs, one
// per SM, so the passes are bound by loads in flight: four vectors per thread and
// 1024 threads instead of scalar loads by 512 (and two passes for three), 179 us,
// 79 us.
constexpr int CT_NT = 1024;
template <typename T>
__global__ void __launch_bounds__(CT_NT) k_colprep_tall(const T *__restrict__ Xt, ColInfo *ci,
                                                        int64_t ldn, int64_t rpc) {
    using V = typename std::conditional<sizeof(T) == 4, float4, double2>::type;
    constexpr int W = 16 / sizeof(T), U = 4;
    cg::cluster_group cl = cg::this_cluster();
    const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const int64_t j = blockIdx.x / C;
    const V *col = reinterpret_cast<const V *>(Xt + j * ldn);
    // whole vectors: ldn and rpc are multiples of 128, rows past n are 0
    const int64_t v0 = std::min<int64_t>(ldn, (int64_t)rank * rpc) / W;
    const int64_t v1 = std::min<int64_t>(ldn, (int64_t)(rank + 1) * rpc) / W;
    __shared__ long long red[CT_NT / 32];
    __shared__ long long p1[3], p2[2];  // this CTA's partials, read by the cluster
    auto each = [&](auto &&f) {
        for (int64_t v = v0 + threadIdx.x; v < v1; v += U * CT_NT) {
            V x[U];
#pragma unroll
            for (int u = 0; u < U; ++u) x[u] = v + u * CT_NT < v1 ? __ldg(col + v + u * CT_NT) : V{};
#pragma unroll
            for (int u = 0; u < U; ++u) {
                f(T(x[u].x));
                f(T(x[u].y));
                if constexpr (W == 4) {
                    f(T(x[u].z));
                    f(T(x[u].w));
                }
            }
        }
    };

    int cnt = 0, emax = -100000, emin = 100000;
    each([&](T b) {
        if (b != T(0)) {
            cnt++;
            const int e = ilog2_pos(b);
            emax = max(emax, e);
            emin = min(emin, e);
        }
    });
    long long x0 = block_reduce_ll<RED_SUM>(cnt, red);
    long long x1 = block_reduce_ll<RED_MAX>(emax, red);
    const long long x2 = block_reduce_ll<RED_MIN>(emin, red);
    if (threadIdx.x == 0) {
        p1[0] = x0;
        p1[1] = x1;
        p1[2] = x2;
    }
    cl.sync();
    long long nvl = 0;
    int E = -100000, Emin = 100000;
    for (int r = 0; r < C; ++r) {
        const long long *q = cl.map_shared_rank(&p1[0], r);
        nvl += q[0];
        E = max(E, (int)q[1]);
        Emin = min(Emin, (int)q[2]);
    }
    const int nv = (int)nvl;
    const int sigma = colprep_sigma(nv, E);

    long long qs = 0;
    int inx = 0;
    each([&](T b) {
        int e = 0;
        qs += fixq(absval(b), sigma, e);
        inx += e;
    });
    x0 = block_reduce_ll<RED_SUM>(qs, red);
    x1 = block_reduce_ll<RED_SUM>(inx, red);
    if (threadIdx.x == 0) {
        p2[0] = x0;
        p2[1] = x1;
    }
    cl.sync();
    if (rank == 0 && threadIdx.x == 0) {
        long long Q = 0, I = 0;
        for (int r = 0; r < C; ++r) {
            const long long *q = cl.map_shared_rank(&p2[0], r);
            Q += q[0];
            I += q[1];
        }
        ci[j] = colprep_make<T>(Q, sigma, nv, (int)I, Emin, E, 0, 0, 0);
    }
    cl.sync();  // no CTA leaves while rank 0 may still read its partials
}

template <typename T>
cudaError_t launch_prep(const T *X, T *Xt, float *Xf, ColInfo *ci, int64_t n, int64_t m,
                        int64_t ldn, uint32_t *status, cudaStream_t st, int &launches) {
    dim3 tb(32, 8);
    const int64_t tiles_r = (ldn + 31) / 32;
    dim3 tg((unsigned)((m + 31) / 32), (unsigned)std::min<int64_t>(tiles_r, 65535));
    // fewer rows than that leave SMs without a CTA of NR_ROWS
    if (m <= NARROW && n >= 152 * NR_ROWS)
        k_transpose_narrow<T><<<(unsigned)((ldn + NR_ROWS - 1) / NR_ROWS), 256, 0, st>>>(
            X, Xt, Xf, n, (int)m, ldn, status);
    else
        k_transpose<T><<<tg, tb, 0, st>>>(X, Xt, Xf, n, m, ldn, status, tiles_r);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    launches++;
    const int C = large_cluster_size(ldn);
    if (C == 1) {
        launches++;
        return launch_after(k_colprep<T>, dim3((unsigned)m), dim3(256), 0, st, (const T *)Xt, ci,
                            n, ldn);
    }
    // tall columns: one cluster of C CTAs per column
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(m * C));
    cfg.blockDim = dim3(CT_NT);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    const int64_t rpc = ((ldn + C - 1) / C + ROW_PAD - 1) & ~int64_t(ROW_PAD - 1);
    e = cudaLaunchKernelEx(&cfg, k_colprep_tall<T>, (const T *)Xt, ci, ldn, rpc);
    launches++;
    return e;
}

template cudaError_t launch_prep<float>(const float *, float *, float *, ColInfo *, int64_t,
                                        int64_t, int64_t, uint32_t *, cudaStream_t, int &);
template cudaError_t launch_prep<double>(const double *, double *, float *, ColInfo *, int64_t,
                                         int64_t, int64_t, uint32_t *, cudaStream_t, int &);

}  // namespace l1l
