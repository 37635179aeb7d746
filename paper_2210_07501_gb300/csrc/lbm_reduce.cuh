// lbm_reduce.cuh -- the field reduction (sum phi, sum |u - u_prev|^2, sum |u|^2, non-finite count) in its
// one order of operations, shared by the handles, the batches and the call that allocates nothing:
// equal fields give equal bits wherever they are summed.
#pragma once

#include <cuda_runtime.h>

namespace lbm {

constexpr int RED_THREADS = 256;
constexpr int RED_BLOCKS = 304;   // 2 x 152 SMs; fixed, so that the order is

__device__ __forceinline__ double warp_sum_(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// Block `blk` of RED_BLOCKS: every RED_BLOCKS-th run of RED_THREADS nodes; the four sums of the block go
// to out[0..3].  up, vp: the earlier velocity (NULL: zero), replaced by u, v if keep.
__device__ __forceinline__ void reduce_block_(const double *phi, const double *u, const double *v, const double *T,
                                              double *up, double *vp, long long N, int blk, bool keep, double *out)
{
    double m = 0.0, du2 = 0.0, u2 = 0.0, bad = 0.0;
    for (long long i = blk * (long long)RED_THREADS + threadIdx.x; i < N; i += (long long)RED_BLOCKS * RED_THREADS) {
        const double p = phi[i], a = u[i], b = v[i], t = T[i];
        const double da = a - (up ? up[i] : 0.0), db = b - (vp ? vp[i] : 0.0);
        m += p;
        du2 += fma(da, da, db * db);
        u2 += fma(a, a, b * b);
        if (!isfinite(p) || !isfinite(a) || !isfinite(b) || !isfinite(t)) bad += 1.0;
        if (keep) up[i] = a, vp[i] = b;
    }
    __shared__ double sh[4][RED_THREADS / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    m = warp_sum_(m);
    du2 = warp_sum_(du2);
    u2 = warp_sum_(u2);
    bad = warp_sum_(bad);
    if (lane == 0) sh[0][wid] = m, sh[1][wid] = du2, sh[2][wid] = u2, sh[3][wid] = bad;
    __syncthreads();
    if (threadIdx.x < 4) {
        double t = 0.0;
        for (int w = 0; w < RED_THREADS / 32; ++w) t += sh[threadIdx.x][w];
        out[threadIdx.x] = t;
    }
}

// The four results from the blocks' sums, 128 threads: a warp per result, its lanes over every 32nd
// block, then the lanes in a tree.  (One thread per result added the 304 in sequence: 17 us a check.)
__device__ __forceinline__ void reduce_blocks_(const double *partials, double *result)
{
    const int q = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double s = 0.0;
#pragma unroll
    for (int b = 0; b < (RED_BLOCKS + 31) / 32; ++b)
        if (lane + 32 * b < RED_BLOCKS) s += partials[4 * (lane + 32 * b) + q];
    s = warp_sum_(s);
    if (lane == 0) result[q] = s;
}

}  // namespace lbm
