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

// On the bits: a comparison would take the FP64 pipe, which bounds the reduction (7 instructions a node;
// 17 with comparisons and separate products: 485 us at 8192 x 2048).
__device__ __forceinline__ bool finite_(double v) { return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000; }

// Block `blk` of RED_BLOCKS: every RED_BLOCKS-th run of RED_THREADS nodes; the four sums of the block go
// to out[0..3].  up, vp: the earlier velocity (NULL: zero), replaced by u, v if keep.
__device__ __forceinline__ void reduce_block_(const double *phi, const double *u, const double *v, const double *T,
                                              double *up, double *vp, long long N, int blk, bool keep, double *out)
{
    double m = 0.0, du2 = 0.0, u2 = 0.0;
    int bad = 0;
    // four nodes in flight per thread (one at a time, with the stores between, waited for memory: 1570 us
    // at 8192 x 2048), added in order
    const long long step = (long long)RED_BLOCKS * RED_THREADS;
    for (long long i0 = blk * (long long)RED_THREADS + threadIdx.x; i0 < N; i0 += 4 * step) {
        double p[4], a[4], b[4], t[4], pa[4], pb[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const long long i = i0 + k * step;
            if (i < N) {
                p[k] = phi[i], a[k] = u[i], b[k] = v[i], t[k] = T[i];
                pa[k] = up ? up[i] : 0.0, pb[k] = vp ? vp[i] : 0.0;
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const long long i = i0 + k * step;
            if (i >= N) break;
            const double da = a[k] - pa[k], db = b[k] - pb[k];
            m += p[k];
            du2 = fma(db, db, fma(da, da, du2));
            u2 = fma(b[k], b[k], fma(a[k], a[k], u2));
            if (!(finite_(p[k]) && finite_(a[k]) && finite_(b[k]) && finite_(t[k]))) ++bad;
            if (keep) up[i] = a[k], vp[i] = b[k];
        }
    }
    __shared__ double sh[4][RED_THREADS / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    m = warp_sum_(m);
    du2 = warp_sum_(du2);
    u2 = warp_sum_(u2);
    bad = __reduce_add_sync(0xffffffffu, bad);
    if (lane == 0) sh[0][wid] = m, sh[1][wid] = du2, sh[2][wid] = u2, sh[3][wid] = double(bad);
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
