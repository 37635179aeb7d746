// lbm_cnn.cu -- the learned warm start: a small convolutional surrogate that maps the
// channel's parameters and heating profile to its steady phi, u, v, T, with hand-written
// inference and training kernels (forward, backward-data, backward-weight, loss, Adam).
//
// Network: 6 layers of 3x3 convolutions, channels 12 -> 32 -> 32 -> 32 -> 32 -> 32 -> 4, SiLU
// between layers, none after the last.  Periodic in x (the channel is periodic), zero
// padding in y.  Weights, gradients and optimiser state are FP32; activations are stored in
// BF16 (or FP32, for gradient checks), every accumulation is FP32.  Layout NCHW.
// Deterministic: the weight gradients are summed in a fixed order (two passes).
#include <cuda_bf16.h>
#include <math.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>

#include <new>
#include <type_traits>
#include <vector>

#include "../../include/lbm_gb300.h"
#include "lbm_pdl.h"

namespace {

constexpr int NL = 6;
constexpr int CH[NL + 1] = {12, 32, 32, 32, 32, 32, 4};
template <typename A> __device__ __forceinline__ float to_f(A v)
{
    if constexpr (std::is_same<A, __nv_bfloat16>::value) return __bfloat162float(v);
    else return v;
}
template <typename A> __device__ __forceinline__ A from_f(float v)
{
    if constexpr (std::is_same<A, __nv_bfloat16>::value) return __float2bfloat16_rn(v);
    else return v;
}
// a float as the activation type holds it
template <typename A> __device__ __forceinline__ float rounded(float v) { return to_f(from_f<A>(v)); }
__device__ __forceinline__ float silu(float z) { return z / (1.0f + __expf(-z)); }
__device__ __forceinline__ float dsilu(float z)
{
    const float s = 1.0f / (1.0f + __expf(-z));
    return s * (1.0f + z * (1.0f - s));
}

// four consecutive aligned values
__device__ __forceinline__ void load4(const float *p, float *v)
{
    const float4 u = *reinterpret_cast<const float4 *>(p);
    v[0] = u.x, v[1] = u.y, v[2] = u.z, v[3] = u.w;
}
__device__ __forceinline__ void store4(float *p, const float *v)
{
    *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void load4(const __nv_bfloat16 *p, __nv_bfloat16 *v)
{
    const uint2 u = *reinterpret_cast<const uint2 *>(p);
    reinterpret_cast<uint32_t *>(v)[0] = u.x, reinterpret_cast<uint32_t *>(v)[1] = u.y;
}
__device__ __forceinline__ void store4(__nv_bfloat16 *p, const __nv_bfloat16 *v)
{
    const uint32_t *w = reinterpret_cast<const uint32_t *>(v);
    *reinterpret_cast<uint2 *>(p) = make_uint2(w[0], w[1]);
}
// s + c + x -> s + c: x onto the sum s, the rounding error onto c (Knuth's two-sum: exact in s + c). total: the
// sum rounded once; an infinite or overflowed s has no error to add.
__device__ __forceinline__ void add_exact(float &s, float &c, float x)
{
    const float t = s + x, z = t - s;
    c += (s - (t - z)) + (x - z);
    s = t;
}
__device__ __forceinline__ float total(float s, float c) { return isfinite(s) ? s + c : s; }
__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

// ---- 3x3 convolutions on the FP32 pipes ----------------------------------------------------
// Forward (BWD = false): y[b][co][h][w] = bias[co] + sum_{ci, dy, dx} w[co][ci][dy][dx] a[b][ci][h+dy-1][w+dx-1].
// Data gradient (BWD = true): the same sum over the layer's output channels with the kernel flipped, times
// silu'(z) of the pixel; silu(z) goes to act if given, for the weight gradient that follows.
//
// Bound: FP32 multiply-adds (2.4 G per 32 -> 32 layer at batch 16 of 256 x 64: 62 us at 80 TFLOP/s).  The
// weights are kept in FP32 and the sums in FP32 in one order (per input channel the nine taps in
// sequence, then the channel's sum onto the accumulator), which the matrix units cannot give.
// The weights come laid out as they are read: [input][tap][output], for the data gradient flipped and
// with the layer's channels swapped (weight_place, kept by set_params and the Adam step).
// A thread holds 4 pixels of a row x COG output channels: per weight quad from shared memory (one
// 16-byte broadcast) 8 packed FMAs (two channels each), per input channel 18 input values for 36 taps.
// The inputs come as the values that are multiplied, in float (silu is applied once, where the layer
// before stores), so staging is asynchronous copies, the next channels' while these are multiplied.
// 110 us a 32 -> 32 layer at 16 x 256 x 64, 0.6 of the FP32 peak (304 us with one pixel a thread and one
// scalar FMA per weight read; 124 with silu and its division applied on staging).
constexpr int CCH = 8;         // input channels staged per pass
template <int CO, int COG_, int TWQ_, int TH_> struct Tile {
    static constexpr int COG = COG_, TWQ = TWQ_, TH = TH_;   // channels a thread, pixel quads a row, rows
    static constexpr int NC = TWQ * TH * (CO / COG);         // threads that compute
    static constexpr int NT = NC < 128 ? 128 : NC;           // threads (all stage)
};

// ---- staging by asynchronous copies ----
__device__ __forceinline__ void copy_async16(float *dst, const float *src, bool in)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
                 "r"(in ? 16 : 0)
                 : "memory");
}
__device__ __forceinline__ void copy_async4(float *dst, const float *src, bool in)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
                 "r"(in ? 4 : 0)
                 : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// The rows iy < ROWS (image rows h0 - 1 + iy, zero outside) of nc planes of x into dst[c PLANE + iy PW +
// 4 + column]: COLS columns from w0 on, the column before at 3 and the one after (wrapped: the image
// is periodic in x; past the wrapped one zero).  vec: W a multiple of 4 and x on a 16-byte boundary.
template <int NT, int COLS, int ROWS, int PW, int PLANE>
__device__ __forceinline__ void stage_planes(const float *x, int nc, int h0, int w0, int H, int W, float *dst, bool vec)
{
    const int rows = nc * ROWS;
    if (vec) {
        for (int e = threadIdx.x; e < rows * (COLS / 4); e += NT) {
            const int r = e / (COLS / 4), q = e % (COLS / 4), c = r / ROWS, iy = r - c * ROWS, hh = h0 + iy - 1;
            const int ww = w0 + 4 * q;
            float *d = dst + c * PLANE + iy * PW + 4 + 4 * q;
            const bool in = hh >= 0 && hh < H;
            const float *row = x + ((long long)c * H + (in ? hh : 0)) * W;
            if (ww < W) copy_async16(d, row + ww, in);
            else *reinterpret_cast<float4 *>(d) = make_float4(ww == W && in ? row[0] : 0.f, 0.f, 0.f, 0.f);
        }
        for (int e = threadIdx.x; e < 2 * rows; e += NT) {
            const int r = e >> 1, c = r / ROWS, iy = r - c * ROWS, hh = h0 + iy - 1;
            const int ww = e & 1 ? w0 + COLS : (w0 == 0 ? W - 1 : w0 - 1);
            const bool in = hh >= 0 && hh < H && ww <= W;
            copy_async4(dst + c * PLANE + iy * PW + (e & 1 ? 4 + COLS : 3),
                        x + ((long long)c * H + (in ? hh : 0)) * W + (ww < W ? ww : 0), in);
        }
    } else {
        for (int e = threadIdx.x; e < rows * (COLS + 2); e += NT) {
            const int r = e / (COLS + 2), ix = e - r * (COLS + 2), c = r / ROWS, iy = r - c * ROWS, hh = h0 + iy - 1;
            const int ww = w0 + ix - 1;
            const bool in = hh >= 0 && hh < H && ww <= W;
            copy_async4(dst + c * PLANE + iy * PW + 3 + ix,
                        x + ((long long)c * H + (in ? hh : 0)) * W + (ww < 0 ? W - 1 : (ww < W ? ww : 0)), in);
        }
    }
}

template <int CI, int CO, typename T, bool BWD, bool LAST, typename A, typename Out>
__global__ void __launch_bounds__(T::NT, 512 / T::NT)
conv3x3(const float *x, const float *wgt, const float *bias, const A *zin, Out *y, float *act, int H, int W, bool vec_in)
{
    constexpr int COG = T::COG, TWQ = T::TWQ, TH = T::TH, NT = T::NT;
    constexpr int PW = TWQ * 4 + 8, PLANE = (TH + 2) * PW, NCHUNK = (CI + CCH - 1) / CCH;
    constexpr int STAGES = NCHUNK > 1 ? 2 : 1;
    __shared__ __align__(16) float s_x[STAGES][CCH * PLANE];
    __shared__ __align__(16) float s_w[STAGES][CCH * 9 * CO];
    const int q = threadIdx.x % TWQ, row = threadIdx.x / TWQ % TH, cg = threadIdx.x / (TWQ * TH);
    const bool on = T::NC == NT || threadIdx.x < T::NC;
    const int tw = (W + TWQ * 4 - 1) / (TWQ * 4), ty = blockIdx.x / tw, b = blockIdx.z;
    const int w0 = (blockIdx.x - ty * tw) * (TWQ * 4), h0 = ty * TH;
    lbm::pdl_wait_();   // (no __restrict__: nothing may be read before the wait)
    auto stage = [&](int k) {   // channels k CCH .. of the input and their weights, one copy group
        const int c0 = k * CCH, nc = CI - c0 < CCH ? CI - c0 : CCH;
        for (int e = threadIdx.x; e < nc * 9 * CO / 4; e += NT)
            copy_async16(s_w[k % STAGES] + 4 * e, wgt + c0 * 9 * CO + 4 * e, true);
        stage_planes<NT, TWQ * 4, TH + 2, PW, PLANE>(x + ((long long)b * CI + c0) * H * W, nc, h0, w0, H, W,
                                                     s_x[k % STAGES], vec_in);
        copy_commit();
    };
    stage(0);
    float2 acc[4][COG / 2];
#pragma unroll
    for (int j = 0; j < COG / 2; ++j) {
        const float2 v = BWD || !on ? f2(0.f, 0.f) : f2(bias[cg * COG + 2 * j], bias[cg * COG + 2 * j + 1]);
#pragma unroll
        for (int p = 0; p < 4; ++p) acc[p][j] = v;
    }
#pragma unroll 1
    for (int k = 0; k < NCHUNK; ++k) {
        if (k + 1 < NCHUNK) {
            stage(k + 1);
            copy_wait<1>();
        } else {
            copy_wait<0>();
        }
        __syncthreads();
        const int nc = CI - k * CCH < CCH ? CI - k * CCH : CCH;
        if (on)
#pragma unroll 1
            for (int c = 0; c < nc; ++c) {
                const float *xs = s_x[k % STAGES] + c * PLANE + row * PW + 4 * q;
                float xv[3][6];
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    const float4 u = *reinterpret_cast<const float4 *>(xs + i * PW + 4);
                    xv[i][0] = xs[i * PW + 3], xv[i][1] = u.x, xv[i][2] = u.y, xv[i][3] = u.z, xv[i][4] = u.w;
                    xv[i][5] = xs[i * PW + 8];
                }
                const float *ws = s_w[k % STAGES] + c * 9 * CO + cg * COG;
#pragma unroll
                for (int j = 0; j < COG / 2; j += 2) {
                    float2 sa[4], sb[4];
#pragma unroll
                    for (int p = 0; p < 4; ++p) sa[p] = sb[p] = f2(0.f, 0.f);
#pragma unroll
                    for (int t = 0; t < 9; ++t) {
                        const float4 u = *reinterpret_cast<const float4 *>(ws + t * CO + 2 * j);
#pragma unroll
                        for (int p = 0; p < 4; ++p) {
                            const float v = xv[t / 3][t % 3 + p];
                            sa[p] = fma2(f2(u.x, u.y), f2(v, v), sa[p]);
                            sb[p] = fma2(f2(u.z, u.w), f2(v, v), sb[p]);
                        }
                    }
#pragma unroll
                    for (int p = 0; p < 4; ++p) {
                        acc[p][j] = __fadd2_rn(acc[p][j], sa[p]);
                        acc[p][j + 1] = __fadd2_rn(acc[p][j + 1], sb[p]);
                    }
                }
            }
        if (k + 1 < NCHUNK) __syncthreads();   // the next round's copies go where this one read
    }
    lbm::pdl_launch_next_();
    const int ho = h0 + row, wo = w0 + 4 * q;
    if (!on || ho >= H) return;
    const bool quad = W % 4 == 0;   // then the four pixels lie in the image together, aligned in the library's buffers
#pragma unroll
    for (int j = 0; j < COG; ++j) {
        const long long o = (((long long)b * CO + cg * COG + j) * H + ho) * W + wo;
        float v[4];
#pragma unroll
        for (int p = 0; p < 4; ++p) v[p] = j & 1 ? acc[p][j / 2].y : acc[p][j / 2].x;
        if constexpr (BWD) {
            if (quad) {
                if (wo < W) {
                    __align__(8) A z[4];
                    load4(zin + o, z);
                    *reinterpret_cast<float4 *>(y + o) = make_float4(v[0] * dsilu(to_f(z[0])), v[1] * dsilu(to_f(z[1])),
                                                                     v[2] * dsilu(to_f(z[2])), v[3] * dsilu(to_f(z[3])));
                    if (act)
                        *reinterpret_cast<float4 *>(act + o) =
                            make_float4(silu(to_f(z[0])), silu(to_f(z[1])), silu(to_f(z[2])), silu(to_f(z[3])));
                }
            } else {
#pragma unroll
                for (int p = 0; p < 4; ++p)
                    if (wo + p < W) {
                        const float z = to_f(zin[o + p]);
                        y[o + p] = v[p] * dsilu(z);
                        if (act) act[o + p] = silu(z);
                    }
            }
        } else if constexpr (LAST) {
#pragma unroll
            for (int p = 0; p < 4; ++p)
                if (wo + p < W) {
                    if constexpr (std::is_same<Out, A>::value) y[o + p] = from_f<A>(v[p]);
                    else y[o + p] = rounded<A>(v[p]);
                }
        } else {   // the pre-activation as the activation type holds it, and silu of that
            __align__(8) A z[4];
            float s[4];
#pragma unroll
            for (int p = 0; p < 4; ++p) z[p] = from_f<A>(v[p]), s[p] = silu(to_f(z[p]));
            if (quad) {
                if (wo < W) {
                    store4(y + o, z);
                    *reinterpret_cast<float4 *>(act + o) = make_float4(s[0], s[1], s[2], s[3]);
                }
            } else {
#pragma unroll
                for (int p = 0; p < 4; ++p)
                    if (wo + p < W) y[o + p] = z[p], act[o + p] = s[p];
            }
        }
    }
}

// ---- weight and bias gradients -------------------------------------------------------------
// dw[co][ci][k] = sum_p a[ci][p + k] dz[co][p], db[co] = sum_p dz[co][p], over all pixels.  A contraction
// over the pixels with 32 x 288 results: a thread holds 4 output channels x 1 input channel x 9 taps, each as
// the packed sums of its even and odd columns (72 registers; with the operands 128, so the 36 sums
// over the tiles are spilled and touched once a tile); per four pixels 72 packed FMAs on 3 + 4
// 16-byte shared loads (the inputs by lane, the dz by broadcast).  A CTA walks over tiles of 8 x 32
// pixels, and only gridDim partial sums reach memory (before: one per 16 x 16 tile, reduced by one
// strided thread per result, 154 us a layer).  140 us a 32 -> 32 layer, 718 us with one FMA per two
// shared loads.
// Order of the sums: the two chains of 128 pixels of a tile, up to GRUN tiles in FP32 (so no FP32 chain is
// longer than the 256 pixels of a 16 x 16 tile), and those runs, where a CTA has more tiles than one
// (LONG), with their rounding errors carried along.  Carrying them tile by tile cost 4 % of a training
// step at 16 x 256 x 64 (3 to 4 tiles a CTA), the code for it alone 1 %, hence the two instances;
// without it the gradients of 16 x 512 x 512 images of constant dz were 4e-7 off.
constexpr int GW = 32, GH = 8, GT = 256, GRUN = 4;
constexpr int GP = GW + 8, GPLANE = (GH + 2) * GP + 4;   // plane stride = 4 x odd words: no bank conflicts
static_assert(GPLANE % 32 % 8 == 4, "16-byte loads of 8 lanes must hit distinct banks");
constexpr int GD = GH * GW;
template <int CI, int CO> constexpr int grad_groups() { return GT / (CI * CO / 4) < GH ? GT / (CI * CO / 4) : GH; }
template <int CI, int CO> constexpr size_t grad_smem() { return (CI * GPLANE + CO * GD) * sizeof(float); }

template <int CI, int CO, bool LONG>
__global__ void __launch_bounds__(GT, 2) conv_grad(const float *x, const float *dz, float *part, int H, int W, int B,
                                                   bool vec_in)
{
    constexpr int NG = grad_groups<CI, CO>(), PER = CI * CO / 4, NW = CO * CI * 9;
    constexpr int BL = GT / CO;   // threads per bias sum
    extern __shared__ __align__(16) float s_a[];   // [CI][GPLANE], then dz [CO][GH][GW]
    float *s_d = s_a + CI * GPLANE;
    const int t = threadIdx.x, ci = t % CI, cog = t / CI % (CO / 4), grp = t / PER;
    const bool on = grp < NG;
    float tot[4][9], db = 0.f, db_err = 0.f;
    float sum[LONG ? 36 : 1], err[LONG ? 36 : 1];   // LONG: the earlier runs' sums, once flushed
    int n_run = 0;                                  // tiles in tot
    bool flushed = false;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int k = 0; k < 9; ++k) tot[i][k] = 0.f;
    const int tw = (W + GW - 1) / GW, th = (H + GH - 1) / GH, tiles = tw * th * B;
    lbm::pdl_wait_();
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int b = tile / (tw * th), r0 = tile - b * (tw * th), h0 = r0 / tw * GH, w0 = r0 % tw * GW;
        __syncthreads();
        stage_planes<GT, GW, GH + 2, GP, GPLANE>(x + (long long)b * CI * H * W, CI, h0, w0, H, W, s_a, vec_in);
        const float *dzb = dz + (long long)b * CO * H * W;   // dz: zero outside
        if (W % 4 == 0) {
            for (int e = t; e < CO * GD / 4; e += GT) {
                const int c = e / (GD / 4), r = e - c * (GD / 4), hh = h0 + r / (GW / 4), ww = w0 + r % (GW / 4) * 4;
                const bool in = hh < H && ww < W;
                copy_async16(s_d + 4 * e, dzb + ((long long)c * H + (in ? hh : 0)) * W + (in ? ww : 0), in);
            }
        } else {
            for (int e = t; e < CO * GD; e += GT) {
                const int c = e / GD, r = e - c * GD, hh = h0 + r / GW, ww = w0 + r % GW;
                const bool in = hh < H && ww < W;
                copy_async4(s_d + e, dzb + ((long long)c * H + (in ? hh : 0)) * W + (in ? ww : 0), in);
            }
        }
        copy_commit();
        copy_wait<0>();
        __syncthreads();
        {
            float s = 0.f;   // the thread's share of a bias sum: columns t % BL, + BL, ..
            const float *d = s_d + t / BL * GD;
            for (int p = t % BL; p < GD; p += BL) s += d[p];
            add_exact(db, db_err, s);
        }
        if (!on) continue;
        float2 acc[4][9];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int k = 0; k < 9; ++k) acc[i][k] = f2(0.f, 0.f);
#pragma unroll 1
        for (int y = grp; y < GH; y += NG) {
            const float *as = s_a + ci * GPLANE + y * GP, *ds = s_d + 4 * cog * GD + y * GW;
            float4 cur[3];      // columns c .. c + 3 of the image rows y - 1 .. y + 1, and the one before
            float before[3];
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                before[i] = as[i * GP + 3];
                cur[i] = *reinterpret_cast<const float4 *>(as + i * GP + 4);
            }
#pragma unroll 2
            for (int c = 0; c < GW; c += 4) {
                float4 d[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) d[i] = *reinterpret_cast<const float4 *>(ds + i * GD + c);
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    const float4 u = cur[i], n = *reinterpret_cast<const float4 *>(as + i * GP + c + 8);
                    const float2 m = f2(u.y, u.z);
                    const float2 p0[3] = {f2(before[i], u.x), f2(u.x, u.y), m};
                    const float2 p1[3] = {m, f2(u.z, u.w), f2(u.w, n.x)};
#pragma unroll
                    for (int o = 0; o < 4; ++o)
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            acc[o][3 * i + k] = fma2(p0[k], f2(d[o].x, d[o].y), acc[o][3 * i + k]);
                            acc[o][3 * i + k] = fma2(p1[k], f2(d[o].z, d[o].w), acc[o][3 * i + k]);
                        }
                    before[i] = u.w;
                    cur[i] = n;
                }
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int k = 0; k < 9; ++k) tot[i][k] += acc[i][k].x + acc[i][k].y;
        if constexpr (LONG)
            if (++n_run == GRUN && tile + gridDim.x < tiles) {
#pragma unroll
                for (int i = 0; i < 36; ++i) {
                    if (!flushed) sum[i] = err[i] = 0.f;
                    add_exact(sum[i], err[i], tot[i / 9][i % 9]);
                    tot[i / 9][i % 9] = 0.f;
                }
                flushed = true;
                n_run = 0;
            }
    }
    if constexpr (LONG)
        if (flushed)
#pragma unroll
            for (int i = 0; i < 36; ++i) {
                add_exact(sum[i], err[i], tot[i / 9][i % 9]);
                tot[i / 9][i % 9] = total(sum[i], err[i]);
            }
    lbm::pdl_launch_next_();
    // the pixel groups' sums onto the first group's, in sequence, through shared memory
    if constexpr (NG > 1) {
        static_assert((NG - 1) * PER * 36 * sizeof(float) <= grad_smem<CI, CO>(), "the groups' sums fit the tile's memory");
        __syncthreads();
        if (on && grp > 0)
#pragma unroll
            for (int i = 0; i < 36; ++i)
                s_a[((grp - 1) * 36 + i) * PER + t % PER] = tot[i / 9][i % 9];
        __syncthreads();
        if (grp == 0)
#pragma unroll
            for (int i = 0; i < 36; ++i) {
                float v = tot[i / 9][i % 9], e = 0.f;
                for (int g = 0; g < NG - 1; ++g) add_exact(v, e, s_a[(g * 36 + i) * PER + t]);
                tot[i / 9][i % 9] = total(v, e);
            }
    }
    db = total(db, db_err);
    float *out = part + (long long)blockIdx.x * (NW + CO);
    if (grp == 0)
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int k = 0; k < 9; ++k) out[((4 * cog + i) * CI + ci) * 9 + k] = tot[i][k];
#pragma unroll
    for (int o = BL / 2 < 16 ? BL / 2 : 16; o > 0; o >>= 1) db += __shfl_down_sync(0xffffffffu, db, o);
    constexpr int PB = BL > 32 ? BL / 32 : 1;   // warps per bias sum
    __syncthreads();
    if (t % 32 % BL == 0) s_a[t / (BL < 32 ? BL : 32)] = db;
    __syncthreads();
    if (t < CO) {
        float v = s_a[t * PB];
        for (int i = 1; i < PB; ++i) v += s_a[t * PB + i];
        out[NW + t] = v;
    }
}

// MSE loss on the last layer: dz = 2 (y - t) / N; per-block partial sums of (y - t)^2.
template <typename A>
__global__ void mse_grad(const A *__restrict__ y, const float *__restrict__ t, long long n, float *__restrict__ dz,
                         double *__restrict__ part)
{
    __shared__ double sh[256];
    double s = 0.0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const float d = to_f(y[i]) - t[i];
        dz[i] = 2.0f * d / (float)n;
        s += (double)d * d;
    }
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

// The input as the activation type holds it, in float (what the convolutions read).  Twice a training
// step: a dependent launch, like its neighbours, which lets the next one start only at its end (the
// convolution's CTAs would settle among its own: 121 us a prediction at 16 x 64 x 32 instead of 112).
template <typename A> __global__ void __launch_bounds__(256) round_input(const float *x, float *y, long long n)
{
    lbm::pdl_wait_();   // (no __restrict__: nothing may be read before the wait)
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        y[i] = rounded<A>(x[i]);
}

// Where parameter i = weight [co][ci][k] of its layer goes in the two layouts the convolutions read;
// false for a bias.
struct Layers {
    int n, off_w[NL], off_b[NL];
};
__device__ __forceinline__ bool weight_place(const Layers &L, int i, int &fwd, int &bwd)
{
    constexpr int ch[NL + 1] = {12, 32, 32, 32, 32, 32, 4};
    int l = 0;
    while (l + 1 < NL && i >= L.off_w[l + 1]) ++l;
    if (i >= L.off_b[l]) return false;
    const int r = i - L.off_w[l], co = r / (ch[l] * 9), ci = r / 9 % ch[l], k = r % 9;
    fwd = L.off_w[l] + (ci * 9 + k) * ch[l + 1] + co;
    bwd = L.off_w[l] + (co * 9 + 8 - k) * ch[l] + ci;
    return true;
}

// grad[j] = sum over the n_part partial sums of its layer (layer l's lie at part + n_part off_w[l],
// [n_part][parameters of the layer]), in a fixed order: 8 threads per result, each every 8th
// partial sum, then the 8 in sequence.  The threads' sums carry their rounding errors along (two-sum:
// as good as FP64, whose one pipe per SM alone would take 20 us for the 12.7 M terms of the largest
// batch); the last eight are added in FP64.
__global__ void __launch_bounds__(256) reduce_parts(const float *part, int n_part, Layers L, float *grad)
{
    __shared__ double sh[8][32];
    const int lane = threadIdx.x % 32, g = threadIdx.x / 32, j = blockIdx.x * 32 + lane;
    int l = 0;
    while (l + 1 < NL && j >= L.off_w[l + 1]) ++l;
    const int n = (l + 1 < NL ? L.off_w[l + 1] : L.n) - L.off_w[l];
    const float *p0 = part + (long long)n_part * L.off_w[l] + (j - L.off_w[l]);
    lbm::pdl_wait_();
    float s = 0.f, c = 0.f;
    if (j < L.n) {
#pragma unroll 8
        for (int p = g; p < n_part; p += 8) {
            const float x = p0[(long long)p * n], t = s + x, z = t - s;
            c += (s - (t - z)) + (x - z);
            s = t;
        }
    }
    double d = (double)s + (double)c;
    if (!isfinite(s)) {   // infinite or overflowed: its rounding errors mean nothing
        d = 0.0;
        for (int p = g; p < n_part; p += 8) d += p0[(long long)p * n];
    }
    sh[g][lane] = d;
    __syncthreads();
    if (g == 0 && j < L.n) {
        d = sh[0][lane];
        for (int i = 1; i < 8; ++i) d += sh[i][lane];
        grad[j] = (float)d;
    }
}

__global__ void lay_out(const float *__restrict__ p, float *__restrict__ pf, float *__restrict__ pb, Layers L)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    int f, b;
    if (i < L.n && weight_place(L, i, f, b)) pf[f] = p[i], pb[b] = p[i];
}

__global__ void adam_step(float *__restrict__ p, float *__restrict__ pf, float *__restrict__ pb,
                          const float *__restrict__ g, float *__restrict__ m, float *__restrict__ v, Layers L, float lr,
                          float b1, float b2, float eps, float c1, float c2)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= L.n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float pi = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    p[i] = pi;
    int f, b;
    if (weight_place(L, i, f, b)) pf[f] = pi, pb[b] = pi;
}

}  // namespace

struct lbm_cnn {
    int H = 0, W = 0, Bmax = 0, bf16 = 1;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    int n_params = 0, sms = 0;
    Layers L;
    float *p = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;   // params, grads, Adam state
    float *pf = nullptr, *pb = nullptr;   // the weights as the convolutions read them (weight_place)
    void *z[NL + 1] = {nullptr};      // z[l+1] = pre-activation output of layer l, in the activation type
    // Of what the layers read, in float (the rounded input with BF16 activations, then silu(z[l])), only what
    // is being read is held: forward, the layers' in the two dz, the input's in act; backward, the last two
    // layers' where the forward pass left them, then act, formed again from z beside each data
    // gradient.  (Kept for every layer they took 688 bytes a pixel, 1272 in all with BF16; now 712.)
    float *act = nullptr;
    float *dz[2] = {nullptr, nullptr};
    float *part = nullptr;            // partial weight gradients
    double *loss_part = nullptr, *loss_host = nullptr;
    int64_t t = 0;                    // Adam step
};

static thread_local char g_cnn_err[160] = "";

// Whether rows of W floats at x can be copied 16 bytes at a time.
static bool aligned_rows(const void *x, int W) { return W % 4 == 0 && reinterpret_cast<uintptr_t>(x) % 16 == 0; }

template <typename K, typename... Args>
static cudaError_t go(lbm_cnn *c, K kernel, dim3 grid, int block, size_t smem, Args... args)
{
    lbm::PdlLaunch l(grid, dim3(block), smem, c->stream);
    return cudaLaunchKernelEx(&l.cfg, kernel, args...);
}

// One convolution.  Tiles of 32 x 8 pixels (16 channels a thread) where they fill the GPU, else of
// 16 x 8 (8 channels a thread: half the pixels per CTA, 1.25 times the time per pixel).
template <int CI, int CO, bool BWD, bool LAST, typename A, typename Out>
static cudaError_t conv(lbm_cnn *c, int B, const float *x, const float *w, const float *bias, const A *zin, Out *y, float *act)
{
    using Big = Tile<CO, CO < 16 ? CO : 16, 8, 8>;
    using Small = Tile<CO, CO < 8 ? CO : 8, 4, 8>;
    const int rows = (c->H + 7) / 8;
    const dim3 gb((unsigned)((c->W + 31) / 32) * rows, 1, B), gs((unsigned)((c->W + 15) / 16) * rows, 1, B);
    const long long nb = (long long)gb.x * B, ns = (long long)gs.x * B;
    const double tb = 2.0 * ((nb + 4 * c->sms - 1) / (4 * c->sms)), ts = 1.25 * ((ns + 4 * c->sms - 1) / (4 * c->sms));
    const bool vec = aligned_rows(x, c->W);
    if (tb <= ts)
        return go(c, conv3x3<CI, CO, Big, BWD, LAST, A, Out>, gb, Big::NT, 0, x, w, bias, zin, y, act, c->H, c->W, vec);
    return go(c, conv3x3<CI, CO, Small, BWD, LAST, A, Out>, gs, Small::NT, 0, x, w, bias, zin, y, act, c->H, c->W, vec);
}

// What the first layer reads: the caller's input, or a copy in act rounded to the activation type.
template <typename A> static cudaError_t first_input(lbm_cnn *c, const float *x, int B, const float **in)
{
    *in = c->bf16 ? c->act : x;
    if (!c->bf16) return cudaSuccess;
    return go(c, round_input<A>, dim3(1024), 256, 0, x, c->act, (long long)B * CH[0] * c->H * c->W);
}

// Forward pass; the last layer's output goes to y (its activation type, or float).
template <typename A, typename Out> static cudaError_t cnn_forward_impl(lbm_cnn *c, const float *x, int B, Out *y)
{
    const A *none = nullptr;
    float *no_act = nullptr;
    const float *w = c->pf, *p = c->p;
    const int *ow = c->L.off_w, *ob = c->L.off_b;
    const float *in;
    cudaError_t e = first_input<A>(c, x, B, &in);
    if (e == cudaSuccess) e = conv<CH[0], 32, false, false>(c, B, in, w + ow[0], p + ob[0], none, (A *)c->z[1], c->dz[0]);
    for (int l = 1; l < NL - 1 && e == cudaSuccess; ++l)
        e = conv<32, 32, false, false>(c, B, (const float *)c->dz[(l - 1) & 1], w + ow[l], p + ob[l], none, (A *)c->z[l + 1],
                                       c->dz[l & 1]);
    if (e == cudaSuccess)
        e = conv<32, 4, false, true>(c, B, (const float *)c->dz[(NL - 2) & 1], w + ow[NL - 1], p + ob[NL - 1], none, y, no_act);
    return e;
}

// Two CTAs per SM walk over the tiles (fewer where there are fewer tiles).
static long long grad_tiles(const lbm_cnn *c, int B) { return (long long)((c->W + GW - 1) / GW) * ((c->H + GH - 1) / GH) * B; }
static int grad_ctas(const lbm_cnn *c, int B)
{
    const long long tiles = grad_tiles(c, B);
    return (int)(tiles < 2 * c->sms ? tiles : 2 * c->sms);
}

template <int CI, int CO> static cudaError_t conv_gradient(lbm_cnn *c, int l, int B, const float *x, const float *dz)
{
    constexpr size_t sm = grad_smem<CI, CO>();
    const int ctas = grad_ctas(c, B);
    auto *kernel = grad_tiles(c, B) > (long long)GRUN * ctas ? conv_grad<CI, CO, true> : conv_grad<CI, CO, false>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e == cudaSuccess)
        e = go(c, kernel, dim3(ctas), GT, sm, x, dz, c->part + (size_t)ctas * c->L.off_w[l], c->H, c->W, B,
               aligned_rows(x, c->W));
    return e;
}

template <typename A>
static cudaError_t cnn_backward_impl(lbm_cnn *c, const float *x, int B, const float *target, double *loss)
{
    const long long nout = (long long)B * CH[NL] * c->H * c->W;
    const int lb = 512;
    mse_grad<A><<<lb, 256, 0, c->stream>>>((const A *)c->z[NL], target, nout, c->act, c->loss_part);
    cudaError_t e = cudaGetLastError();
    const float *w = c->pb, *none = nullptr, *in;
    const int *ow = c->L.off_w;
    float *no_act = nullptr, *last = c->act;
    // the inputs of the last two layers are in dz[0] and dz[1]
    if (e == cudaSuccess) e = conv_gradient<32, 4>(c, NL - 1, B, c->dz[0], last);
    if (e == cudaSuccess)
        e = conv<4, 32, true, false>(c, B, (const float *)last, w + ow[NL - 1], none, (const A *)c->z[NL - 1], c->dz[0], no_act);
    if (e == cudaSuccess) e = conv_gradient<32, 32>(c, NL - 2, B, c->dz[1], c->dz[0]);
    if (e == cudaSuccess)
        e = conv<32, 32, true, false>(c, B, (const float *)c->dz[0], w + ow[NL - 2], none, (const A *)c->z[NL - 2], c->dz[1],
                                      no_act);
    int cur = 1;
    for (int l = NL - 3; l > 0 && e == cudaSuccess; --l, cur = 1 - cur) {   // the data gradient first: it forms the input
        e = conv<32, 32, true, false>(c, B, (const float *)c->dz[cur], w + ow[l], none, (const A *)c->z[l], c->dz[1 - cur],
                                      c->act);
        if (e == cudaSuccess) e = conv_gradient<32, 32>(c, l, B, c->act, c->dz[cur]);
    }
    if (e == cudaSuccess) e = first_input<A>(c, x, B, &in);
    if (e == cudaSuccess) e = conv_gradient<CH[0], 32>(c, 0, B, in, c->dz[cur]);
    if (e == cudaSuccess)
        e = go(c, reduce_parts, dim3((c->n_params + 31) / 32), 256, 0, (const float *)c->part, grad_ctas(c, B), c->L, c->g);
    if (e != cudaSuccess) return e;
    e = cudaMemcpyAsync(c->loss_host, c->loss_part, lb * sizeof(double), cudaMemcpyDeviceToHost, c->stream);
    if (e != cudaSuccess) return e;
    e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) return e;
    double s = 0.0;
    for (int i = 0; i < lb; ++i) s += c->loss_host[i];
    if (loss) *loss = s / (double)nout;
    return cudaSuccess;
}

static cudaError_t lay_out_weights(lbm_cnn *c)
{
    lay_out<<<(c->n_params + 255) / 256, 256, 0, c->stream>>>(c->p, c->pf, c->pb, c->L);
    return cudaGetLastError();
}

static int cnn_fail(cudaError_t e, const char *what)
{
    snprintf(g_cnn_err, sizeof(g_cnn_err), "%s: %s", what, cudaGetErrorString(e));
    return LBM_ECUDA;
}

extern "C" {

void lbm_cnn_destroy(lbm_cnn *c)
{
    if (!c) return;
    if (c->stream) cudaStreamSynchronize(c->stream);
    float *fs[] = {c->p, c->pf, c->pb, c->g, c->m, c->v, c->dz[0], c->dz[1], c->act, c->part};
    for (float *f : fs)
        if (f) cudaFree(f);
    for (int l = 0; l <= NL; ++l)
        if (c->z[l]) cudaFree(c->z[l]);
    if (c->loss_part) cudaFree(c->loss_part);
    if (c->loss_host) cudaFreeHost(c->loss_host);
    if (c->own_stream && c->stream) cudaStreamDestroy(c->stream);
    delete c;
}

int lbm_cnn_create(int32_t H, int32_t W, int32_t batch_max, int32_t bf16_activations, uint64_t seed, void *stream,
                   lbm_cnn **out)
{
    if (!out || H < 1 || W < 3 || batch_max < 1) return LBM_EINVAL;
    *out = nullptr;
    lbm_cnn *c = new (std::nothrow) lbm_cnn();
    if (!c) return LBM_ENOMEM;
    c->H = H;
    c->W = W;
    c->Bmax = batch_max;
    c->bf16 = bf16_activations ? 1 : 0;
    if (stream) c->stream = (cudaStream_t)stream;
    else {
        if (cudaStreamCreateWithFlags(&c->stream, cudaStreamNonBlocking) != cudaSuccess) { delete c; return LBM_ECUDA; }
        c->own_stream = true;
    }
    int off = 0;
    for (int l = 0; l < NL; ++l) {
        c->L.off_w[l] = off;
        off += CH[l + 1] * CH[l] * 9;
        c->L.off_b[l] = off;
        off += CH[l + 1];
    }
    c->n_params = c->L.n = off;
    const size_t asz = c->bf16 ? 2 : 4;
    const long long plane = (long long)H * W;
    bool ok = true;
    for (float **f : {&c->p, &c->pf, &c->pb, &c->g, &c->m, &c->v}) ok = ok && cudaMalloc((void **)f, off * sizeof(float)) == cudaSuccess;
    for (int l = 1; l <= NL && ok; ++l) ok = cudaMalloc(&c->z[l], (size_t)batch_max * CH[l] * plane * asz) == cudaSuccess;
    ok = ok && cudaMalloc((void **)&c->act, (size_t)batch_max * 32 * plane * sizeof(float)) == cudaSuccess;
    for (int k = 0; k < 2 && ok; ++k) ok = cudaMalloc((void **)&c->dz[k], (size_t)batch_max * 32 * plane * sizeof(float)) == cudaSuccess;
    int dev = 0;
    ok = ok && cudaGetDevice(&dev) == cudaSuccess &&
         cudaDeviceGetAttribute(&c->sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess;
    const size_t part_floats = (size_t)grad_ctas(c, batch_max) * off;
    ok = ok && cudaMalloc((void **)&c->part, part_floats * sizeof(float)) == cudaSuccess;
    ok = ok && cudaMalloc((void **)&c->loss_part, 512 * sizeof(double)) == cudaSuccess;
    ok = ok && cudaMallocHost((void **)&c->loss_host, 512 * sizeof(double)) == cudaSuccess;
    if (!ok) { cudaGetLastError(); lbm_cnn_destroy(c); return LBM_ENOMEM; }
    // He-style initialisation from a 64-bit LCG (weights ~ U(-a, a), a = sqrt(6 / fan_in)), zero biases
    std::vector<float> h(off, 0.0f);
    uint64_t s = seed * 6364136223846793005ULL + 1442695040888963407ULL;
    for (int l = 0; l < NL; ++l) {
        const float a = sqrtf(6.0f / (CH[l] * 9.0f)) * (l == NL - 1 ? 0.1f : 1.0f);
        for (int i = 0; i < CH[l + 1] * CH[l] * 9; ++i) {
            s = s * 6364136223846793005ULL + 1442695040888963407ULL;
            const double u01 = (double)(s >> 11) / 9007199254740992.0;
            h[c->L.off_w[l] + i] = (float)((2.0 * u01 - 1.0) * a);
        }
    }
    const int rc = lbm_cnn_set_params(c, h.data());   // on the network's stream, like all that reads them
    if (rc != LBM_OK) { lbm_cnn_destroy(c); return rc; }
    *out = c;
    return LBM_OK;
}

int lbm_cnn_num_params(const lbm_cnn *c, int64_t *n)
{
    if (!c || !n) return LBM_EINVAL;
    *n = c->n_params;
    return LBM_OK;
}

int lbm_cnn_get_params(lbm_cnn *c, float *host)
{
    if (!c || !host) return LBM_EINVAL;
    cudaError_t e = cudaMemcpyAsync(host, c->p, c->n_params * sizeof(float), cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    return e == cudaSuccess ? LBM_OK : cnn_fail(e, "lbm_cnn_get_params");
}

int lbm_cnn_set_params(lbm_cnn *c, const float *host)
{
    if (!c || !host) return LBM_EINVAL;
    cudaError_t e = cudaMemcpyAsync(c->p, host, c->n_params * sizeof(float), cudaMemcpyHostToDevice, c->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(c->m, 0, c->n_params * sizeof(float), c->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(c->v, 0, c->n_params * sizeof(float), c->stream);
    if (e == cudaSuccess) e = lay_out_weights(c);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    c->t = 0;
    return e == cudaSuccess ? LBM_OK : cnn_fail(e, "lbm_cnn_set_params");
}

int lbm_cnn_forward(lbm_cnn *c, const float *x, int32_t B, float *y)
{
    if (!c || !x || !y || B < 1 || B > c->Bmax) return LBM_EINVAL;
    const cudaError_t e = c->bf16 ? cnn_forward_impl<__nv_bfloat16>(c, x, B, y) : cnn_forward_impl<float>(c, x, B, y);
    return e == cudaSuccess ? LBM_OK : cnn_fail(e, "lbm_cnn_forward");
}

int lbm_cnn_gradients(lbm_cnn *c, const float *x, const float *target, int32_t B, float *grad_host, double *loss)
{
    if (!c || !x || !target || B < 1 || B > c->Bmax) return LBM_EINVAL;
    cudaError_t e = c->bf16 ? cnn_forward_impl<__nv_bfloat16>(c, x, B, (__nv_bfloat16 *)c->z[NL])
                            : cnn_forward_impl<float>(c, x, B, (float *)c->z[NL]);
    if (e == cudaSuccess)
        e = c->bf16 ? cnn_backward_impl<__nv_bfloat16>(c, x, B, target, loss)
                    : cnn_backward_impl<float>(c, x, B, target, loss);
    if (e == cudaSuccess && grad_host) {
        e = cudaMemcpyAsync(grad_host, c->g, c->n_params * sizeof(float), cudaMemcpyDeviceToHost, c->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    }
    return e == cudaSuccess ? LBM_OK : cnn_fail(e, "lbm_cnn_gradients");
}

int lbm_cnn_train_step(lbm_cnn *c, const float *x, const float *target, int32_t B, float lr, double *loss)
{
    int rc = lbm_cnn_gradients(c, x, target, B, nullptr, loss);
    if (rc) return rc;
    c->t += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.0f - powf(b1, (float)c->t), c2 = 1.0f - powf(b2, (float)c->t);
    adam_step<<<(c->n_params + 255) / 256, 256, 0, c->stream>>>(c->p, c->pf, c->pb, c->g, c->m, c->v, c->L, lr, b1,
                                                                b2, 1e-8f, c1, c2);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? LBM_OK : cnn_fail(e, "lbm_cnn_train_step");
}

const char *lbm_cnn_strerror(void) { return g_cnn_err; }

}  // extern "C"
