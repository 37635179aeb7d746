// lbm_tile.cu -- the step on 2-D tiles: one node per thread, all rows of a tile at once.
//
// The row-marching kernel (lbm_step.cu) walks a strip row by row, so a channel with few strips
// pays its ~1.5 us per row in series on a few SMs: 22 us a step at 128 x 32 (4 CTAs; 3.2 here), 21 us
// at 1024 x 256 (256 CTAs of 8 + 6 rows; 8.8 here).  Here every node has its thread; the two rows and columns
// around a tile are pulled again by its CTA (phi; sigma and p on the inner ring), the normals of
// the inner ring are formed again, and the step is one latency: load, barrier, normals,
// barrier, collide, store.  Bound in FP32 arithmetic by instruction issue and the latency
// of the loads and of the two barriers, in FP64 by the FP64 pipe.  The arithmetic of a node is that of
// lbm_node.cuh, so the results are the march's bit for bit.
#include "lbm_internal.h"
#include "lbm_node.cuh"
#include "lbm_once.h"

namespace lbm {

// FP32 arithmetic: tiles of 32 x 8 with compile-time strides; FP64: any shape of up to 256 nodes,
// chosen for the channel (choose_tile).
template <typename Real, typename Store, int QF = 5, int QT = 5> struct TileGeo {
    static constexpr bool FIXED = sizeof(Real) == 4;
    static constexpr int NT = 256, TX = 32;
    // FP32: four CTAs per SM (64 registers; three: 9.8 us instead of 8.8 at 1024 x 256, five: 9.1, and 14.3
    // instead of 11.8 with three D2Q9 lattices).  FP16, latency bound on its smaller loads: five (48
    // registers; 220 us at 8192 x 1024, 237 with four).  With one D2Q9 scalar lattice 16 to 28 bytes spill at
    // 48 and five still win on large channels (271 us, 288 with four) and lose on small ones (1024 x
    // 256: 13.1, 10.8); with two, four win (309 us, 329 with five).  The batch kernels take the same
    // numbers; that of more than PACK_CASES channels spills up to 100 bytes (FP16), 20 (FP32).
    // FP64 takes the registers it needs.
    static constexpr int CTAS = sizeof(Real) == 8 ? 1 : (sizeof(Store) == 2 && QF + QT < 18 ? 5 : 4);
};

template <typename Real, typename Store, int QF, int QT>
__device__ __forceinline__ void tile_body(const StepArgs<Real, Store> &A, int tx_, int ty_, int bx, int by,
                                          unsigned char *smem)
{
    using R2 = typename Vec2<Real>::T;
    using G = TileGeo<Real, Store>;
    const int NT = G::FIXED ? G::NT : blockDim.x;
    const int tx = G::FIXED ? G::TX : tx_, ty = G::FIXED ? G::NT / G::TX : ty_;
    const int PX = tx + 4, SX = tx + 2;
    R2 *s_sp = reinterpret_cast<R2 *>(smem);           // [ty + 2][SX]: (sigma - sigma0, p - p0)
    R2 *s_n = s_sp + (ty + 2) * SX;                    // [ty + 2][SX]: unit normal (n_x, n_y - 1)
    Real *s_phi = reinterpret_cast<Real *>(s_n + (ty + 2) * SX);   // [ty + 4][PX]: phi - phi0
    const int nx = A.nx, ny = A.ny, pitch = A.pitch, t = threadIdx.x;
    const int x0 = bx * tx, y0 = by * ty;
    const int ex = min(tx, nx - x0), ey = min(ty, ny - y0);
    const int ly = t / tx, lx = t - ly * tx;
    const bool own = lx < ex && ly < ey;
    const int x = x0 + lx, y = y0 + ly;
    const Real *t_dR = A.rtab + (ny + 2) * RT_DR + 1, *t_dRlo = A.rtab + (ny + 2) * RT_DRLO + 1;
    const Real *t_gref = A.rtab + (ny + 2) * RT_GREF + 1;

    Real fm[2], hm[3], g[9], dphi;
    auto load = [&](auto walls) {
        constexpr bool WALLS = decltype(walls)::value;
        Real f[QF], h[QT], dp = Real(0);
        if (own) {
            const int xm = x == 0 ? nx - 1 : x - 1, xp = x == nx - 1 ? 0 : x + 1;
            pull_row_<0, QF, WALLS>(A.fi, pitch, ny, nx, y, x, xm, xp, A.sf, A.twall, A.P.dTcold, f);
            pull_row_<2, QT, WALLS>(A.hi, pitch, ny, nx, y, x, xm, xp, A.sh, A.twall, A.P.dTcold, h);
            dp = A.dp_in[y * pitch + x];
            pull_row_<1, 9, WALLS>(A.gi, pitch, ny, nx, y, x, xm, xp, A.sg, A.twall, A.P.dTcold, g);
        }
        // the two halo rows and columns around the tile: phi, and sigma and p on the inner ring
        auto halo = [&](int hx, int hy) {
            int X = x0 + hx;
            X = X < 0 ? X + nx : (X >= nx ? X - nx : X);
            const int xm = X == 0 ? nx - 1 : X - 1, xp = X == nx - 1 ? 0 : X + 1;
            const int r = y0 + hy, gy = WALLS ? mirror_row_(r, ny) : r;
            Real q[QF];
            pull_row_<0, QF, WALLS>(A.fi, pitch, ny, nx, gy, X, xm, xp, A.sf, A.twall, A.P.dTcold, q);
            if (hx >= -1 && hx <= ex && hy >= -1 && hy <= ey) {
                Real v[QT];
                pull_row_<2, QT, WALLS>(A.hi, pitch, ny, nx, gy, X, xm, xp, A.sh, A.twall, A.P.dTcold, v);
                const Real pv = A.dp_in[gy * pitch + X];
                s_sp[(hy + 1) * SX + hx + 1] = sig_p_(A, r, X, temp_dev_<QT>(A, v), pv);
            }
            s_phi[(hy + 2) * PX + hx + 2] = phi_dev_<QF>(A, q, t_dR[gy], t_dRlo[gy]);
        };
        if constexpr (G::FIXED) {
            // a warp per halo row (the columns of the tile), then the side columns, four a row:
            // no division (by the ragged width) on the way to the loads
            static_assert(G::TX == 32 && 4 * 32 + 4 * (G::NT / 32 + 4) <= G::NT, "one halo node per thread");
            if (t < 4 * 32) {
                const int r = t >> 5, hx = t & 31;
                if (hx < ex) halo(hx, r < 2 ? r - 2 : ey + r - 2);
            } else if (t < 4 * 32 + 4 * (ey + 4)) {
                const int j = t - 4 * 32, k = j & 3;
                halo(k < 2 ? k - 2 : ex + k - 2, (j >> 2) - 2);
            }
        } else {
            const int nr = 4 * (ex + 4 + ey);
            for (int i = t; i < nr; i += NT) {
                if (i < 4 * (ex + 4)) {
                    const int r = i / (ex + 4);
                    halo(i - r * (ex + 4) - 2, r < 2 ? r - 2 : ey + r - 2);
                } else {
                    const int j = i - 4 * (ex + 4), k = j & 3;
                    halo(k < 2 ? k - 2 : ex + k - 2, j >> 2);
                }
            }
        }
        if (own) {
            dphi = phi_dev_<QF>(A, f, t_dR[y], t_dRlo[y]);
            s_phi[(ly + 2) * PX + lx + 2] = dphi;
            keep_f_<QF>(A, f, fm);
            const Real dT = temp_dev_<QT>(A, h);
            s_sp[(ly + 1) * SX + lx + 1] = sig_p_(A, y, x, dT, dp);
            keep_h_<QT>(A, h, dT, hm);
        }
    };
    // rows y0 - 2 .. y0 + ey + 1 are pulled into
    if (y0 >= 3 && y0 + ey + 2 < ny) load(std::false_type());
    else load(std::true_type());
    __syncthreads();
    auto put_n = [&](int hx, int hy, Real &gx, Real &gy) {
        const Real *r = s_phi + (hy + 2) * PX;
        grad_ref_(r - PX, r, r + PX, hx + 2, t_gref[y0 + hy], gx, gy);
        s_n[(hy + 1) * SX + hx + 1] = normal_(gx, gy, A.P.g2min);
    };
    Real gpx, gpy;   // grad phi of the thread's own node
    if (own) put_n(lx, ly, gpx, gpy);
    {
        Real gx, gy;
        if constexpr (G::FIXED) {   // the last warps: the rows below and above, then the sides
            const int i = NT - 1 - t;
            if (i < 2 * 32) {
                if ((i & 31) < ex) put_n(i & 31, i < 32 ? -1 : ey, gx, gy);
            } else if (i < 2 * 32 + 2 * (ey + 2)) {
                put_n((i & 1) ? -1 : ex, ((i - 2 * 32) >> 1) - 1, gx, gy);
            }
        } else {
            for (int i = NT - 1 - t; i < 2 * (ex + 2 + ey); i += NT) {
                if (i < 2 * (ex + 2)) put_n(i < ex + 2 ? i - 1 : i - (ex + 2) - 1, i < ex + 2 ? -1 : ey, gx, gy);
                else put_n((i & 1) ? -1 : ex, (i - 2 * (ex + 2)) >> 1, gx, gy);
            }
        }
    }
    Real rx[RX_N];   // the row's reference values (on their way across the barrier)
    if (own) load_rowref_(A.rowx + (long long)y * RX_N, rx);
    __syncthreads();
    if (own) {
        const R2 *n = s_n + (ly + 1) * SX, *q = s_sp + (ly + 1) * SX;
        node_step_<Real, Store, QF, QT>(A, x, y, dphi, gpx, gpy, lx + 1, n - SX, n, n + SX, q - SX, q, q + SX, fm, hm,
                                        g, rx[RX_PHI0], rx[RX_TH0], rx[RX_C01], rx[RX_P1]);
    }
}

// Launched with programmatic stream serialisation: the CTAs of the next step's launch may start
// while this one drains; each waits (griddepcontrol.wait) for the complete end of the launch
// before it, so all memory of earlier steps is visible and every launch ends after its
// predecessor.  Saves 2.5 us of 6 us a step at 128 x 32.  FP64 lets the next launch start only at its
// own end: its CTAs would otherwise settle beside running ones and leave other SMs empty (200 x 100,
// tiles of 128: 62 us a step instead of 47; see also tile_smem).
template <typename Real> __device__ __forceinline__ void let_next_start_early_()
{
    if (sizeof(Real) == 4) pdl_launch_next_();
}
template <typename Real> __device__ __forceinline__ void let_next_start_late_()
{
    if (sizeof(Real) == 8) pdl_launch_next_();
}

template <typename Real, typename Store, int QF, int QT>
__global__ void __launch_bounds__(TileGeo<Real, Store>::NT, TileGeo<Real, Store, QF, QT>::CTAS)
tile_kernel(const __grid_constant__ StepArgs<Real, Store> A, int tx, int ty)
{
    extern __shared__ __align__(16) unsigned char smem[];
    let_next_start_early_<Real>();
    pdl_wait_();
    tile_body<Real, Store, QF, QT>(A, tx, ty, blockIdx.x, blockIdx.y, smem);
    let_next_start_late_<Real>();
}

// Many channels in one launch: CTA i works on tile (ctas[i].y, ctas[i].z) of case ctas[i].x, whose
// arguments it copies to shared memory (before the wait: they are constant).
template <typename Real, typename Store, int QF, int QT>
__global__ void __launch_bounds__(TileGeo<Real, Store>::NT, TileGeo<Real, Store, QF, QT>::CTAS)
tile_batch_kernel(const StepArgs<Real, Store> *__restrict__ cases, const int4 *__restrict__ ctas,
                  const int *__restrict__ active, int tx, int ty)
{
    using Args = StepArgs<Real, Store>;
    extern __shared__ __align__(16) unsigned char smem[];
    static_assert(sizeof(Args) % 16 == 0, "copied in 16-byte words");
    __shared__ __align__(16) unsigned char s_args[sizeof(Args)];
    let_next_start_early_<Real>();
    const int4 c = ctas[blockIdx.x];
    for (int i = threadIdx.x; i < (int)(sizeof(Args) / 16); i += blockDim.x)
        reinterpret_cast<uint4 *>(s_args)[i] = reinterpret_cast<const uint4 *>(cases + c.x)[i];
    pdl_wait_();
    __syncthreads();
    if (active[c.x])
        tile_body<Real, Store, QF, QT>(*reinterpret_cast<const Args *>(s_args), tx, ty, c.y, c.z, smem);
    let_next_start_late_<Real>();
}

// The same with up to PACK_CASES channels' arguments in the launch's parameters.
template <typename Real, typename Store, int QF, int QT>
__global__ void __launch_bounds__(TileGeo<Real, Store>::NT, TileGeo<Real, Store, QF, QT>::CTAS)
tile_pack_kernel(const __grid_constant__ BatchPack<Real, Store> B, const int *active, int tx, int ty)
{
    extern __shared__ __align__(16) unsigned char smem[];
    let_next_start_early_<Real>();
    const int c = pack_case_(B, blockIdx.x);
    const int on = active[c];   // (host copies set it between launches that follow one another)
    const int i = blockIdx.x - B.start[c], by = i / B.cols[c], bx = i - by * B.cols[c];
    pdl_wait_();
    if (on) tile_body<Real, Store, QF, QT>(B.a[c], tx, ty, bx, by, smem);
    let_next_start_late_<Real>();
}

// Dynamic shared memory of a launch of `tiles` tiles.  In FP64 a step takes as long as the SM with the
// most tiles, so no SM may take more than its share: the request is raised until only that many
// CTAs fit (otherwise CTAs settle two to an SM while the launch before still holds others: 33 us
// instead of 24 a step at 200 x 100 with 130 tiles on 152 SMs).
constexpr int SM_SMEM_KIB = 228;                          // 1 KiB of it reserved per CTA
constexpr size_t TILE_SMEM_MAX = SM_SMEM_KIB / 2 * 1024;   // the largest request: one tile per SM
template <typename Real> static size_t tile_smem(int tx, int ty, long long tiles, int sms)
{
    const size_t need = ((size_t)(ty + 4) * (tx + 4) + 4 * (size_t)(ty + 2) * (tx + 2)) * sizeof(Real);
    const long long share = (tiles + sms - 1) / sms;   // CTAs an SM has to take
    if (sizeof(Real) == 4 || share > 4) return need;
    const size_t most = (size_t)(SM_SMEM_KIB / (share + 1)) * 1024;   // share + 1 CTAs of more than this do not fit
    return need > most ? need : most;
}

// A launch of one of the tile kernels.  FP64 requests may exceed the 48 KiB that a kernel may ask for
// untold: the limit goes to their maximum once per kernel and device, not to each launch's own
// request (with two threads stepping channels of different size, one lowered it between the
// other's setting and launch).
template <auto kernel, typename Real, typename... Args>
static cudaError_t launch_tiles(dim3 grid, const StepShape &shape, cudaStream_t s, Args... args)
{
    const int tx = shape.tx, ty = shape.ty;
    PdlLaunch l(grid, dim3((tx * ty + 31) / 32 * 32), tile_smem<Real>(tx, ty, (long long)grid.x * grid.y, shape.sms), s);
    if constexpr (sizeof(Real) == 8) {
        static OncePerDevice limit;
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess)
            e = (cudaError_t)limit.run(dev, [] {
                return (int)cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TILE_SMEM_MAX);
            });
        if (e != cudaSuccess) return e;
    }
    return cudaLaunchKernelEx(&l.cfg, kernel, args..., tx, ty);
}

template <typename Real, typename Store, int QF, int QT>
cudaError_t launch_tile(const StepArgs<Real, Store> &A, cudaStream_t s, const StepShape &shape)
{
    const dim3 grid((A.nx + shape.tx - 1) / shape.tx, (A.ny + shape.ty - 1) / shape.ty);
    return launch_tiles<tile_kernel<Real, Store, QF, QT>, Real, const StepArgs<Real, Store> &>(grid, shape, s, A);
}

template <typename Real, typename Store, int QF, int QT>
cudaError_t launch_tile_batch(const StepArgs<Real, Store> *cases, const int4 *ctas, int n_ctas, const int *active,
                              const StepShape &shape, cudaStream_t s)
{
    return launch_tiles<tile_batch_kernel<Real, Store, QF, QT>, Real>(dim3(n_ctas), shape, s, cases, ctas, active);
}

template <typename Real, typename Store, int QF, int QT>
cudaError_t launch_tile_pack(const BatchPack<Real, Store> &B, int n_ctas, const int *active, const StepShape &shape,
                             cudaStream_t s)
{
    return launch_tiles<tile_pack_kernel<Real, Store, QF, QT>, Real, const BatchPack<Real, Store> &>(dim3(n_ctas), shape, s,
                                                                                                B, active);
}

// Tile shape.  FP32 arithmetic: 32 x 8.  FP64 is bound by the SM's one FP64 pipe (16 cycles a warp
// instruction), so what counts is the FP64 instructions of the SM with the most tiles: warps of
// nodes, the inner ring's normals, the outer ring's phi, and a start-up of ~150 (the shapes this
// ranks first are within 3 % of the best measured at 200 x 100, 160 x 320 and 1024 x 256).
template <typename Real, typename Store, int QF, int QT> StepShape choose_tile(int nx, long long ny, int sms)
{
    using G = TileGeo<Real, Store>;
    StepShape best_shape = {0, G::TX, G::NT / G::TX, sms};
    if (G::FIXED) return best_shape;
    const double node = 260.0 + 14.0 * (QF + QT - 10), normal = 36.0, pull = 13.0, start = 150.0;
    auto warps = [](int n) { return double((n + 31) / 32); };
    double best = -1.0;
    for (int w = nx < 64 ? nx : 64; w >= 8 || w == nx; --w)
        for (int h = 2; h <= 32 && w * h <= G::NT; ++h) {
            const long long tiles = (nx + w - 1) / w * ((ny + h - 1) / h);
            const double cost = double((tiles + sms - 1) / sms) *
                                (warps(w * h) * node + warps(2 * (w + 2 + h)) * normal + warps(4 * (w + 4 + h)) * pull + start);
            if (best < 0.0 || cost < best) best = cost, best_shape.tx = w, best_shape.ty = h;
        }
    return best_shape;
}

#define LBM_INST(R, S, QF, QT)                                                                                    \
    template cudaError_t launch_tile<R, S, QF, QT>(const StepArgs<R, S> &, cudaStream_t, const StepShape &);       \
    template cudaError_t launch_tile_batch<R, S, QF, QT>(const StepArgs<R, S> *, const int4 *, int, const int *,    \
                                                         const StepShape &, cudaStream_t);                        \
    template cudaError_t launch_tile_pack<R, S, QF, QT>(const BatchPack<R, S> &, int, const int *,                 \
                                                        const StepShape &, cudaStream_t);                         \
    template StepShape choose_tile<R, S, QF, QT>(int, long long, int);
LBM_INST(double, double, 5, 5)
LBM_INST(double, double, 5, 9)
LBM_INST(double, double, 9, 5)
LBM_INST(double, double, 9, 9)
LBM_INST(float, float, 5, 5)
LBM_INST(float, float, 5, 9)
LBM_INST(float, float, 9, 5)
LBM_INST(float, float, 9, 9)
LBM_INST(float, __half, 5, 5)
LBM_INST(float, __half, 5, 9)
LBM_INST(float, __half, 9, 5)
LBM_INST(float, __half, 9, 9)
#undef LBM_INST

}  // namespace lbm
