// lbm_internal.h -- launchers shared between the kernel and the host translation units.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "lbm_device.cuh"
#include "lbm_pdl.h"

namespace lbm {

// How a step is launched: rows > 0: row-marching strips, each CTA walking that many rows; else
// 2-D tiles of tx x ty nodes (sms: SMs of the device).
struct StepShape {
    int rows, tx, ty, sms;
};

// One time step from A's input buffers to its output buffers.
template <typename Real, typename Store, int QF, int QT>
cudaError_t launch_march(const StepArgs<Real, Store> &A, cudaStream_t s, int rows);
template <typename Real, typename Store, int QF, int QT>
cudaError_t launch_tile(const StepArgs<Real, Store> &A, cudaStream_t s, const StepShape &shape);

// Many cases in one launch.  Up to PACK_CASES of them travel in the launch's parameters: their arguments
// are then uniform values in constant memory, as those of a single channel are (fetched through
// a pointer they cost ~160 instructions a node more and two dependent loads a CTA).  32, the power of
// two that pack_case_ searches: a launch's parameters hold 32,764 bytes, and 32 cases take 27,904 (864 a
// case in FP64).  start[c]: first CTA of case c (INT_MAX beyond the last case), cols[c]: its strips or
// tiles per row.
constexpr int PACK_CASES = 32;
template <typename Real, typename Store> struct BatchPack {
    int start[PACK_CASES], cols[PACK_CASES];
    StepArgs<Real, Store> a[PACK_CASES];
};
// The case of a CTA: the last one that starts at or before it.
template <typename Real, typename Store> __device__ __forceinline__ int pack_case_(const BatchPack<Real, Store> &B, int cta)
{
    int c = 0;
#pragma unroll
    for (int s = PACK_CASES / 2; s > 0; s >>= 1)
        if (cta >= B.start[c + s]) c += s;
    return c;
}
// Larger batches: ctas[i] = (case, strip or tile column, segment or tile row, 0), arguments in device memory.
template <typename Real, typename Store, int QF, int QT>
cudaError_t launch_batch(const StepArgs<Real, Store> *cases, const int4 *ctas, int n_ctas, const int *active, int seg,
                         cudaStream_t s);
template <typename Real, typename Store, int QF, int QT>
cudaError_t launch_tile_batch(const StepArgs<Real, Store> *cases, const int4 *ctas, int n_ctas, const int *active,
                              const StepShape &shape, cudaStream_t s);
template <typename Real, typename Store, int QF, int QT>
cudaError_t launch_march_pack(const BatchPack<Real, Store> &B, int n_ctas, const int *active, int seg, cudaStream_t s);
template <typename Real, typename Store, int QF, int QT>
cudaError_t launch_tile_pack(const BatchPack<Real, Store> &B, int n_ctas, const int *active, const StepShape &shape,
                             cudaStream_t s);
// Columns per strip of the march.
template <typename Real, typename Store, int QF, int QT> int step_strip_width();
// Rows per segment of the march when none is set (choose_segment).
template <typename Real, typename Store, int QF, int QT> int auto_segment(int nx, int ny);
// Tile shape for a channel on a device with `sms` SMs.
template <typename Real, typename Store, int QF, int QT> StepShape choose_tile(int nx, long long ny, int sms);

// Initialisation: macro [5][ny][nx] (phi, u, v, T, dp) holds the fields; entries whose
// bit in `defaults` (1 phi, 2 u, 4 v, 8 T, 16 dp) is set are filled with the defaults
// first.  Then the populations are set to the central-moment equilibria.
template <typename Real, typename Store, int QF, int QT>
cudaError_t launch_init(const StepArgs<Real, Store> &A, double b, double W, int defaults, cudaStream_t s);

// Reductions over the macro fields: partials[reduce_blocks()][4] then result[4] =
// (sum phi, sum |u - u_prev|^2, sum |u|^2, non-finite count); u_prev <- u if update.
cudaError_t launch_reduce(const double *macro, double *uprev, long long N, int update, double *partials, double *result,
                          cudaStream_t s);
// The same (update = 1) for the active ones of n channels, into results[n][4].
struct ReduceCase {
    const double *macro;
    double *uprev, *partials;
    long long N;
};
cudaError_t launch_reduce_batch(const ReduceCase *cases, const int *active, int n, double *results, cudaStream_t s);
int reduce_blocks();

// [Q][ny][nx] doubles <-> [Q][ny][pitch] storage ((value - ref[q][y]) * scale stored; ref
// may be NULL)
template <typename Real, typename Store>
cudaError_t launch_to_store(const double *src, Store *dst, int Q, int nx, int ny, int pitch, Real scale,
                            const double *ref, cudaStream_t s);
template <typename Real, typename Store>
cudaError_t launch_from_store(const Store *src, double *dst, int Q, int nx, int ny, int pitch, Real iscale,
                              const double *ref, cudaStream_t s);
// macro planes -> device arrays of float or double (NULL: not wanted)
cudaError_t launch_export(const double *macro, void *const dst[5], long long N, int to_float, cudaStream_t s);

}  // namespace lbm
