// lbm_noalloc.cu -- the field reduction (mass, velocity-change and velocity norms,
// non-finite count) for callers that cannot allocate device memory.
//
// Some callers cannot call cudaMalloc: code that enqueues work while a stream is being
// captured into a CUDA graph, or a plugin / custom call inside a framework that owns every
// device allocation and only hands it buffers.  lbm_reduce_fields_noalloc serves them: the
// caller passes the input fields and the output array, and the per-block partial sums live
// in the fixed array below, which every GPU that loads this library keeps until the
// process exits.  No cudaMalloc, cudaFree or allocating library routine is called.
#include <mutex>

#include "../../include/lbm_gb300.h"
#include "lbm_internal.h"
#include "lbm_reduce.cuh"

namespace {

// Scratch for the block partials: 304 x 4 doubles = 9.5 KiB per device.
static __device__ __align__(256) double g_noalloc_partials[lbm::RED_BLOCKS * 4];

constexpr int MAX_DEVICES = 64;
std::mutex g_setup_mutex;
double *g_partials_ptr[MAX_DEVICES] = {nullptr};

// The handle's reduction (lbm_reduce.cuh), so both give identical sums for identical fields.  Every
// slot of the scratch is written: no zeroing needed.
__global__ void __launch_bounds__(lbm::RED_THREADS)
noalloc_partial_kernel(const double *phi, const double *u, const double *v, const double *T, const double *up,
                       const double *vp, long long N, double *partials)
{
    lbm::reduce_block_(phi, u, v, T, const_cast<double *>(up), const_cast<double *>(vp), N, blockIdx.x, false,
                       partials + 4 * blockIdx.x);
}

__global__ void __launch_bounds__(128) noalloc_final_kernel(const double *partials, double *result)
{
    lbm::reduce_blocks_(partials, result);
}

// Once per device, with that device current: the device address of the scratch array.
int partials_for_current_device(double **out)
{
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return LBM_ECUDA;
    if (dev < 0 || dev >= MAX_DEVICES) return LBM_EINVAL;
    std::lock_guard<std::mutex> lock(g_setup_mutex);
    if (!g_partials_ptr[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_partials);
        if (e != cudaSuccess || !p) return LBM_ECUDA;
        g_partials_ptr[dev] = (double *)p;
    }
    *out = g_partials_ptr[dev];
    return LBM_OK;
}

}  // namespace

extern "C" int lbm_reduce_fields_noalloc(const double *phi, const double *u, const double *v, const double *T,
                                         const double *u_prev, const double *v_prev, int64_t n_nodes,
                                         double *result, void *stream)
{
    if (!phi || !u || !v || !T || !result) return LBM_EINVAL;
    if (n_nodes < 1 || n_nodes > LBM_NOALLOC_MAX_NODES) return LBM_EINVAL;
    if ((u_prev == nullptr) != (v_prev == nullptr)) return LBM_EINVAL;
    double *partials = nullptr;
    int rc = partials_for_current_device(&partials);
    if (rc) return rc;
    cudaStream_t s = (cudaStream_t)stream;
    noalloc_partial_kernel<<<lbm::RED_BLOCKS, lbm::RED_THREADS, 0, s>>>(phi, u, v, T, u_prev, v_prev, (long long)n_nodes, partials);
    if (cudaGetLastError() != cudaSuccess) return LBM_ECUDA;
    noalloc_final_kernel<<<1, 128, 0, s>>>(partials, result);
    if (cudaGetLastError() != cudaSuccess) return LBM_ECUDA;
    return LBM_OK;
}
