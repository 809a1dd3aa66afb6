// corr_noalloc.cu -- pc_corr_noalloc: the correlation step without any device
// allocation, for callers that cannot call cudaMalloc: applications whose
// device memory is reserved up front by their own pool or budget, and
// latency-critical loops in which a cudaMalloc would synchronise the device.
//
// Its only scratch -- the FP64 column means and reciprocal standard deviations,
// and an error word -- lives in a file-scope __device__ array of fixed size.  Every GPU that
// loads the library holds that array (64 KiB) until the process exits.
#include "internal.h"
#include "../../include/fastpc.h"

#include <mutex>

namespace fpc {

constexpr int NOALLOC_MAXP = 4096;

// [0, NOALLOC_MAXP): column means; [NOALLOC_MAXP, 2*NOALLOC_MAXP): 1/sd.
// Behind them one word for the error flag of the product's bounded waits.
static __device__ __align__(256) double g_noalloc_stats[2 * NOALLOC_MAXP + 1];

// Device address of g_noalloc_stats per device (host code cannot use the
// symbol itself: on the host it names a stand-in, not device memory).
static std::mutex g_noalloc_mu;
static double *g_noalloc_ptr[64] = {nullptr};

static cudaError_t noalloc_scratch(double **out)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_stats);   // with device `dev` current
        if (e != cudaSuccess) return e;
        g_noalloc_ptr[dev] = (double *)p;
    }
    *out = g_noalloc_ptr[dev];
    return cudaSuccess;
}

// True when p is device (or managed) memory of device `dev`, the device the
// kernels will run on: a buffer of another GPU is rejected before any launch.
static bool on_device(const void *p, int dev)
{
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return (a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged) && a.device == dev;
}

}  // namespace fpc

extern "C" pc_status pc_corr_noalloc(const void *X, int32_t dtype, int64_t n, int32_t p, int64_t ld,
                                     double *C_out, int64_t ldc, void *stream)
{
    using namespace fpc;
    if (!X || !C_out || (dtype != PC_F32 && dtype != PC_F64)) return PC_ERR_ARG;
    if (n < 2 || n > (1ll << 31) || p < 1 || p > NOALLOC_MAXP || ld < p || ldc < p) return PC_ERR_ARG;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return PC_ERR_ARG;                  // no usable device: nothing can be on it
    }
    if (!on_device(X, dev) || !on_device(C_out, dev)) return PC_ERR_ARG;
    double *stats = nullptr;
    if (noalloc_scratch(&stats) != cudaSuccess) return PC_ERR_CUDA;
    int *err = (int *)(stats + 2 * NOALLOC_MAXP);
    cudaStream_t s = (cudaStream_t)stream;
    // column statistics into the file-scope scratch (every call overwrites
    // entries 0..p-1 of both halves; nothing accumulates across calls)
    if (launch_col_stats(X, dtype, n, p, ld, stats, stats + NOALLOC_MAXP, C_out, ldc, err, nullptr, s) != cudaSuccess)
        return PC_ERR_CUDA;
    // FP64 correlations by exact integer products on the tensor cores, accumulated in C_out
    // itself (gram_exact.cu): no workspace
    return launch_gram_exact(X, dtype, n, p, ld, stats, stats + NOALLOC_MAXP, C_out, ldc, nullptr, 0, err, s) ==
                   cudaSuccess
               ? PC_OK
               : PC_ERR_CUDA;
}
