// The CUDA runtime and the kernel launchers as far as the host side of the library
// (fastpc_api.cu) needs them on the CPU: device memory is host memory that holds
// anything, copies are immediate, and the launchers write what the host code looks at
// -- among it the error words that a kernel sets when a bounded wait expires.
#include "internal.h"

#include <cmath>
#include <cstdlib>
#include <cstring>
#include <map>

static std::map<char *, size_t> g_mem;
static char g_dummy[64];
// calls of a product until its wait expires (0: none does)
static int g_fail_exact, g_fail_split;
static int g_split;                                      // split-precision products run
static int g_halted;                                     // searches that an error word halted

extern "C" {
void fake_fail(int exact, int split) { g_fail_exact = exact, g_fail_split = split; }
int fake_split() { return g_split; }
int fake_halted() { return g_halted; }
void fake_device(void *p, long long bytes) { g_mem[(char *)p] = (size_t)bytes; }
int pc_corr_noalloc(void *, int, long long, int, long long, void *, long long, void *) { return 1; }

cudaError_t cudaMalloc(void **p, size_t n)
{
    *p = malloc(n);
    memset(*p, 0x5a, n);
    g_mem[(char *)*p] = n;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p)
{
    g_mem.erase((char *)p);
    free(p);
    return cudaSuccess;
}
cudaError_t cudaMallocHost(void **p, size_t n)
{
    *p = malloc(n);
    memset(*p, 0x5a, n);
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void *p) { return free(p), cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *p)
{
    auto it = g_mem.upper_bound((char *)p);
    const bool dev = it != g_mem.begin() && (--it, (char *)p < it->first + it->second);
    a->type = dev ? cudaMemoryTypeDevice : cudaMemoryTypeUnregistered;
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { return memmove(d, s, n), cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t)
{
    return memmove(d, s, n), cudaSuccess;
}
cudaError_t cudaMemcpy2DAsync(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h, cudaMemcpyKind,
                              cudaStream_t)
{
    for (size_t i = 0; i < h; ++i) memmove((char *)d + i * dp, (const char *)s + i * sp, w);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { return memset(d, v, n), cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { return *s = (cudaStream_t)g_dummy, cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *c)
{
    return *c = cudaStreamCaptureStatusNone, cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { return *e = (cudaEvent_t)g_dummy, cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return *e = (cudaEvent_t)g_dummy, cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { return *ms = 0.f, cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { return *d = 0, cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { return *v = 1, cudaSuccess; }
}

namespace fpc {

int mlp_nparam() { return 18817; }
size_t mlp_pack_bytes() { return 64; }
size_t node_loop_xch_bytes(int) { return 64; }
size_t col_stats_ws_bytes(long long, int) { return 64; }
size_t corr_bf16x3_ws_bytes(long long, int) { return 64; }
bool tc_gemm_available() { return true; }
bool ci_list_uses_fp32(int l, const TestParams &tp) { return tp.precision != 0 && l <= 2; }

cudaError_t launch_col_stats(const void *, int, long long, int, long long, double *, double *, double *, long long,
                             int *err, double *ws, cudaStream_t)
{
    err[0] = 0;
    if (ws) err[1] = 0;
    return cudaSuccess;
}
cudaError_t launch_gram_exact(const void *, int, long long, int p, long long, const double *, const double *, double *C,
                              long long ldc, float *C32, int ldc32, int *err, cudaStream_t)
{
    if (g_fail_exact && --g_fail_exact == 0) *err = 7;
    for (int a = 0; a < p; ++a)
        for (int b = 0; b < p; ++b) {
            C[a * ldc + b] = a == b ? 1.0 : *err ? NAN : 0.25;
            if (C32) C32[(size_t)a * ldc32 + b] = (float)C[a * ldc + b];
        }
    return cudaSuccess;
}
cudaError_t launch_col_stats_split(const void *, int, long long, int, long long, double *, double *, double *,
                                   cudaStream_t)
{
    return cudaSuccess;
}
cudaError_t launch_standardize(const void *, int, long long, int, long long, const double *, const double *,
                               const double *, double *, float *, uint16_t *, uint16_t *, long long, cudaStream_t)
{
    return cudaSuccess;
}
cudaError_t launch_corr_bf16x3(const uint16_t *, const uint16_t *, long long, long long, int p, float *C32, int ldc,
                               float *, size_t, int *err, cudaStream_t)
{
    ++g_split;
    if (g_fail_split && --g_fail_split == 0) *err = 7;
    for (int a = 0; a < p; ++a)
        for (int b = 0; b < p; ++b) C32[(size_t)a * ldc + b] = a == b ? 1.f : 0.5f;
    return cudaSuccess;
}
cudaError_t launch_c64_lazy_init(double *, int, unsigned char *, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_c64_lazy_init_block(double *, int, unsigned char *, int, int, int, cudaStream_t)
{
    return cudaSuccess;
}
size_t syrk_f64_ws_bytes(long long, int) { return 64; }
cudaError_t launch_syrk_f64(const double *, long long, long long, int p, double *C, int ldc, double *, size_t,
                            cudaStream_t)
{
    for (int a = 0; a < p; ++a)
        for (int b = 0; b < p; ++b) C[(size_t)a * ldc + b] = a == b ? 1.0 : 0.25;
    return cudaSuccess;
}

// what precedes the first stage
cudaError_t launch_init_adj(GraphDev, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_level_degrees(GraphDev, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_tail(GraphDev g, TestParams, int, int, const int *, int, cudaGraphConditionalHandle, int, StageConds,
                        const int *err, int nerr, cudaStream_t)
{
    for (int i = 0; i < nerr; ++i)
        if (err[i] && !g.info->halt) {
            g.info->error = err[i];
            g.info->halt = 1;
            ++g_halted;
        }
    return cudaSuccess;
}

// a search that ends at once, and the skeleton's expansion
cudaError_t launch_node_loop(GraphDev g, TestParams, const float *, const double *, int, double *, unsigned long long *,
                             double, int, int, cudaStream_t)
{
    g.info->done = 1;
    return cudaSuccess;
}
// the first raw test's r: what the correlation it reads says
cudaError_t launch_ci_list(const int *, const int *, int, long long, const float *C32, const double *C64, int, int,
                           TestParams tp, double *r, uint8_t *, float *, DevCounters *, const int *, const int *,
                           cudaStream_t)
{
    if (r) r[0] = tp.precision == 0 ? C64[1] : C32[1];
    return cudaSuccess;
}
cudaError_t launch_mlp_features(const int *, long long, const float *, int, const long long *, int, long long,
                                const long long *, double, float *, int *, cudaStream_t)
{
    return cudaSuccess;
}
cudaError_t launch_expand_adj(GraphDev g, uint8_t *out, const LevelInfo *gate, const int *err, int nerr, cudaStream_t)
{
    bool bad = gate && (!gate->done || gate->error || gate->pool_overflow || g.ctr->status);
    for (int i = 0; gate && i < nerr; ++i) bad |= err[i] != 0;
    if (!bad) memset(out, 1, (size_t)g.p * g.p);
    return cudaSuccess;
}

}  // namespace fpc
