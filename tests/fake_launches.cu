// The C ABI's host code on fakes: the runtime calls work on host memory, the launchers play the kernels' part in the
// hand-over words and fail where they are told to.  Linked without the CUDA runtime, so it runs where no GPU is.
#include <math.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <mutex>

#include "../paper_2604_25925_b200/csrc/sgbv_common.cuh"

using namespace sgbv;

namespace {
int g_fail_finish, g_capturing, g_fail_memset, g_stale, g_streamed;
const unsigned long long kUnpublished = ~0ull;
unsigned long long *word(const Launch &L) { return reinterpret_cast<unsigned long long *>(L.ws.ratio); }
}  // namespace

extern "C" {
void fake_set(int fail_finish, int capturing, int fail_memset) {
    g_fail_finish = fail_finish;
    g_capturing = capturing;
    g_fail_memset = fail_memset;
}
int fake_stale(void) { return g_stale; }        // words that the last streaming launch found published before it ran
int fake_streamed(void) { return g_streamed; }  // streaming launches so far

}

namespace {
cudaError_t fake_cudaGetDevice(int *dev) { return *dev = 0, cudaSuccess; }
cudaError_t fake_cudaDeviceSynchronize(void) { return cudaSuccess; }
cudaError_t fake_cudaGetLastError(void) { return cudaSuccess; }
cudaError_t fake_cudaMalloc(void **p, size_t n) { return posix_memalign(p, 256, n) ? cudaErrorMemoryAllocation : cudaSuccess; }
cudaError_t fake_cudaFree(void *p) { return free(p), cudaSuccess; }
cudaError_t fake_cudaMemset(void *p, int v, size_t n) { return memset(p, v, n), cudaSuccess; }
cudaError_t fake_cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t) {
    if (g_fail_memset) return cudaErrorUnknown;
    if (!g_capturing) memset(p, v, n);
    return cudaSuccess;
}
cudaError_t fake_cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) { return memcpy(d, s, n), cudaSuccess; }
cudaError_t fake_cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t fake_cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *st) {
    return *st = g_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone, cudaSuccess;
}
cudaError_t fake_cudaGetSymbolAddress(void **, const void *) { return cudaErrorUnknown; }
cudaError_t fake_cudaEventCreate(cudaEvent_t *) { return cudaErrorUnknown; }
cudaError_t fake_cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t fake_cudaEventSynchronize(cudaEvent_t) { return cudaErrorUnknown; }
cudaError_t fake_cudaEventElapsedTime(float *, cudaEvent_t, cudaEvent_t) { return cudaErrorUnknown; }
}  // namespace

#define cudaGetDevice fake_cudaGetDevice
#define cudaDeviceSynchronize fake_cudaDeviceSynchronize
#define cudaGetLastError fake_cudaGetLastError
#define cudaMalloc fake_cudaMalloc
#define cudaFree fake_cudaFree
#define cudaMemset fake_cudaMemset
#define cudaMemsetAsync fake_cudaMemsetAsync
#define cudaMemcpyAsync fake_cudaMemcpyAsync
#define cudaStreamSynchronize fake_cudaStreamSynchronize
#define cudaStreamIsCapturing fake_cudaStreamIsCapturing
#define cudaGetSymbolAddress fake_cudaGetSymbolAddress
#define cudaEventCreate fake_cudaEventCreate
#define cudaEventDestroy fake_cudaEventDestroy
#define cudaEventSynchronize fake_cudaEventSynchronize
#define cudaEventElapsedTime fake_cudaEventElapsedTime
#include "../paper_2604_25925_b200/csrc/sgbv_api.cu"

// what the compiler registers the library's device array with
extern "C" {
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
char __cudaInitModule(void **) { return 0; }
}

namespace sgbv {
bool fused_supported(const Launch &) { return true; }
bool fused_outrun(const Launch &) { return false; }
void fused_set_options(int, int, int, int, int, int) {}
// As many words as batch rows; cleared first where nobody vouches for them, as the real launcher does.
int launch_fused(const Launch &L, int *, int *words_used, bool *aux_apart) {
    *words_used = L.s.B;
    *aux_apart = false;
    const size_t bytes = (size_t)L.s.B * sizeof(double);
    if (!L.ratio_preset && cudaMemsetAsync(L.ws.ratio, 0xff, bytes, L.stream) != cudaSuccess) return SGBV_ERR_CUDA;
    if (g_capturing) return 1;
    ++g_streamed;
    g_stale = 0;
    for (int n = 0; n < L.s.B; ++n) {
        if (word(L)[n] != kUnpublished) ++g_stale;
        word(L)[n] = 0x3ff0000000000000ull;  // 1.0
    }
    return 1;
}
int launch_finish(const Launch &L) {
    if (g_fail_finish) return SGBV_ERR_CUDA;
    if (g_capturing) return 1;
    for (int n = 0; n < L.ws.ratio_used; ++n) word(L)[n] = kUnpublished;
    return 1;
}
int launch_twopass(const Launch &) { return SGBV_ERR_CUDA; }
int launch_auxreduce(const Launch &) { return SGBV_ERR_CUDA; }
int launch_modify_finish(const Launch &, const float *, int32_t *, double *, double *, double *, int32_t *) { return SGBV_ERR_CUDA; }
int launch_kseq(const Launch &, float *, double *, double *, int32_t *) { return SGBV_ERR_CUDA; }
int launch_draw_rows(const void *, int, const float *, const Shape &, float *, int32_t *, double *, int32_t *, cudaStream_t) {
    return SGBV_ERR_CUDA;
}
}  // namespace sgbv
