// A CUDA runtime without a device, for tests of the library's host side: device memory is host memory, copies are memcpy, and a
// launch only leaves a record.  Linked with the library's own host code (and the one-token kernels' launchers) in place of
// cudart and of the other kernels' launchers; tests plant failures, captures and expired waits here.
#include <cstdlib>
#include <cstring>
#include <new>

#include "../paper_2510_18546_b200/csrc/enl_internal.h"

namespace {

struct Record { char kind; int wait_first; size_t bytes; int halves; };   // launch ('w' plan write, 's' store, 'a' attention ...)
Record g_log[4096];
int g_n_log;
int g_heap;                      // allocations of the library's code since the last look
int g_fail_kind;                 // launches of this kind are refused ('e': tensor maps)
int g_wait_expires;              // the next one-token kernel gives up on a wait
unsigned long long g_capture;    // the stream is being captured (as this graph)
bool g_captured_event;           // the last record of any event was captured

cudaError_t note(char kind, int wait_first, size_t bytes = 0, int halves = 0)
{
    if (g_fail_kind == kind) return cudaErrorInvalidValue;
    if (g_n_log < 4096) g_log[g_n_log++] = Record{kind, wait_first, bytes, halves};
    return cudaSuccess;
}
CUresult encode(CUtensorMap *tm, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill)
{
    if (g_fail_kind == 'e') return CUDA_ERROR_INVALID_VALUE;
    std::memset(tm, 0, sizeof *tm);
    return CUDA_SUCCESS;
}

}  // namespace

// ---- heap of the code under test (the library is linked so that its allocations end here) --------------------------------
void *operator new(size_t n) { ++g_heap; return std::malloc(n); }
void operator delete(void *p) noexcept { std::free(p); }
void operator delete(void *p, size_t) noexcept { std::free(p); }

// ---- what tests call ------------------------------------------------------------------------------------------------------
extern "C" {
int fake_heap() { const int n = g_heap; g_heap = 0; return n; }
void fake_fail(int kind) { g_fail_kind = kind; }
void fake_expire(int on) { g_wait_expires = on; }
void fake_capture(unsigned long long id) { g_capture = id; }
void fake_clear() { g_n_log = 0; }
int fake_launches() { return g_n_log; }
int fake_kind(int i) { return g_log[i].kind; }
int fake_wait_first(int i) { return g_log[i].wait_first; }
int fake_halves(int i) { return g_log[i].halves; }
long long fake_bytes(int i) { return static_cast<long long>(g_log[i].bytes); }

// ---- CUDA runtime ---------------------------------------------------------------------------------------------------------
void **__cudaRegisterFatBinary(void *) { static void *handle; return &handle; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, cudaStream_t) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *, dim3 *, size_t *, void *) { return cudaSuccess; }
cudaError_t cudaLaunchKernel(const void *, dim3, dim3, void **, size_t, cudaStream_t) { return note('k', 0); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *, const void *, void **args)
{
    // only the one-token kernels are linked; their parameters begin with a ClusterDecodeParams
    const auto *p = static_cast<const enl::ClusterDecodeParams *>(args[0]);
    const cudaError_t e = note('c', p->wait_first);
    if (e == cudaSuccess && g_wait_expires) *p->status = 2;
    return e;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int *n) { *n = 1; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 148; return cudaSuccess; }
cudaError_t cudaDeviceGetStreamPriorityRange(int *lo, int *hi) { *lo = *hi = 0; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaMalloc(void **p, size_t n) { *p = std::aligned_alloc(256, (n + 255) / 256 * 256); return cudaSuccess; }
cudaError_t cudaFree(void *p) { std::free(p); return cudaSuccess; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return cudaMalloc(p, n); }
cudaError_t cudaFreeHost(void *p) { return cudaFree(p); }
cudaError_t cudaMemset(void *p, int v, size_t n) { std::memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t)
{
    const cudaError_t e = note('p', 0, n);
    if (e == cudaSuccess && !g_capture) std::memcpy(d, s, n);
    return e;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { g_captured_event = g_capture != 0; return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { return g_captured_event ? cudaErrorCapturedEvent : cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return g_captured_event ? cudaErrorCapturedEvent : cudaSuccess; }
cudaError_t cudaStreamCreateWithPriority(cudaStream_t *s, unsigned, int) { *s = nullptr; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s)
{
    *s = g_capture ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamGetCaptureInfo(cudaStream_t st, cudaStreamCaptureStatus *s, unsigned long long *id, cudaGraph_t *, const cudaGraphNode_t **,
                                     size_t *)
{
    *id = g_capture;
    return cudaStreamIsCapturing(st, s);
}
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode *) { return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *, const cudaLaunchConfig_t *c)
{
    *n = 148 / static_cast<int>(c->attrs[0].val.clusterDim.x);
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void **p, const void *symbol) { *p = const_cast<void *>(symbol); return cudaSuccess; }
cudaError_t cudaGetDriverEntryPoint(const char *, void **fn, unsigned long long, cudaDriverEntryPointQueryResult *r)
{
    *fn = reinterpret_cast<void *>(encode);
    if (r) *r = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
}  // extern "C"

// ---- launchers of the kernels that are not linked ---------------------------------------------------------------------------
namespace enl {
cudaError_t launch_attention(const AttnParams &p, int, int, cudaStream_t) { return note('a', p.wait_first, 0, p.halves); }
cudaError_t launch_mass(const MassParams &p, int, int, cudaStream_t) { return note('m', p.wait_first); }
cudaError_t launch_small(const SmallParams &p, int, int, int, int, cudaStream_t) { return note('a', p.wait_first); }
cudaError_t launch_decode(const DecodeParams &p, int, int, cudaStream_t) { return note('d', p.wait_first); }
cudaError_t launch_combine(const CombineParams &, cudaStream_t) { return note('b', 0); }
cudaError_t launch_mass_finish(const FinishParams &, int, cudaStream_t) { return note('f', 0); }
cudaError_t launch_plan_write(void *, const void *, size_t bytes, cudaStream_t) { return note('w', 0, bytes); }
cudaError_t launch_page_scatter(void *, void *, const void *, const void *, const PageRun &, int, int, int, int, int, int, cudaStream_t) { return note('s', 0); }
cudaError_t launch_page_scatter_layers(void *, void *, size_t, int, int, const LayerSrc &, size_t, const PageRun &, int, int, int, int, int, int,
                                       cudaStream_t) { return note('s', 0); }
cudaError_t launch_page_copy(const uint8_t *, const uint8_t *, uint8_t *, uint8_t *, size_t, size_t, const int2 *, int, int, int, int, int,
                             cudaStream_t) { return note('l', 0); }
cudaError_t prepare_attention(int) { return cudaSuccess; }
cudaError_t prepare_mass(int) { return cudaSuccess; }
cudaError_t prepare_small(int) { return cudaSuccess; }
cudaError_t prepare_decode(int) { return cudaSuccess; }
bool attention_pairs_supported() { return true; }
int attention_park_slots() { return 25; }
}  // namespace enl
