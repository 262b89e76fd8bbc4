// A CUDA runtime on host memory, for tests of the host side of the C ABI where
// no GPU is: kernels do not run, copies are memcpy.  A test sets which copy
// fails and on which device memory lives; fake_launches.cu writes down the
// library's launches.
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <cuda_runtime_api.h>
#include "fake_device.h"

namespace {

std::string g_log, g_status_at;
int g_status_bits = 0, g_copies_left = -1, g_last = 0;
std::map<uintptr_t, std::pair<size_t, int>> g_mem;   // device memory: start -> size, device

cudaError_t done(cudaError_t e)
{
    if (e != cudaSuccess) g_last = e;
    return e;
}

cudaError_t copy(void* d, const void* s, size_t n, cudaMemcpyKind k)
{
    if (g_copies_left == 0) return done(cudaErrorInvalidValue);
    if (g_copies_left > 0) g_copies_left--;
    const bool from = k == cudaMemcpyDeviceToDevice || k == cudaMemcpyDeviceToHost;
    const bool to = k == cudaMemcpyDeviceToDevice || k == cudaMemcpyHostToDevice;
    if ((from && fake_device_of(s) < 0) || (to && fake_device_of(d) < 0)) return done(cudaErrorInvalidValue);
    if (k == cudaMemcpyDeviceToDevice) fake_note("copy", nullptr);
    memcpy(d, s, n);
    return cudaSuccess;
}

}  // namespace

int fake_device_of(const void* p)
{
    auto it = g_mem.upper_bound((uintptr_t)p);
    if (it == g_mem.begin()) return -1;
    --it;
    return (uintptr_t)p < it->first + it->second.first ? it->second.second : -1;
}

void fake_note(const char* what, int* status)
{
    g_log += what;
    g_log += ' ';
    if (status && g_status_at == what) *status |= g_status_bits;
}

extern "C" {

// ---- the test's controls
const char* fake_log() { return g_log.c_str(); }
void fake_reset(const char* status_at, int bits, int copies_left)
{
    g_log.clear();
    g_status_at = status_at;
    g_status_bits = bits;
    g_copies_left = copies_left;
}
void* fake_alloc(size_t n, int device)
{
    void* p = calloc(1, n ? n : 1);
    g_mem[(uintptr_t)p] = {n, device};
    return p;
}

// ---- the runtime
cudaError_t cudaMalloc(void** p, size_t n)
{
    *p = fake_alloc(n, 0);
    return cudaSuccess;
}
cudaError_t cudaFree(void* p)
{
    g_mem.erase((uintptr_t)p);
    free(p);
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned)
{
    *p = calloc(1, n);
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p)
{
    free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind k) { return copy(d, s, n, k); }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t) { return copy(d, s, n, k); }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t)
{
    memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p)
{
    memset(a, 0, sizeof(*a));
    const int dev = fake_device_of(p);
    a->type = dev < 0 ? cudaMemoryTypeUnregistered : cudaMemoryTypeDevice;
    a->device = dev < 0 ? -2 : dev;
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int* n) { *n = 2; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 4; return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "fake error"; }
cudaError_t cudaGetLastError()
{
    const int e = g_last;
    g_last = 0;
    return (cudaError_t)e;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)1; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaErrorNotSupported; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t*) { return cudaErrorNotSupported; }
cudaError_t cudaEventCreate(cudaEvent_t*) { return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.0f; return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphGetNodes(cudaGraph_t, cudaGraphNode_t*, size_t*) { return cudaErrorNotSupported; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t*, cudaGraph_t, unsigned long long) { return cudaErrorNotSupported; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t cudaGraphNodeGetType(cudaGraphNode_t, cudaGraphNodeType*) { return cudaErrorNotSupported; }

// ---- kernel launches of sph_api.cu itself: nothing runs
void** __cudaRegisterFatBinary(void*) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
char __cudaInitModule(void**) { return 1; }
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, void*, void*, void*, void*, int*) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, cudaStream_t) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaSuccess; }
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void*) { *k = nullptr; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void**, size_t, cudaStream_t) { return cudaSuccess; }

}  // extern "C"
