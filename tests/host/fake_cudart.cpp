// A CUDA runtime without a GPU, linked in place of the real one by
// tests/test_devices_cpu.py: two devices whose memory is host memory and whose
// kernels do nothing. It keeps what the real runtime keeps per device and
// answers with its error codes: a kernel's dynamic shared memory limit holds on
// the device that was current when it was raised (48 KiB before), memory is
// used with its own device current. Lowering a kernel's limit is an error here:
// another thread may stand between raising it and its launch.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <map>
#include <utility>

namespace {
constexpr int kDevices = 2;
int g_device = 0;
std::map<const char *, std::pair<size_t, int>> g_mem;   // begin -> bytes, device
std::map<std::pair<int, const void *>, int> g_limit;    // (device, kernel) -> dynamic shared memory
struct Call {
    dim3 grid, block;
    size_t smem;
    cudaStream_t stream;
} g_call;
long g_launches = 0, g_optin = 0;
size_t g_most = (size_t)-1;   // larger device and page-locked allocations fail

bool wrong_device(const void *p) {
    auto it = g_mem.upper_bound(static_cast<const char *>(p));
    if (it == g_mem.begin()) return false;
    --it;
    return static_cast<const char *>(p) < it->first + it->second.first && it->second.second != g_device;
}
cudaError_t launch(const void *f, size_t smem) {
    ++g_launches;
    if (smem > 48 * 1024) {
        ++g_optin;
        auto it = g_limit.find({g_device, f});
        if (it == g_limit.end() || (size_t)it->second < smem) return cudaErrorInvalidValue;
    }
    return cudaSuccess;
}
cudaError_t alloc(void **p, size_t n) {
    *p = std::calloc(1, std::max<size_t>(n, 1));
    return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
}  // namespace

extern "C" {
long fake_launches() { return g_launches; }
long fake_optin_launches() { return g_optin; }
void fake_limit_alloc(size_t bytes) { g_most = bytes; }

void **__cudaRegisterFatBinary(void *) {
    static void *h;
    return &h;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, struct CUstream_st *s) {
    g_call = Call{g, b, smem, s};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *smem, void *s) {
    *g = g_call.grid;
    *b = g_call.block;
    *smem = g_call.smem;
    *static_cast<cudaStream_t *>(s) = g_call.stream;
    return cudaSuccess;
}
static cudaError_t g_last = cudaSuccess;
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) {
    *k = reinterpret_cast<cudaKernel_t>(const_cast<void *>(f));
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void **, size_t smem, cudaStream_t) {
    return g_last = launch(reinterpret_cast<const void *>(k), smem);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **) {
    return g_last = launch(f, c->dynamicSmemBytes);
}
cudaError_t cudaGetLastError() {
    const cudaError_t e = g_last;
    g_last = cudaSuccess;
    return e;
}
const char *cudaGetErrorName(cudaError_t e) { return e == cudaErrorInvalidValue ? "cudaErrorInvalidValue" : "error"; }
const char *cudaGetErrorString(cudaError_t) { return "reported by the test's runtime"; }

cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute a, int v) {
    if (a != cudaFuncAttributeMaxDynamicSharedMemorySize) return cudaSuccess;
    int &limit = g_limit[{g_device, f}];
    if (v < limit || v > 227 * 1024) return cudaErrorInvalidValue;
    limit = v;
    return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *a, const void *) {
    std::memset(a, 0, sizeof *a);
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) {
    *n = 1;
    return cudaSuccess;
}

cudaError_t cudaGetDeviceCount(int *n) {
    *n = kDevices;
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int d) {
    if (d < 0 || d >= kDevices) return cudaErrorInvalidDevice;
    g_device = d;
    return cudaSuccess;
}
cudaError_t cudaGetDeviceProperties(cudaDeviceProp *p, int) {
    std::memset(p, 0, sizeof *p);
    p->multiProcessorCount = 4;
    p->major = 10;
    p->minor = 3;
    return cudaSuccess;
}

cudaError_t cudaMalloc(void **p, size_t n) {
    const cudaError_t e = n > g_most ? (g_last = cudaErrorMemoryAllocation) : alloc(p, n);
    if (e == cudaSuccess) g_mem[static_cast<const char *>(*p)] = {n, g_device};
    return e;
}
cudaError_t cudaFree(void *p) {
    g_mem.erase(static_cast<const char *>(p));
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) {
    return n > g_most ? (g_last = cudaErrorMemoryAllocation) : alloc(p, n);
}
cudaError_t cudaFreeHost(void *p) {
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaHostGetDevicePointer(void **d, void *h, unsigned) {
    *d = h;
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void **p, const void *) {
    static void *mem[kDevices] = {};
    if (!mem[g_device]) mem[g_device] = std::calloc(1, 16u << 20);
    *p = mem[g_device];
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) {
    if (wrong_device(d) || wrong_device(s)) return cudaErrorInvalidValue;
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) {
    if (wrong_device(d)) return cudaErrorInvalidValue;
    std::memset(d, v, n);
    return cudaSuccess;
}

static cudaError_t handle(void **h) {
    static char some;
    *h = &some;
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) { return handle(reinterpret_cast<void **>(e)); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return handle(reinterpret_cast<void **>(e)); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) {
    *ms = 1.0f;
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { return handle(reinterpret_cast<void **>(s)); }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) { return handle(reinterpret_cast<void **>(g)); }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t, unsigned long long) {
    return handle(reinterpret_cast<void **>(x));
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
}
