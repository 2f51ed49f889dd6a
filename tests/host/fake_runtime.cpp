// A CUDA runtime without a GPU, for tests of the library's host code: csrc/api.cu is linked against this
// file instead of the runtime (and against fake_launchers.cu). Device memory is host memory, a launch does
// nothing but count, and the calls follow the rules that the host code has to keep:
//   * a cudaMemcpy from host memory may return before it has arrived; only a wait on the legacy stream or
//     the device says that it has, and a launch on another stream before that reads what was there
//     before (fake_early_launches counts such launches).
#include <cuda_runtime.h>

#include <cstdlib>
#include <cstring>

namespace {
struct Fake {
    int device = 0;
    int pending = 0;  // copies that may not have arrived
    int early = 0;    // launches that could have read them too early
    int launches[4] = {0, 0, 0, 0};  // single steps, ring passes, tiled passes, line launches
    cudaError_t last = cudaSuccess;
};
Fake g;

bool legacy(cudaStream_t s) { return s == nullptr || s == cudaStreamLegacy; }

cudaError_t done(cudaError_t e) {
    if (e != cudaSuccess) g.last = e;
    return e;
}
}  // namespace

extern "C" {
int fake_launched(cudaStream_t s, int kind) {
    if (g.pending && !legacy(s)) ++g.early;
    if (kind >= 0) ++g.launches[kind];
    return 1;
}
void fake_reset() { g = Fake(); }
int fake_early_launches() { return g.early; }
int fake_launches(int kind) { return g.launches[kind]; }

cudaError_t cudaGetDevice(int* d) { *d = g.device; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { g.device = d; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrL2CacheSize ? 129 << 20 : 0;
    return cudaSuccess;
}
cudaError_t cudaMemGetInfo(size_t* f, size_t* t) { *f = *t = (size_t)1 << 38; return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) {
    *p = calloc(n, 1);
    return done(*p ? cudaSuccess : cudaErrorMemoryAllocation);
}
cudaError_t cudaFree(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind k) {
    memcpy(d, s, n);
    if (k == cudaMemcpyHostToDevice) ++g.pending;
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
    memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
    if (legacy(s)) g.pending = 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { g.pending = 0; return cudaSuccess; }
cudaError_t cudaGetLastError() {
    const cudaError_t e = g.last;
    g.last = cudaSuccess;
    return e;
}
const char* cudaGetErrorString(cudaError_t) { return "fake runtime error"; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
    static double scratch[1 << 16];
    *p = scratch;
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 0.f; return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* out) { *out = nullptr; return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t, unsigned long long) { *x = nullptr; return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t s) { fake_launched(s, -1); return cudaSuccess; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void*, void**) {
    fake_launched(c->stream, -1);
    return cudaSuccess;
}

// What the compiler's host code calls to register and launch kernels.
void** __cudaRegisterFatBinary(void*) { static void* handle; return &handle; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
cudaError_t __cudaGetKernel(cudaKernel_t*, const void*) { return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void**, size_t, cudaStream_t s) {
    fake_launched(s, -1);
    return cudaSuccess;
}
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaSuccess; }
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, struct CUstream_st*) { return 0; }
}  // extern "C"
