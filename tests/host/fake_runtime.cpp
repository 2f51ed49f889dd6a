// A CUDA runtime without a GPU, for tests of the library's host code: the library's own objects are linked
// against this file instead of the runtime. Device memory is host memory, a launch runs nothing and is only
// counted, there are several devices, and the calls follow the rules that the host code has to keep:
//   * a cudaMemcpy from host memory may return before it has arrived; only a wait on the legacy stream or
//     the device says that it has, and a launch on another stream before that reads what was there
//     before (fake_early_launches counts such launches);
//   * while a stream is captured, allocations break the capture unless the thread's mode is relaxed, and so
//     does anything on the legacy stream;
//   * a kernel takes more than 48 KB of dynamic shared memory only on devices where that was allowed.
#include <cuda_runtime.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <utility>

namespace {
struct Fake {
    int device = 0;
    int pending = 0;  // copies that may not have arrived: on the legacy stream,
    int pending_own = 0;  // and on streams that the library made
    int capturing = 0, broken = 0;  // the caller captures a stream; a call that broke the capture
    cudaStreamCaptureMode mode = cudaStreamCaptureModeGlobal;  // of the calling thread
    int early = 0;    // launches that could have read them too early
    int launches[5] = {0, 0, 0, 0, 0};  // single steps, ring passes, tiled passes, line launches, batched steps
    std::map<std::pair<const void*, int>, int> shared;  // dynamic shared memory allowed, by kernel and device
    bool refuse_shared = false;
    cudaError_t last = cudaSuccess;
};
Fake g;

std::map<const void*, std::string>& names() {  // of the kernels, filled while the library is loaded
    static std::map<const void*, std::string> n;
    return n;
}

struct CallConfig {
    dim3 grid, block;
    size_t shared;
    cudaStream_t stream;
} call;

// A call that a capture under way does not allow unless the thread asked for it.
bool unsafe() {
    if (!g.capturing || g.mode == cudaStreamCaptureModeRelaxed) return false;
    g.broken = 1;
    return true;
}

const cudaStream_t kOwnStream = reinterpret_cast<cudaStream_t>(0x2000);

bool legacy(cudaStream_t s) { return s == nullptr || s == cudaStreamLegacy; }

cudaError_t done(cudaError_t e) {
    if (e != cudaSuccess) g.last = e;
    return e;
}

bool fits(const void* kernel, size_t bytes) {
    const auto it = g.shared.find({kernel, g.device});
    return bytes <= 48 << 10 || (it != g.shared.end() && bytes <= (size_t)it->second);
}

cudaError_t launch(const void* kernel, size_t shared, cudaStream_t s) {
    if (!fits(kernel, shared)) return done(cudaErrorInvalidValue);
    if ((g.pending && !legacy(s)) || g.pending_own) ++g.early;
    const std::string& name = names()[kernel];
    const char* kinds[5][2] = {{"step_kernel", "step_early_kernel"}, {"fused2_kernel", ""}, {"tile2_kernel", ""},
                               {"line_kernel", ""}, {"batch_kernel", ""}};
    for (int k = 0; k < 5; ++k)
        for (const char* part : kinds[k])
            if (*part && name.find(part) != std::string::npos) ++g.launches[k];
    return cudaSuccess;
}
}  // namespace

extern "C" {
void fake_reset() {  // what was allowed stays: the library remembers it too
    const auto shared = g.shared;
    g = Fake();
    g.shared = shared;
}
void fake_set_device(int d) { g.device = d; }
void fake_capture(int on) { g.capturing = on; g.broken = 0; }
int fake_capture_broken() { return g.broken; }
void fake_refuse_shared(int refuse) { g.refuse_shared = refuse != 0; }
int fake_early_launches() { return g.early; }
int fake_launches(int kind) { return g.launches[kind]; }

cudaError_t cudaGetDevice(int* d) { *d = g.device; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { g.device = d; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrL2CacheSize ? 129 << 20 : 0;
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void* kernel, cudaFuncAttribute a, int v) {
    if (g.refuse_shared) return done(cudaErrorInvalidValue);
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) g.shared[{kernel, g.device}] = v;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* blocks, const void* kernel, int, size_t shared, unsigned) {
    *blocks = fits(kernel, shared) ? 2 : 0;
    return cudaSuccess;
}
cudaError_t cudaMemGetInfo(size_t* f, size_t* t) { *f = *t = (size_t)1 << 38; return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) {
    if (unsafe()) return done(cudaErrorStreamCaptureUnsupported);
    *p = calloc(n, 1);
    return done(*p ? cudaSuccess : cudaErrorMemoryAllocation);
}
cudaError_t cudaFree(void* p) {
    if (p && unsafe()) return done(cudaErrorStreamCaptureUnsupported);
    free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind k) {
    if (g.capturing) g.broken = 1;  // on the legacy stream: never beside a capture
    if (g.capturing) return done(cudaErrorStreamCaptureImplicit);
    memcpy(d, s, n);
    if (k == cudaMemcpyHostToDevice) ++g.pending;
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t st) {
    memcpy(d, s, n);
    if (st == kOwnStream && k == cudaMemcpyHostToDevice) ++g.pending_own;
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
    if (s != kOwnStream && unsafe()) return done(cudaErrorStreamCaptureUnsupported);
    if (legacy(s)) g.pending = 0;
    if (s == kOwnStream) g.pending_own = 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { g.pending = g.pending_own = 0; return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = kOwnStream; return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* st) {
    *st = g.capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode* m) { std::swap(*m, g.mode); return cudaSuccess; }
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
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* kernel, void**) {
    return launch(kernel, c->dynamicSmemBytes, c->stream);
}

// What the compiler's host code calls to register kernels and for <<<>>> launches.
void** __cudaRegisterFatBinary(void*) { static void* handle; return &handle; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* kernel, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
    names()[kernel] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
cudaError_t __cudaGetKernel(cudaKernel_t* out, const void* kernel) {
    *out = reinterpret_cast<cudaKernel_t>(const_cast<void*>(kernel));
    return cudaSuccess;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t shared, struct CUstream_st* s) {
    call = CallConfig{grid, block, shared, s};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* shared, void* s) {
    *grid = call.grid;
    *block = call.block;
    *shared = call.shared;
    *static_cast<cudaStream_t*>(s) = call.stream;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t kernel, dim3, dim3, void**, size_t shared, cudaStream_t s) {
    return launch(kernel, shared, s);
}
}  // extern "C"
