// A CUDA runtime for tests of the library's host code without a GPU: librg's
// objects are linked against it instead of libcudart.  Kernels do not run;
// memory is host memory, and copies and fills happen at once.  Every call that
// orders work is written to a log (fake_log), one line each, naming streams
// and events by number (stream 0 is the legacy default stream).  Launches are
// refused as the real runtime refuses them: more dynamic shared memory than
// the kernel was allowed on the current device, or a grid beyond the limits.
#include <cuda_runtime.h>

#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <set>
#include <string>

namespace {
std::string g_log;
std::map<const void*, std::string> g_kernels;
std::map<std::pair<int, const void*>, size_t> g_smem;  // (device, kernel): dynamic shared memory allowed
std::map<void*, int> g_stream_prio, g_capturing;
std::set<void*> g_pending;                             // events that cudaEventQuery finds unfinished
void* g_cleared = nullptr;                             // by the last cudaMemset
int g_dev = 0, g_fail_launch = 0, g_launches = 0, g_mallocs = 0, g_fail_malloc = 0, g_next = 1;
cudaError_t g_last = cudaSuccess;
cudaStreamCaptureMode g_capture_mode = cudaStreamCaptureModeGlobal;

void log(const char* fmt, ...) {
    char b[256];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(b, sizeof b, fmt, ap);
    va_end(ap);
    g_log += b;
    g_log += '\n';
}
cudaError_t ret(cudaError_t e) { return e == cudaSuccess ? e : g_last = e; }
void* handle() { return reinterpret_cast<void*>((size_t)g_next++ * 16); }
int id(const void* h) { return (int)((size_t)h / 16); }  // (the legacy stream has the handle 1)

cudaError_t launch(const void* f, dim3 g, size_t smem, cudaStream_t s) {
    if (++g_launches == g_fail_launch) return ret(cudaErrorLaunchOutOfResources);
    const auto it = g_smem.find({g_dev, f});
    if (smem > (it == g_smem.end() ? 48u * 1024u : it->second)) return ret(cudaErrorInvalidValue);
    if (g.x == 0 || g.y == 0 || g.z == 0 || g.x > 0x7FFFFFFFu || g.y > 65535 || g.z > 65535)
        return ret(cudaErrorInvalidConfiguration);
    log("launch %s s%d %u %u %u", g_kernels[f].c_str(), id(s), g.x, g.y, g.z);
    return cudaSuccess;
}
cudaError_t get(void** p, size_t n) {
    *p = aligned_alloc(256, (n + 255) & ~(size_t)255);
    if (!*p) return ret(cudaErrorMemoryAllocation);
    memset(*p, 0, n);
    return cudaSuccess;
}
}  // namespace

extern "C" {
// ---- the test's own
const char* fake_log() { return g_log.c_str(); }
void fake_reset() { g_log.clear(), g_launches = g_fail_launch = 0; }
void fake_fail_launch(int k) { g_launches = 0, g_fail_launch = k; }
void fake_fail_malloc(int k) { g_mallocs = 0, g_fail_malloc = k; }
void* fake_stream(int prio) {
    void* s = handle();
    g_stream_prio[s] = prio;
    return s;
}
void fake_set_capturing(void* s, int on) { g_capturing[s] = on; }
const char* fake_kernels() {  // the names of the library's kernels
    static std::string all;
    all.clear();
    for (const auto& k : g_kernels) all += k.second + '\n';
    return all.c_str();
}
void* fake_cleared() { return g_cleared; }
void fake_finish() { g_pending.clear(); }  // the device catches up

// ---- the runtime
cudaError_t cudaGetLastError() {
    const cudaError_t e = g_last;
    g_last = cudaSuccess;
    return e;
}
const char* cudaGetErrorString(cudaError_t) { return "fake error"; }
cudaError_t cudaGetDevice(int* d) { return *d = g_dev, cudaSuccess; }
cudaError_t cudaSetDevice(int d) { return g_dev = d, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) { return memset(p, 0, sizeof *p), cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return log("devsync"), g_pending.clear(), cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) { return ++g_mallocs == g_fail_malloc ? ret(cudaErrorMemoryAllocation) : get(p, n); }
cudaError_t cudaMallocHost(void** p, size_t n) { return get(p, n); }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { return get(p, n); }
cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t, cudaStream_t) { return get(p, n); }
cudaError_t cudaFree(void* p) { return free(p), cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { return free(p), cudaSuccess; }
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { return free(p), cudaSuccess; }
cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps*) {
    return *p = reinterpret_cast<cudaMemPool_t>(handle()), log("pool d%d", g_dev), cudaSuccess;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t n) { return log("trim d%d %zu", g_dev, n), cudaSuccess; }
cudaError_t cudaMemset(void* p, int v, size_t n) { return log("memset s0"), memset(g_cleared = p, v, n), cudaSuccess; }
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t s) {
    return log("memset s%d", id(s)), memset(p, v, n), cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
    return log("copy s0"), memcpy(d, s, n), cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* p, size_t n, cudaMemcpyKind, cudaStream_t s) {
    return log("copy s%d %zu", id(s), n), memcpy(d, p, n), cudaSuccess;
}
cudaError_t cudaMemcpy2D(void*, size_t, const void*, size_t, size_t, size_t, cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void* sym) { return *p = const_cast<void*>(sym), cudaSuccess; }
cudaError_t cudaStreamCreateWithPriority(cudaStream_t* s, unsigned flags, int prio) {
    *s = static_cast<cudaStream_t>(fake_stream(prio));
    return log("stream s%d flags %u prio %d", id(*s), flags, prio), cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned f) { return cudaStreamCreateWithPriority(s, f, 0); }
cudaError_t cudaStreamGetPriority(cudaStream_t s, int* p) { return *p = g_stream_prio[s], cudaSuccess; }
cudaError_t cudaStreamGetId(cudaStream_t s, unsigned long long* n) { return *n = (size_t)s, cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { return log("destroy s%d", id(s)), cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
    return g_capturing[s] ? ret(cudaErrorStreamCaptureUnsupported) : (log("streamsync s%d", id(s)), cudaSuccess);
}
cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus* c) {
    return *c = g_capturing[s] ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone, cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
    return log("wait s%d e%d", id(s), id(e)), cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return ret(cudaErrorNotSupported); }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t*) { return ret(cudaErrorNotSupported); }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t*, cudaGraph_t, unsigned long long) { return ret(cudaErrorNotSupported); }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return ret(cudaErrorNotSupported); }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) {
    return *e = reinterpret_cast<cudaEvent_t>(handle()), cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return g_pending.erase(e), cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
    return log("record e%d s%d", id(e), id(s)), g_pending.insert(e), cudaSuccess;
}
cudaError_t cudaEventQuery(cudaEvent_t e) {
    if (g_capture_mode != cudaStreamCaptureModeRelaxed) log("query outside of the relaxed capture mode");
    return g_pending.count(e) ? ret(cudaErrorNotReady) : cudaSuccess;
}
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode* m) {
    std::swap(*m, g_capture_mode);
    return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t e) { return g_pending.erase(e), cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { return *ms = 0, cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) g_smem[{g_dev, f}] = (size_t)v;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
    return *n = 8, cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
    return launch(f, c->gridDim, c->dynamicSmemBytes, c->stream);
}
// ---- what nvcc's host stubs call
cudaError_t __cudaLaunchKernel(cudaKernel_t f, dim3 g, dim3, void**, size_t smem, cudaStream_t s) {
    return launch(reinterpret_cast<const void*>(f), g, smem, s);
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
    return *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(f)), cudaSuccess;
}
static thread_local struct { dim3 g, b; size_t smem; cudaStream_t s; } t_config;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, cudaStream_t s) {
    t_config = {g, b, smem, s};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* s) {
    *g = t_config.g, *b = t_config.b, *smem = t_config.smem, *static_cast<cudaStream_t*>(s) = t_config.s;
    return cudaSuccess;
}
void** __cudaRegisterFatBinary(void*) {
    static void* h;
    return &h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* f, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
    g_kernels[f] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
}
