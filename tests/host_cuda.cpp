// A CUDA runtime for the library's host code alone, on a machine without a GPU:
// device memory is host memory, copies are memcpy, and a kernel launch records
// the kernel's name and does nothing.  A launch whose name contains a chosen
// text can be made to fail, and a stream capture of another thread can be
// declared to be under way, in which an unsafe call (an event query outside
// the relaxed mode) breaks that capture, as CUDA's documentation of
// cudaThreadExchangeStreamCaptureMode has it.
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>
#include <cuda_runtime_api.h>

namespace {
std::map<const void*, std::string> names;      // host stub -> kernel name
std::string launched;                          // names, one per line, and waits for events
std::string fail_name;
int fail_code = 0, fail_after = 0;
cudaError_t last = cudaSuccess;
cudaStreamCaptureMode mode = cudaStreamCaptureModeGlobal;
bool capturing = false, foreign = false, foreign_broken = false, event_busy = false;
struct Config {
    dim3 grid, block;
    size_t smem;
    void* stream;
};
std::vector<Config> configs;
long long allocated = 0;                       // bytes, over all calls

cudaError_t ret(cudaError_t e) {
    if (e != cudaSuccess) last = e;
    return e;
}
cudaError_t launch(const void* f) {
    const std::string& n = names[f];
    if (fail_code && n.find(fail_name) != std::string::npos && fail_after-- <= 0) return ret((cudaError_t)fail_code);
    launched += n + "\n";
    return cudaSuccess;
}
}  // namespace

extern "C" {
// ---- for the tests
const char* host_cuda_launched() { return launched.c_str(); }
void host_cuda_clear() { launched.clear(); }
void host_cuda_fail(const char* name, int code, int after) {   // launches of `name` fail, but for the first `after`
    fail_name = name;
    fail_after = after;
    fail_code = code;
}
void host_cuda_leave_error(int code) { last = (cudaError_t)code; }
void host_cuda_foreign_capture(int on) {
    foreign = on != 0;
    foreign_broken = false;
}
int host_cuda_foreign_capture_broken() { return foreign_broken; }
long long host_cuda_allocated() { return allocated; }
int host_cuda_mode() { return (int)mode; }
int host_cuda_last_error() { return (int)last; }
void host_cuda_capture(int on) { capturing = on != 0; }
void host_cuda_event_busy(int on) { event_busy = on != 0; }

// ---- what nvcc's host code calls
void** __cudaRegisterFatBinary(void*) {
    static void* handle[1];
    return handle;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* stub, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
    names[stub] = name;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, void* stream) {
    configs.push_back({grid, block, smem, stream});
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* stream) {
    *grid = configs.back().grid;
    *block = configs.back().block;
    *smem = configs.back().smem;
    *static_cast<void**>(stream) = configs.back().stream;
    configs.pop_back();
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* kernel, const void* stub) {
    *kernel = (cudaKernel_t)stub;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t kernel, dim3, dim3, void**, size_t, cudaStream_t) { return launch(kernel); }

// ---- the runtime calls of the library
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void* f, void**) { return launch(f); }
cudaError_t cudaGetLastError() {
    const cudaError_t e = last;
    last = cudaSuccess;
    return e;
}
cudaError_t cudaPeekAtLastError() { return last; }
const char* cudaGetErrorString(cudaError_t) { return "host CUDA error"; }
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
    return *n = 1, cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
    static char room[65536];
    return *p = room, cudaSuccess;
}
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) {
    allocated += (long long)n;
    return *p = calloc(1, n), cudaSuccess;
}
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { return free(p), cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { return memcpy(d, s, n), cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
    return memcpy(d, s, n), cudaSuccess;
}
cudaError_t cudaMemcpy2DAsync(void* d, size_t dp, const void* s, size_t sp, size_t w, size_t h, cudaMemcpyKind, cudaStream_t) {
    for (size_t i = 0; i < h; ++i) memcpy((char*)d + i * dp, (const char*)s + i * sp, w);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) { return memset(p, v, n), cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return *e = (cudaEvent_t)calloc(1, 1), cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return free(e), cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { return *ms = 1.0f, cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) {
    if (foreign && mode != cudaStreamCaptureModeRelaxed) {
        foreign_broken = true;
        return ret(cudaErrorStreamCaptureUnsupported);
    }
    return event_busy ? ret(cudaErrorNotReady) : cudaSuccess;
}
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode* m) {
    const cudaStreamCaptureMode old = mode;
    mode = *m;
    *m = old;
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return *s = (cudaStream_t)calloc(1, 1), cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { return free(s), cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) {
    launched += "wait\n";
    return cudaSuccess;
}
cudaError_t cudaStreamGetId(cudaStream_t s, unsigned long long* id) { return *id = (unsigned long long)s, cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* c) {
    return *c = capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone, cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return capturing = true, cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
    capturing = false;
    return *g = (cudaGraph_t)calloc(1, 1), cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t, unsigned long long) {
    return *x = (cudaGraphExec_t)calloc(1, 1), cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) { return free(g), cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) { return free(x), cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) {
    launched += "graph\n";
    return cudaSuccess;
}
}
