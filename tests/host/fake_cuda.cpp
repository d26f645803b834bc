// fake_cuda.cpp -- a CUDA runtime on the host, linked with the library's own host code so that
// tests can follow what it allocates, copies and launches without a GPU, and make a call fail.
// Device memory is host memory, copies happen at once, kernels do nothing.  Every call that a
// test may ask about adds a line to a log: "what stream details".
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>

#include <cuda_runtime_api.h>

namespace {

// made before the constructors by which the library's own files register their kernels
#define EARLY __attribute__((init_priority(200)))
std::string g_log EARLY;
std::map<std::string, long long> g_set EARLY;     // fake_set: what a test asks for
std::map<const void*, std::string> g_names EARLY; // host stub -> kernel
std::map<const void*, long long> g_attr EARLY;    // kernel -> its dynamic shared memory limit
std::map<const void*, int> g_stream EARLY;        // streams by number, 1 the first created
int g_device = 0;

int number(cudaStream_t s) {
    if (!s) return 0;
    const auto it = g_stream.find(s);
    return it == g_stream.end() ? -1 : it->second;
}
void say(const std::string& what, cudaStream_t s, const std::string& more = "") {
    g_log += what + " " + std::to_string(number(s)) + (more.empty() ? "" : " " + more) + "\n";
}
// a kernel's name and its first template argument from the mangled name "...<length>k_...I<argument>..."
std::string kernel(const void* f) {
    const std::string m = g_names.count(f) ? g_names[f] : "?";
    const size_t a = m.find("k_");
    if (a == std::string::npos) return m;
    size_t d = a;
    while (d > 0 && isdigit((unsigned char)m[d - 1])) --d;
    const size_t n = (size_t)atoi(m.c_str() + d);
    return m.substr(a, n) + (a + n + 1 < m.size() && m[a + n] == 'I' ? std::string("<") + m[a + n + 1] + ">" : "");
}
cudaError_t launched(const void* f, dim3 grid, size_t smem, cudaStream_t s, const char* kind) {
    const long long limit = g_attr.count(f) ? g_attr[f] : 48 * 1024;
    say(kind, s, kernel(f) + " blocks " + std::to_string(grid.x) + " smem " + std::to_string(smem) + " limit " +
                     std::to_string(limit));
    return (long long)smem > limit ? cudaErrorInvalidValue : cudaSuccess;
}

struct Config {
    dim3 grid, block;
    size_t smem;
    cudaStream_t stream;
} g_cfg;

}  // namespace

extern "C" {

const char* fake_log() { return g_log.c_str(); }
void fake_clear() { g_log.clear(); }
void fake_set(const char* what, long long v) { g_set[what] = v; }
void fake_say(const char* what, cudaStream_t s, const char* more) { say(what, s, more); }

cudaError_t cudaGetDeviceCount(int* n) { *n = g_set.count("devices") ? (int)g_set["devices"] : 1; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { g_device = d; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 4; return cudaSuccess; }   // multiprocessors
cudaError_t cudaDeviceSynchronize() { say("sync-device", nullptr); return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "ok" : "fake failure"; }

cudaError_t cudaMalloc(void** p, size_t n) {
    say("malloc", nullptr, "device " + std::to_string(g_device));
    return (*p = aligned_alloc(256, (n + 255) / 256 * 256)) ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaFree(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return (*p = calloc(1, n)) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFreeHost(void* p) { free(p); return cudaSuccess; }
static cudaError_t copied() {
    if (g_set["failing_copies"] <= 0) return cudaSuccess;
    --g_set["failing_copies"];
    return cudaErrorUnknown;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
    say("copy-unordered", nullptr);
    if (copied() != cudaSuccess) return cudaErrorUnknown;
    memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t st) {
    say("copy", st);
    if (copied() != cudaSuccess) return cudaErrorUnknown;
    memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemset(void* d, int v, size_t n) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t st) { say("set", st); memset(d, v, n); return cudaSuccess; }

cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
    *s = reinterpret_cast<cudaStream_t>(malloc(1));
    g_stream[*s] = (int)g_stream.size() + 1;
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { say("sync", s); return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) { say("record", s); return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t* g) { say("recorded", s); *g = reinterpret_cast<cudaGraph_t>(1); return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) { *e = reinterpret_cast<cudaGraphExec_t>(1); return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t s) { say("replay", s); return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = reinterpret_cast<cudaEvent_t>(1); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }

cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute, int v) {
    say("limit", nullptr, kernel(f) + " " + std::to_string(v));
    g_attr[f] = v;
    return cudaSuccess;
}
void fake_cycles(void** args);
void fake_residual(void** args, cudaStream_t s);
cudaError_t cudaLaunchCooperativeKernel(const void* f, dim3 grid, dim3, void** args, size_t smem, cudaStream_t s) {
    if (g_set.count("cooperative_limit") && grid.x > g_set["cooperative_limit"]) {
        say("refused", s, kernel(f) + " blocks " + std::to_string(grid.x));
        return cudaErrorCooperativeLaunchTooLarge;
    }
    if (g_set["wait_runs_out"]) fake_cycles(args);
    return launched(f, grid, smem, s, "cooperative");
}

// what a compiled kernel launch calls
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
char __cudaInitModule(void**) { return 0; }
void __cudaRegisterFunction(void**, const char* f, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
    g_names[f] = name;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, cudaStream_t s) {
    g_cfg = Config{grid, block, smem, s};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* s) {
    *grid = g_cfg.grid;
    *block = g_cfg.block;
    *smem = g_cfg.smem;
    *static_cast<cudaStream_t*>(s) = g_cfg.stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3, void** args, size_t smem, cudaStream_t s) {
    if (kernel((const void*)k).rfind("k_residual", 0) == 0) fake_residual(args, s);
    return launched((const void*)k, grid, smem, s, "launch");
}

}  // extern "C"
