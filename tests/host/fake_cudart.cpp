// A stand-in for the CUDA runtime (test program part, preloaded before librtpn.so): the calls the library makes,
// with device memory as reserved host address space and kernels that are counted, not run.  A test can
// make the n-th next call of a name fail, bound the memory, give a pointer another device, and read the
// kernels launched and the copies made.  Small copies between known ranges are carried out.
#include <cuda_runtime.h>
#include <sys/mman.h>

#include <cstring>
#include <map>
#include <string>
#include <vector>

// cudaTypedefs' signature of the one driver entry point the library asks for
extern "C" int fake_encode(void* map, ...) {
    std::memset(map, 1, 128);
    return 0;
}

namespace {
struct Range {
    size_t bytes;
    int device;
};
auto& g_mem = *new std::map<const char*, Range>;  // never destroyed: the library frees at exit
auto& g_names = *new std::map<const void*, std::string>;
auto& g_fail = *new std::map<std::string, std::pair<int, int>>;  // api -> (calls until it fails, code)
auto& g_log = *new std::string;
auto& g_out = *new std::string;
size_t g_used = 0, g_limit = (size_t)1 << 60;
cudaError_t g_last = cudaSuccess;
bool g_capturing = false;
float g_ms = 0, g_ms_step = 1;  // the next elapsed time, and how the ones after it change

cudaError_t check(const char* api) {
    auto it = g_fail.find(api);
    if (it != g_fail.end() && --it->second.first < 0) {
        const int code = it->second.second;
        g_fail.erase(it);
        return g_last = (cudaError_t)code;
    }
    return cudaSuccess;
}
cudaError_t launched(const void* fn, dim3 block) {
    if (cudaError_t e = check("launch")) return e;
    auto it = g_names.find(fn);
    g_log += "K " + (it == g_names.end() ? std::string("?") : it->second) + " threads " +
             std::to_string(block.x * block.y * block.z) + "\n";
    return cudaSuccess;
}
struct Config {
    dim3 grid, block;
    size_t smem;
    void* stream;
};
std::vector<Config> g_configs;
}  // namespace

extern "C" {
// ---- the test's side
void fake_fail(const char* api, int after, int code) { g_fail[api] = {after, code}; }
void fake_limit(size_t bytes) { g_limit = bytes; }
size_t fake_used() { return g_used; }
void fake_capturing(int on) { g_capturing = on != 0; }
void fake_elapsed(float first, float step) {
    g_ms = first;
    g_ms_step = step;
}
void fake_clear() { g_log.clear(); }
const char* fake_log() {
    g_out = g_log;
    return g_out.c_str();
}
// device memory of another GPU
void* fake_remote(size_t bytes) {
    void* p = nullptr;
    cudaMalloc(&p, bytes);
    g_mem[(const char*)p].device = 1;
    return p;
}

// ---- memory
cudaError_t cudaMalloc(void** p, size_t n) {
    *p = nullptr;
    if (cudaError_t e = check("cudaMalloc")) return e;
    if (g_used + n > g_limit) return g_last = cudaErrorMemoryAllocation;
    void* m = mmap(nullptr, n + 1, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
    if (m == MAP_FAILED) return g_last = cudaErrorMemoryAllocation;
    g_mem[(const char*)m] = {n, 0};
    g_used += n;
    *p = m;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
    auto it = g_mem.find((const char*)p);
    if (it == g_mem.end()) return cudaSuccess;
    g_used -= it->second.bytes;
    munmap(p, it->second.bytes + 1);
    g_mem.erase(it);
    return cudaSuccess;
}
static cudaError_t copy(const char* api, void* d, const void* s, size_t n) {
    if (cudaError_t e = check(api)) return e;
    g_log += std::string("C ") + api + " " + std::to_string(n) + "\n";
    if (n <= (1u << 24)) std::memmove(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { return copy("cudaMemcpy", d, s, n); }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
    return copy("cudaMemcpyAsync", d, s, n);
}
cudaError_t cudaMemcpy2DAsync(void*, size_t, const void*, size_t, size_t, size_t, cudaMemcpyKind, cudaStream_t) {
    return check("cudaMemcpy2DAsync");
}
cudaError_t cudaMemset(void*, int, size_t) { return check("cudaMemset"); }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return check("cudaMemsetAsync"); }
cudaError_t cudaMemcpyToSymbol(const void*, const void*, size_t, size_t, cudaMemcpyKind) { return check("cudaMemcpyToSymbol"); }
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
    *p = nullptr;
    return cudaErrorInvalidSymbol;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
    std::memset(a, 0, sizeof *a);
    a->type = cudaMemoryTypeUnregistered;
    auto it = g_mem.upper_bound((const char*)p);
    if (it != g_mem.begin()) {
        --it;
        if ((const char*)p < it->first + it->second.bytes) {
            a->type = cudaMemoryTypeDevice;
            a->device = it->second.device;
            a->devicePointer = const_cast<void*>(p);
        }
    }
    return cudaSuccess;
}

// ---- device, errors
cudaError_t cudaGetDevice(int* d) {
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : 0;
    return cudaSuccess;
}
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) {
    std::memset(p, 0, sizeof *p);
    std::strcpy(p->name, "fake");
    return cudaSuccess;
}
cudaError_t cudaGetLastError() {
    const cudaError_t e = g_last;
    g_last = cudaSuccess;
    return e;
}
const char* cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "injected"; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** fn, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* r) {
    *fn = (void*)&fake_encode;
    if (r) *r = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}

// ---- streams, events, graphs
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
    *s = (cudaStream_t)0x10;
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) {
    g_log += "S\n";
    return check("cudaStreamSynchronize");
}
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
    *s = g_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
    *g = (cudaGraph_t)0x20;
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
    *e = (cudaGraphExec_t)0x30;
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) {
    *e = (cudaEvent_t)0x40;
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
    *ms = g_ms += g_ms_step;
    return cudaSuccess;
}

// ---- kernels
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t) {
    *n = 1;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
    *n = 1;
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* fn, void**) { return launched(fn, c->blockDim); }
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* fn) {
    *k = (cudaKernel_t)fn;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3 block, void**, size_t, cudaStream_t) {
    return launched((const void*)k, block);
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, void* stream) {
    g_configs.push_back({grid, block, smem, stream});
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* stream) {
    const Config c = g_configs.back();
    g_configs.pop_back();
    *grid = c.grid;
    *block = c.block;
    *smem = c.smem;
    *(void**)stream = c.stream;
    return cudaSuccess;
}
void** __cudaRegisterFatBinary(void*) {
    static void* handle = nullptr;
    return &handle;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
    g_names[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
}
