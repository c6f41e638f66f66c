// A CUDA runtime on the host, for tests of the C ABI's host side without a GPU: the solver library's own
// objects are linked against it.  Device memory is host memory with a list of the blocks handed out; copies
// check the blocks' ends and run at once; kernels are recorded, not run.  The test scripts failures
// (fake_fail), a memory limit (fake_limit) and the current device (fake_device).
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

#define API extern "C" __attribute__((visibility("default")))

namespace {
struct Block {
    size_t bytes;
    int device;
};
struct Launch {
    std::string kernel;
    std::vector<void*> pointers;  // the pointer arguments from the third on (after KParams and the store)
    unsigned blocks;
};
std::map<char*, Block> blocks;
std::map<const void*, std::string> names;
std::vector<Launch> launches;
std::map<std::string, int> calls, fail_at;  // calls of a function so far; the one that fails
std::map<std::pair<const void*, int>, int> attributes;
long long limit = 1LL << 40, used = 0;
int device = 0, pending = 0;
cudaError_t last = cudaSuccess;  // a launch's error, for cudaGetLastError

cudaError_t tick(const char* fn, cudaError_t e = cudaErrorUnknown) {
    const int n = ++calls[fn];
    return fail_at.count(fn) && fail_at[fn] == n ? e : cudaSuccess;
}
const std::pair<char* const, Block>* find(const void* p) {
    auto it = blocks.upper_bound((char*)p);
    if (it == blocks.begin()) return nullptr;
    --it;
    return (char*)p < it->first + it->second.bytes ? &*it : nullptr;
}
bool inside(const void* p, size_t n) {
    const auto* b = find(p);
    return !b || (char*)p + n <= b->first + b->second.bytes;
}
cudaError_t launch(const void* fn, dim3 grid, void** args) {
    if ((last = tick("launch")) != cudaSuccess) return last;
    Launch l;
    l.kernel = names.count(fn) ? names[fn] : "?";
    l.blocks = grid.x * grid.y * grid.z;
    // fields kernels: (KParams, store, four arrays)
    if (l.kernel.find("k_init_equilibrium") != std::string::npos || l.kernel.find("k_macroscopic") != std::string::npos)
        for (int k = 2; k < 6; ++k) l.pointers.push_back(*(void**)args[k]);
    launches.push_back(l);
    ++pending;
    return cudaSuccess;
}
CUresult pointer_attributes(unsigned n, CUpointer_attribute* a, void** out, CUdeviceptr ptr) {
    const auto* b = find((void*)ptr);
    for (unsigned k = 0; k < n; ++k) switch (a[k]) {
        case CU_POINTER_ATTRIBUTE_MEMORY_TYPE: *(unsigned*)out[k] = b ? CU_MEMORYTYPE_DEVICE : 0; break;
        case CU_POINTER_ATTRIBUTE_IS_MANAGED: *(unsigned*)out[k] = 0; break;
        case CU_POINTER_ATTRIBUTE_DEVICE_ORDINAL: *(int*)out[k] = b ? b->second.device : -2; break;
        case CU_POINTER_ATTRIBUTE_RANGE_START_ADDR: *(void**)out[k] = b ? b->first : nullptr; break;
        case CU_POINTER_ATTRIBUTE_RANGE_SIZE: *(size_t*)out[k] = b ? b->second.bytes : 0; break;
        default: return CUDA_ERROR_INVALID_VALUE;
        }
    return CUDA_SUCCESS;
}
CUresult encode_tiled(...) { return CUDA_SUCCESS; }
}  // namespace

// ---- what the test calls
API void fake_reset() {
    calls.clear();
    fail_at.clear();
    launches.clear();
    limit = 1LL << 40;
    pending = device = 0;
    last = cudaSuccess;
}
API void fake_fail(const char* fn, int nth) { calls[fn] = 0; fail_at[fn] = nth; }
API void fake_limit(long long bytes) { limit = bytes; }
API long long fake_used() { return used; }
API void fake_device(int d) { device = d; }
API int fake_pending() { return pending; }
API int fake_calls(const char* fn) { return calls[fn]; }
API void* fake_alloc(size_t bytes) {
    void* p = nullptr;
    return cudaMalloc(&p, bytes) == cudaSuccess ? p : nullptr;
}
API int fake_launches(const char* kernel) {
    int n = 0;
    for (const Launch& l : launches) n += l.kernel.find(kernel) != std::string::npos;
    return n;
}
API void* fake_pointer(const char* kernel, int k) {  // of the last launch of the kernel
    for (size_t i = launches.size(); i-- > 0;)
        if (launches[i].kernel.find(kernel) != std::string::npos) return launches[i].pointers[k];
    return nullptr;
}

API int fake_blocks(const char* kernel) {  // of the last launch of the kernel
    for (size_t i = launches.size(); i-- > 0;)
        if (launches[i].kernel.find(kernel) != std::string::npos) return (int)launches[i].blocks;
    return 0;
}

// ---- the runtime
API cudaError_t cudaMalloc(void** p, size_t n) {
    ++calls["cudaMalloc"];
    if (used + (long long)n > limit) return cudaErrorMemoryAllocation;
    *p = aligned_alloc(256, (n + 255) / 256 * 256 + 256);
    memset(*p, 0, n);
    blocks[(char*)*p] = Block{n, device};
    used += n;
    return cudaSuccess;
}
API cudaError_t cudaFree(void* p) {
    auto it = blocks.find((char*)p);
    if (it != blocks.end()) {
        used -= it->second.bytes;
        blocks.erase(it);
        free(p);
    }
    return cudaSuccess;
}
API cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { *p = calloc(1, n + 1); return cudaSuccess; }
API cudaError_t cudaFreeHost(void* p) { free(p); return cudaSuccess; }
API cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
    const cudaError_t e = tick("cudaMemcpyAsync");
    if (e != cudaSuccess) return e;
    if (!inside(d, n) || !inside(s, n)) return cudaErrorInvalidValue;
    memmove(d, s, n);
    ++pending;
    return cudaSuccess;
}
API cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { memmove(d, s, n); return cudaSuccess; }
API cudaError_t cudaMemset(void* d, int v, size_t n) { memset(d, v, n); return cudaSuccess; }
API cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { memset(d, v, n); return cudaSuccess; }
API cudaError_t cudaStreamSynchronize(cudaStream_t) { pending = 0; return tick("cudaStreamSynchronize"); }
API cudaError_t cudaGetLastError() {
    const cudaError_t e = last;
    last = cudaSuccess;
    return e;
}
API const char* cudaGetErrorString(cudaError_t) { return "scripted"; }
API const char* cudaGetErrorName(cudaError_t) { return "scripted"; }
API cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
API cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int d) {
    *v = a == cudaDevAttrMultiProcessorCount ? 100 + d : 1 << 20;
    return cudaSuccess;
}
API cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
    const auto* b = find(p);
    memset(a, 0, sizeof(*a));
    a->type = b ? cudaMemoryTypeDevice : cudaMemoryTypeUnregistered;
    a->device = b ? b->second.device : -2;
    return cudaSuccess;
}
API cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute, int v) {
    const cudaError_t e = tick("cudaFuncSetAttribute");
    if (e == cudaSuccess) attributes[{f, device}] = v;
    return e;
}
API cudaError_t cudaGetDriverEntryPointByVersion(const char* name, void** fn, unsigned, unsigned long long, cudaDriverEntryPointQueryResult* q) {
    *fn = strcmp(name, "cuPointerGetAttributes") == 0 ? (void*)pointer_attributes : (void*)encode_tiled;
    *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
// as on the device: a launch beyond the kernel's default 48 KB of dynamic shared memory needs the opt-in there
API cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* fn, void** args) {
    if (c->dynamicSmemBytes > 48 * 1024 && attributes[{fn, device}] < (int)c->dynamicSmemBytes) return last = cudaErrorInvalidValue;
    return launch(fn, c->gridDim, args);
}
API cudaError_t cudaLaunchKernel(const void* fn, dim3 g, dim3, void** args, size_t, cudaStream_t) { return launch(fn, g, args); }
API cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) { *n = 2; return cudaSuccess; }
API cudaError_t cudaGetSymbolAddress(void** p, const void*) { static char room[1 << 20]; *p = room; return cudaSuccess; }
API cudaError_t cudaEventCreate(cudaEvent_t*) { return cudaSuccess; }
API cudaError_t cudaEventCreateWithFlags(cudaEvent_t*, unsigned) { return cudaSuccess; }
API cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
API cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1; return cudaSuccess; }
API cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
API cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
API cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
API cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = nullptr; return cudaSuccess; }
API cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
API cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
API cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { *g = nullptr; return cudaSuccess; }
API cudaError_t cudaGraphInstantiate(cudaGraphExec_t*, cudaGraph_t, unsigned long long) { return cudaSuccess; }
API cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
API cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
API cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }

// ---- what the compiler's host stubs call
static dim3 cfg_grid, cfg_block;
static size_t cfg_smem;
static void* cfg_stream;
API unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t m, void* s) { cfg_grid = g; cfg_block = b; cfg_smem = m; cfg_stream = s; return 0; }
API cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* m, void* s) {
    *g = cfg_grid; *b = cfg_block; *m = cfg_smem; *(void**)s = cfg_stream;
    return cudaSuccess;
}
API cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* fn) { *k = (cudaKernel_t)fn; return cudaSuccess; }
API cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3, void** args, size_t, cudaStream_t) { return launch((const void*)k, g, args); }
API void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
API void __cudaRegisterFatBinaryEnd(void**) {}
API void __cudaUnregisterFatBinary(void**) {}
API void __cudaRegisterFunction(void**, const char* fn, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) { names[fn] = name; }
API void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
