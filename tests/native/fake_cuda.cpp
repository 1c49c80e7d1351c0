// A CUDA runtime in host memory, linked with the library's own objects in the
// place of the real one: allocations are lazily backed host mappings under a
// byte limit, copies and memsets act on them, and launches run nothing but are
// recorded. What the library allocates, frees, sizes and launches can so be
// tested without a GPU, failed allocations included.
#include <sys/mman.h>

#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <vector>

#include <cuda_runtime_api.h>

extern "C" void fk_on_launch(const char* kernel);  // sketch_fields.cu

namespace {

constexpr size_t kPage = 4096;
constexpr size_t kTouch = 1u << 26;  // larger copies and memsets are left out (no test reads what they move)

struct Launch {
    std::string name;
    unsigned grid, block;
};
struct State {
    std::recursive_mutex mu;
    std::map<char*, size_t> live;  // device allocations
    uint64_t limit = ~0ull, used = 0, allocs = 0;
    int64_t fail_at = 0;
    bool fail_on = false;                  // and every one after it
    cudaError_t last = cudaSuccess;        // until cudaGetLastError takes it
    std::map<const void*, std::string> names;
    std::vector<Launch> launches;
};
State& state() {
    static State* s = new State;  // outlives the library's static destructors
    return *s;
}

cudaError_t alloc(void** p, size_t bytes) {
    State& S = state();
    std::lock_guard<std::recursive_mutex> lk(S.mu);
    *p = nullptr;
    ++S.allocs;
    bool fail = S.fail_at > 0 && --S.fail_at == 0;
    if (fail && S.fail_on) S.fail_at = 1;
    fail = fail || bytes > S.limit || S.used > S.limit - bytes;
    void* q = fail ? MAP_FAILED
                   : mmap(nullptr, (bytes + kPage - 1) / kPage * kPage, PROT_READ | PROT_WRITE,
                          MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
    if (q == MAP_FAILED) return S.last = cudaErrorMemoryAllocation;
    S.live[(char*)q] = bytes;
    S.used += bytes;
    *p = q;
    return cudaSuccess;
}

cudaError_t release(void* p) {
    State& S = state();
    std::lock_guard<std::recursive_mutex> lk(S.mu);
    if (!p) return cudaSuccess;
    auto it = S.live.find((char*)p);
    if (it == S.live.end()) return cudaErrorInvalidValue;
    munmap(p, (it->second + kPage - 1) / kPage * kPage);
    S.used -= it->second;
    S.live.erase(it);
    return cudaSuccess;
}

cudaError_t launch(const void* f, dim3 grid, dim3 block) {
    State& S = state();
    std::lock_guard<std::recursive_mutex> lk(S.mu);
    const std::string& name = S.names[f];
    S.launches.push_back({name, grid.x, block.x});
    fk_on_launch(name.c_str());
    return cudaSuccess;
}

struct Config {
    dim3 grid, block;
    size_t smem;
    cudaStream_t stream;
};
thread_local std::vector<Config> g_config;

}  // namespace

extern "C" {

// ------------------------------------------------------- the runtime's names
void** __cudaRegisterFatBinary(void* p) { return (void**)p; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* device, int, uint3*, uint3*, dim3*, dim3*, int*) {
    state().names[host] = device;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t m, struct CUstream_st* st) {
    g_config.push_back({g, b, m, st});
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* m, void* st) {
    const Config c = g_config.back();
    g_config.pop_back();
    *g = c.grid;
    *b = c.block;
    *m = c.smem;
    *(cudaStream_t*)st = c.stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
    *k = (cudaKernel_t)f;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void**, size_t, cudaStream_t) {
    return launch((const void*)k, g, b);
}
cudaError_t cudaLaunchCooperativeKernel(const void* f, dim3 g, dim3 b, void**, size_t, cudaStream_t) {
    return launch(f, g, b);
}
cudaError_t cudaMalloc(void** p, size_t n) { return alloc(p, n); }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { return alloc(p, n); }
cudaError_t cudaFree(void* p) { return release(p); }
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { return release(p); }
cudaError_t cudaMallocHost(void** p, size_t n) { return (*p = malloc(n)) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFreeHost(void* p) {
    free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
    if (n <= kTouch) memmove(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
    if (n <= kTouch) memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : 1;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetDefaultMemPool(cudaMemPool_t* p, int) {
    *p = nullptr;
    return cudaSuccess;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t) { return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) {
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaGetLastError() {
    const cudaError_t e = state().last;
    state().last = cudaSuccess;
    return e;
}
const char* cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "error"; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
    *p = nullptr;
    return cudaErrorInvalidSymbol;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t) {
    *n = 4;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
    *n = 4;
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
    *s = nullptr;
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) {
    *e = (cudaEvent_t)malloc(1);
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) {
    free(e);
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
    *ms = 0;
    return cudaSuccess;
}

// ---------------------------------------------------------- the test's side
// bytes the device holds in all from now on; failures and the launch record start anew
void fk_start(uint64_t limit) {
    State& S = state();
    S.limit = limit;
    S.allocs = 0;
    S.fail_at = 0;
    S.last = cudaSuccess;
    S.launches.clear();
}
// the k-th allocation from here fails, and every one after it if `on` (0: none)
void fk_fail_at(int64_t k, int on) {
    state().fail_at = k;
    state().fail_on = on != 0;
}
uint64_t fk_allocs() { return state().allocs; }
uint64_t fk_live(const void* p) {  // bytes of the live allocation that starts at p, 0 if there is none
    State& S = state();
    auto it = S.live.find((char*)p);
    return p && it != S.live.end() ? it->second : 0;
}
uint64_t fk_used() { return state().used; }
int fk_launch(uint64_t i, char* name, uint64_t len, unsigned* grid, unsigned* block) {
    State& S = state();
    if (i >= S.launches.size()) return 0;
    strncpy(name, S.launches[i].name.c_str(), len - 1);
    name[len - 1] = 0;
    *grid = S.launches[i].grid;
    *block = S.launches[i].block;
    return 1;
}
}  // extern "C"
