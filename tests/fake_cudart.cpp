// A stand-in for the CUDA runtime, linked under the library's own host code so that what it asks of the runtime can be
// checked without a GPU: two devices, device memory in host memory, kernels that do nothing.  Two rules of the real
// runtime are kept, because code can break them unnoticed on an idle single GPU:
//   - work given to a stream happens when that stream is waited for, not before: a copy that nobody waited for has not
//     happened, and a non-blocking stream does not wait for the legacy stream;
//   - a function's shared-memory opt-in belongs to one device: a launch with more than 48 KB is refused on a device that
//     the attribute was not set on.
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdlib>
#include <cstring>
#include <functional>
#include <map>
#include <mutex>
#include <set>
#include <utility>
#include <vector>

namespace {
std::mutex g_mu;
thread_local int t_device = 0;
thread_local cudaError_t t_last = cudaSuccess;
struct Stream {
    bool blocking;
    std::vector<std::function<void()>> work;
};
Stream g_legacy{true, {}};
std::set<Stream*> g_streams;
std::map<std::pair<int, const void*>, int> g_dynamic_smem;
std::map<std::pair<int, const void*>, std::vector<unsigned char>> g_symbols;
std::map<const void*, size_t> g_symbol_bytes;
std::map<const void*, const char*> g_names;
int g_launches[2];
const char* g_last_name = "";
int g_last_grid = 0, g_last_cluster = 0;
unsigned g_fill = 1;
int g_mallocs, g_frees;   // calls; of null pointers not counted
int g_fail_in = 0;        // the allocation that fails, counted from the next one (0: none)

void run(Stream* s) {
    for (auto& w : s->work) w();
    s->work.clear();
}
void wait_for(Stream* s) {
    if (s == &g_legacy) {
        for (Stream* o : g_streams)
            if (o->blocking) run(o);
        run(&g_legacy);
    } else {
        if (s->blocking) run(&g_legacy);
        run(s);
    }
}
Stream* stream_of(cudaStream_t s) { return s ? reinterpret_cast<Stream*>(s) : &g_legacy; }

cudaError_t copy(void* dst, const void* src, size_t n, cudaMemcpyKind kind, Stream* s) {
    std::lock_guard<std::mutex> lock(g_mu);
    if (kind == cudaMemcpyDeviceToHost) {   // to pageable memory: the call returns when the bytes are there
        wait_for(s);
        std::memcpy(dst, src, n);
    } else if (kind == cudaMemcpyHostToDevice) {   // from pageable memory: staged, then on its way
        std::vector<unsigned char> staged(static_cast<const unsigned char*>(src), static_cast<const unsigned char*>(src) + n);
        s->work.push_back([dst, staged] { std::memcpy(dst, staged.data(), staged.size()); });
    } else {
        s->work.push_back([dst, src, n] { std::memcpy(dst, src, n); });
    }
    return cudaSuccess;
}
cudaError_t launch(const void* func, dim3 grid, size_t dynamic_smem) {
    std::lock_guard<std::mutex> lock(g_mu);
    auto it = g_dynamic_smem.find({t_device, func});
    if (dynamic_smem > static_cast<size_t>(it == g_dynamic_smem.end() ? 48 * 1024 : it->second)) return t_last = cudaErrorInvalidValue;
    ++g_launches[t_device];
    g_last_name = g_names[func];
    g_last_grid = static_cast<int>(grid.x * grid.y * grid.z);
    return cudaSuccess;
}
int cluster_of(const cudaLaunchConfig_t* c) {
    for (unsigned i = 0; i < c->numAttrs; ++i)
        if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) return static_cast<int>(c->attrs[i].val.clusterDim.x);
    return 1;
}
CUresult encode_tiled() { return CUDA_SUCCESS; }
thread_local struct { dim3 grid, block; size_t smem; cudaStream_t stream; } t_config;
}  // namespace

extern "C" {
int fake_launches(int device) { return g_launches[device]; }
const char* fake_last_kernel() { return g_last_name; }   // mangled
int fake_last_grid() { return g_last_grid; }             // CTAs
int fake_last_cluster() { return g_last_cluster; }       // CTAs per cluster
int fake_mallocs() { return g_mallocs; }
int fake_frees() { return g_frees; }
void fake_fail_malloc(int nth) { g_fail_in = nth; }
int fake_pending() {   // operations that no wait has covered yet
    std::lock_guard<std::mutex> lock(g_mu);
    size_t n = g_legacy.work.size();
    for (Stream* s : g_streams) n += s->work.size();
    return static_cast<int>(n);
}

cudaError_t cudaGetDevice(int* d) { *d = t_device; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { if (d < 0 || d > 1) return cudaErrorInvalidDevice; t_device = d; return cudaSuccess; }
cudaError_t cudaGetDeviceProperties_v2(cudaDeviceProp* p, int) { std::memset(p, 0, sizeof(*p)); p->major = 10; p->multiProcessorCount = 148; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 148; return cudaSuccess; }
cudaError_t cudaGetLastError() { const cudaError_t e = t_last; t_last = cudaSuccess; return e; }
cudaError_t cudaMalloc(void** p, size_t n) {   // fresh memory: different bytes every time
    std::lock_guard<std::mutex> lock(g_mu);
    if (g_fail_in > 0 && --g_fail_in == 0) return t_last = cudaErrorMemoryAllocation;
    *p = std::aligned_alloc(1024, (n + 1023) / 1024 * 1024);
    if (!*p) return cudaErrorMemoryAllocation;
    std::memset(*p, static_cast<int>(g_fill++ * 37 & 0xff), n);
    ++g_mallocs;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
    std::lock_guard<std::mutex> lock(g_mu);
    for (Stream* s : g_streams) run(s);
    run(&g_legacy);
    if (p) ++g_frees;
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind k) { return copy(d, s, n, k, &g_legacy); }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t st) { return copy(d, s, n, k, stream_of(st)); }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t st) {
    std::lock_guard<std::mutex> lock(g_mu);
    stream_of(st)->work.push_back([d, v, n] { std::memset(d, v, n); });
    return cudaSuccess;
}
cudaError_t cudaMemset(void* d, int v, size_t n) { return cudaMemsetAsync(d, v, n, nullptr); }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned flags) {
    std::lock_guard<std::mutex> lock(g_mu);
    Stream* n = new Stream{!(flags & cudaStreamNonBlocking), {}};
    g_streams.insert(n);
    *s = reinterpret_cast<cudaStream_t>(n);
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) {
    std::lock_guard<std::mutex> lock(g_mu);
    wait_for(stream_of(s));
    g_streams.erase(stream_of(s));
    delete stream_of(s);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
    std::lock_guard<std::mutex> lock(g_mu);
    wait_for(stream_of(s));
    return cudaSuccess;
}
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode*) { return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
    std::lock_guard<std::mutex> lock(g_mu);
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) g_dynamic_smem[{t_device, f}] = v;
    return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) { std::memset(a, 0, sizeof(*a)); a->numRegs = 112; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void* f, const cudaLaunchConfig_t* c) {
    std::lock_guard<std::mutex> lock(g_mu);
    auto it = g_dynamic_smem.find({t_device, f});
    if (c->dynamicSmemBytes > static_cast<size_t>(it == g_dynamic_smem.end() ? 48 * 1024 : it->second)) return cudaErrorInvalidValue;
    // what a B200 answers for one CTA and for two per SM
    static const int two_per_sm[9] = {0, 296, 148, 93, 71, 56, 45, 37, 33};
    const int size = cluster_of(c);
    *n = size > 8 ? 0 : 2 * (c->dynamicSmemBytes + 1024) <= 233472 ? two_per_sm[size] : two_per_sm[size] / 2;
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) { g_last_cluster = cluster_of(c); return launch(f, c->gridDim, c->dynamicSmemBytes); }
cudaError_t cudaLaunchKernel(const void* f, dim3 grid, dim3, void**, size_t smem, cudaStream_t) { return launch(f, grid, smem); }
cudaError_t cudaGetSymbolAddress(void** p, const void* symbol) {
    std::lock_guard<std::mutex> lock(g_mu);
    auto& mem = g_symbols[{t_device, symbol}];
    if (mem.empty()) mem.resize(g_symbol_bytes[symbol]);
    *p = mem.data();
    return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPoint(const char*, void** p, unsigned long long, cudaDriverEntryPointQueryResult* q) {
    *p = reinterpret_cast<void*>(encode_tiled);
    if (q) *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}

// what the compiler's registration code calls
void** __cudaRegisterFatBinary(void*) { static void* handle; return &handle; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
char __cudaInitModule(void**) { return 0; }
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) { g_names[host] = name; }
void __cudaRegisterVar(void**, char* host, char*, const char*, int, size_t bytes, int, int) { g_symbol_bytes[host] = bytes; }
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, struct CUstream_st* s) { t_config = {g, b, smem, s}; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* s) {
    *g = t_config.grid; *b = t_config.block; *smem = t_config.smem; *static_cast<cudaStream_t*>(s) = t_config.stream;
    return cudaSuccess;
}
}
