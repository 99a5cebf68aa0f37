// A stand-in for the CUDA runtime, for tests of libgs's host code without a GPU: the
// library's own objects are linked against this file instead of the runtime.  Device
// memory is host memory mapped on first touch (so sizes are those of a real device),
// kernels do not run; the ones named in check() have the arrays they would be given
// looked up among the live allocations, and those named in hook() leave the counts
// that the host reads back.
#include <cuda_runtime_api.h>
#include <sys/mman.h>

#include <cstdint>
#include <cstring>
#include <map>
#include <mutex>
#include <string>

namespace {

std::recursive_mutex mu;
std::map<uintptr_t, size_t> live;                 // device allocations
std::map<const void*, std::string> names;         // kernels by their host address
std::string report;                               // what went wrong, one line each
size_t limit = ~(size_t)0, total_live = 0;
uint64_t n_alloc = 0, pairs = 0;
uint64_t list_mean = 0, block_mean = 0;           // entries of a pixel's blend list, of a block's list
uint64_t npix = 0, scan_n = 0;                    // pixels of the view that is built, length of the scan under way

struct Cfg {
    dim3 g, b;
    size_t smem;
    void* st;
};
thread_local Cfg cfg;

void say(const std::string& s) {
    if (report.size() < 4000) report += s + "\n";
}

cudaError_t take(void** p, size_t n) {
    std::lock_guard<std::recursive_mutex> lk(mu);
    n_alloc++;
    *p = nullptr;
    if (n > limit || total_live > limit - n) return cudaErrorMemoryAllocation;
    const size_t len = ((n + 4095) & ~(size_t)4095) + 4096;   // a gap behind each allocation
    void* q = mmap(nullptr, len, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
    if (q == MAP_FAILED) return cudaErrorMemoryAllocation;
    live[(uintptr_t)q] = n;
    total_live += n;
    *p = q;
    return cudaSuccess;
}

cudaError_t give(void* p) {
    if (!p) return cudaSuccess;
    std::lock_guard<std::recursive_mutex> lk(mu);
    auto it = live.find((uintptr_t)p);
    if (it == live.end()) {
        say("freed twice, or never allocated");
        return cudaErrorInvalidValue;
    }
    total_live -= it->second;
    munmap(p, ((it->second + 4095) & ~(size_t)4095) + 4096);
    live.erase(it);
    return cudaSuccess;
}

// is [p, p + bytes) inside one live allocation?
void inside(const std::string& k, const char* what, const void* p, size_t bytes) {
    if (bytes == 0) return;
    auto it = live.upper_bound((uintptr_t)p);
    if (p && it != live.begin()) {
        --it;
        if ((uintptr_t)p + bytes <= it->first + it->second) return;
    }
    say(k + ": " + what + " needs " + std::to_string(bytes) + " bytes that are not allocated");
}

template <class T>
T arg(void** a, int i) {
    T v;
    memcpy(&v, a[i], sizeof(v));
    return v;
}

void check(const std::string& name, void** a) {
    const auto is = [&](const char* s) { return name.find(s) != std::string::npos; };
    if (is("k_tile_hist")) {
        const size_t tpad = ((size_t)arg<int>(a, 5) + 7) & ~(size_t)7, warps = cfg.b.x / 32;
        inside("k_tile_hist", "the warps' counts", arg<void*>(a, 7), 2 * tpad * warps * cfg.g.x);
        inside("k_tile_hist", "the segments' counts", arg<void*>(a, 8), 4 * tpad * cfg.g.x);
    }
    if (is("k_tile_place")) {
        const size_t nt = (size_t)arg<int>(a, 5);
        inside("k_tile_place", "the tiles' starts", arg<void*>(a, 9), 4 * nt);
        inside("k_tile_place", "the lists", arg<void*>(a, 10), 4 * (size_t)arg<unsigned long long*>(a, 6)[0]);
    }
    if (is("12k_preprocessI") || is("16k_preprocess_tmaI")) {   // the file's name is part of its other kernels' names
        const uint64_t n = arg<uint64_t>(a, 1);
        const int at = is("16k_preprocess_tmaI") ? 4 : 5;   // records, rects, keys, values
        const size_t each[4] = {48, 8, 4, 4};
        for (int i = 0; i < 4; i++)
            if (arg<void*>(a, at + i)) inside("k_preprocess", "an output", arg<void*>(a, at + i), each[i] * n);
    }
}

void hook(const std::string& name, void** a) {
    const auto is = [&](const char* s) { return name.find(s) != std::string::npos; };
    const auto put = [&](unsigned long long* t, uint64_t sum, uint64_t cap) {
        t[0] = sum < cap ? sum : cap;
        t[1] = sum > cap ? 1 : 0;
        t[2] = sum;
    };
    if (is("k_order_small")) put(arg<unsigned long long*>(a, 7), pairs, arg<uint64_t>(a, 8));
    if (is("k_list_lens")) npix = arg<uint64_t>(a, 1);
    if (is("15k_scan_partialsP")) scan_n = arg<uint64_t>(a, 1);
    if (is("k_scan_partials_top")) {
        const uint64_t cap = arg<uint64_t>(a, 3);
        // a view's build: list lengths, its blocks' entries, or rows (one a tile)
        const uint64_t each = scan_n == npix ? (list_mean + 4) & ~(uint64_t)3 : (scan_n == npix / 64 ? block_mean : 1);
        put(arg<unsigned long long*>(a, 2), cap == ~0ull ? scan_n * each : pairs, cap);
    }
}

constexpr size_t kSmall = 1 << 20;   // larger copies and fills are left out: nobody reads them

}  // namespace

extern "C" {

// what the tests set and read
__attribute__((visibility("default"))) void fake_limit(uint64_t bytes) { limit = bytes; }
__attribute__((visibility("default"))) void fake_counts(uint64_t p, uint64_t list, uint64_t block) {
    pairs = p;
    list_mean = list;
    block_mean = block;
}
__attribute__((visibility("default"))) uint64_t fake_live() { return total_live; }
__attribute__((visibility("default"))) uint64_t fake_allocations() { return n_alloc; }
__attribute__((visibility("default"))) const char* fake_report() { return report.c_str(); }

cudaError_t cudaMalloc(void** p, size_t n) { return take(p, n); }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { return take(p, n); }
cudaError_t cudaFree(void* p) { return give(p); }
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { return give(p); }
cudaError_t cudaMallocHost(void** p, size_t n) {
    *p = calloc(1, n);
    return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaFreeHost(void* p) {
    free(p);
    return cudaSuccess;
}
cudaError_t cudaMemGetInfo(size_t* f, size_t* t) {
    std::lock_guard<std::recursive_mutex> lk(mu);
    *t = limit;
    *f = limit - total_live;
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind k) {
    if (n <= kSmall && k != cudaMemcpyDeviceToDevice) memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t) {
    return cudaMemcpy(d, s, n, k);
}
cudaError_t cudaMemset(void* d, int v, size_t n) {
    if (n <= kSmall) memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { return cudaMemset(d, v, n); }

cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "error"; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
    *n = 4;
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) {
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) {
    *v = 152;   // the only one asked for: multiprocessors
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) { return take(p, 4096); }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
    *s = (cudaStream_t)calloc(1, 8);
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) {
    free(s);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
    *g = (cudaGraph_t)calloc(1, 8);
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
    *e = (cudaGraphExec_t)calloc(1, 8);
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) {
    free(e);
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) {
    free(g);
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) {
    *e = (cudaEvent_t)calloc(1, 8);
    return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t e) {
    free(e);
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
    *ms = 1.0f;
    return cudaSuccess;
}

// the compiler's launch interface
void** __cudaRegisterFatBinary(void*) {
    static void* h;
    return &h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
    std::lock_guard<std::recursive_mutex> lk(mu);
    names[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, void* st) {
    cfg = Cfg{g, b, smem, st};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* st) {
    *g = cfg.g;
    *b = cfg.b;
    *smem = cfg.smem;
    *(void**)st = cfg.st;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
    *k = (cudaKernel_t)f;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void** a, size_t, cudaStream_t) {
    std::lock_guard<std::recursive_mutex> lk(mu);
    const std::string& name = names[(const void*)k];
    check(name, a);
    hook(name, a);
    return cudaSuccess;
}

}  // extern "C"
