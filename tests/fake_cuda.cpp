// A stand-in for the CUDA runtime, for tests of the library's host code that a
// GPU must not run: allocations that fail, a second device, a launch that is
// refused.  Device memory is host memory (zeroed), copies and memsets happen at
// once, kernels do nothing.  Linked with the library's own objects in place of
// the runtime.  A copy or memset whose device range is not wholly inside one
// allocation is counted (fake_bad) and refused.
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <vector>

namespace {
std::recursive_mutex mu;
std::map<char *, size_t> blocks;              // start -> size, device and pinned
std::map<const void *, std::string> kernels;
std::map<std::string, void *> symbols;
std::map<std::pair<int, const void *>, int> dyn_smem;     // (device, kernel) -> bytes allowed
std::map<std::string, long> calls;            // runtime calls and kernels launched, by name
long n_alloc = 0, fail_at = 0, bad = 0;
size_t in_use = 0, peak = 0, limit = ~(size_t)0;
bool clusters = true;
thread_local int device = 0;
thread_local cudaError_t last = cudaSuccess;
struct Config { dim3 grid, block; size_t smem; void *stream; };
thread_local std::vector<Config> configs;
using Lock = std::lock_guard<std::recursive_mutex>;

cudaError_t ret(cudaError_t e) {
    if (e != cudaSuccess) last = e;
    return e;
}
cudaError_t note(const char *name, cudaError_t e = cudaSuccess) {
    Lock l(mu);
    calls[name]++;
    return ret(e);
}
cudaError_t alloc(void **p, size_t n, bool counts) {
    Lock l(mu);
    *p = nullptr;
    if ((++n_alloc >= fail_at && fail_at) || (counts && in_use + n > limit)) return ret(cudaErrorMemoryAllocation);
    char *q = (char *)std::calloc(n ? n : 1, 1);
    if (!q) return ret(cudaErrorMemoryAllocation);
    blocks[q] = n;
    if (counts) in_use += n;
    if (in_use > peak) peak = in_use;
    *p = q;
    return cudaSuccess;
}
cudaError_t release(void *p, bool counts) {
    Lock l(mu);
    if (!p) return cudaSuccess;
    auto it = blocks.find((char *)p);
    if (it == blocks.end()) { bad++; return ret(cudaErrorInvalidValue); }
    if (counts) in_use -= it->second;
    blocks.erase(it);
    std::free(p);
    return cudaSuccess;
}
// [p, p + n): not null, and inside its block if it starts in one
bool ok(const void *p, size_t n) {
    if (!p) return n == 0;
    auto it = blocks.upper_bound((char *)p);
    if (it == blocks.begin()) return true;                    // caller's own host memory
    --it;
    const size_t at = (size_t)((char *)p - it->first);
    return at >= (it->second ? it->second : 1) || at + n <= it->second;
}
cudaError_t copy(void *d, const void *s, size_t n) {
    Lock l(mu);
    if (!ok(d, n) || !ok(s, n)) { bad++; return ret(cudaErrorInvalidValue); }
    if (n) std::memmove(d, s, n);
    return cudaSuccess;
}
cudaError_t launch(const void *k, size_t smem) {
    Lock l(mu);
    const std::string &name = kernels[k];
    calls[name]++;
    auto it = dyn_smem.find({device, k});
    const size_t allowed = it == dyn_smem.end() ? 48 * 1024 : (size_t)it->second;
    return ret(smem > allowed ? cudaErrorInvalidValue : cudaSuccess);
}
}  // namespace

extern "C" {

// ---- controls
void fake_reset() {
    Lock l(mu);
    n_alloc = fail_at = bad = 0;
    limit = ~(size_t)0;
    clusters = true;
    last = cudaSuccess;
    calls.clear();
}
// the k-th allocation from now and all later ones are refused (0: none)
void fake_fail_at(long k) { Lock l(mu); n_alloc = 0; fail_at = k; }
// `bytes` more than now; fake_peak: the most from there on
void fake_limit(size_t bytes) { Lock l(mu); limit = in_use + bytes; peak = in_use; }
void fake_clusters(int allowed) { clusters = allowed != 0; }
long fake_allocs() { Lock l(mu); return n_alloc; }
long fake_bad() { Lock l(mu); return bad; }
size_t fake_in_use() { Lock l(mu); return in_use; }
size_t fake_peak() { Lock l(mu); return peak; }
// calls of a runtime function or launches of kernels whose name contains `what`
long fake_calls(const char *what) {
    Lock l(mu);
    long n = 0;
    for (auto &c : calls) if (c.first.find(what) != std::string::npos) n += c.second;
    return n;
}

// ---- registration and launches
void **__cudaRegisterFatBinary(void *) { static void *h[1]; return h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *,
                            int *) {
    Lock l(mu);
    kernels[host] = name;
}
void __cudaRegisterVar(void **, char *host, char *, const char *, int, size_t size, int, int) {
    Lock l(mu);
    char *p = (char *)std::calloc(size, 1);
    blocks[p] = size;
    symbols[std::to_string((size_t)host)] = p;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t s, struct CUstream_st *stream) {
    configs.push_back({g, b, s, stream});
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *s, void *stream) {
    const Config c = configs.back();
    configs.pop_back();
    *g = c.grid;
    *b = c.block;
    *s = c.smem;
    *(void **)stream = c.stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void **, size_t smem, cudaStream_t) {
    return launch((const void *)k, smem);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *k, void **) {
    if (!clusters && c->numAttrs) return note("refused", cudaErrorLaunchOutOfResources);
    return launch(k, c->dynamicSmemBytes);
}
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *, const cudaLaunchConfig_t *) {
    *n = clusters ? 8 : 0;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) {
    *n = 4;
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute, int v) {
    Lock l(mu);
    dyn_smem[{device, f}] = v;
    return cudaSuccess;
}

// ---- devices, streams, events
cudaError_t cudaSetDevice(int d) { device = d; return ret(d >= 0 && d < 2 ? cudaSuccess : cudaErrorInvalidDevice); }
cudaError_t cudaGetDevice(int *d) { *d = device; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 8; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return note("cudaDeviceSynchronize"); }
cudaError_t cudaGetLastError() { const cudaError_t e = last; last = cudaSuccess; return e; }
const char *cudaGetErrorString(cudaError_t e) {
    thread_local std::string s;
    s = "fake error " + std::to_string((int)e);
    return s.c_str();
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = (cudaStream_t)1; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return note("cudaStreamSynchronize"); }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = (cudaEvent_t)1; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { *e = (cudaEvent_t)1; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t) {
    if (!e) { Lock l(mu); bad++; return ret(cudaErrorInvalidResourceHandle); }
    return cudaSuccess;
}
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }

// ---- memory
cudaError_t cudaMalloc(void **p, size_t n) { return alloc(p, n, true); }
cudaError_t cudaFree(void *p) { note("cudaFree"); return release(p, true); }
cudaError_t cudaMallocHost(void **p, size_t n) { return alloc(p, n, false); }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return alloc(p, n, false); }
cudaError_t cudaFreeHost(void *p) { return release(p, false); }
cudaError_t cudaGetSymbolAddress(void **p, const void *s) { *p = symbols[std::to_string((size_t)s)]; return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { return copy(d, s, n); }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) { return copy(d, s, n); }
cudaError_t cudaMemcpy2DAsync(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h, cudaMemcpyKind,
                              cudaStream_t) {
    for (size_t i = 0; i < h; i++)
        if (copy((char *)d + i * dp, (const char *)s + i * sp, w) != cudaSuccess) return last;
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) {
    Lock l(mu);
    if (!ok(d, n)) { bad++; return ret(cudaErrorInvalidValue); }
    if (n) std::memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaMemset(void *d, int v, size_t n) { return cudaMemsetAsync(d, v, n, nullptr); }

}  // extern "C"
