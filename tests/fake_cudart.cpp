// Stand-in for the CUDA runtime under the host code of the library, for CPU tests of what
// happens when a call fails.  Device memory is host memory, kernels do nothing, every
// fallible call is counted and one of them can be made to fail, and copies and fills are
// checked against the blocks they touch.  Loaded with RTLD_GLOBAL before the library, in a
// process that does not load the real runtime.
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <string>

namespace {
struct Block {
    size_t size;
    bool old;   // allocated before fake_mark
};
std::map<char*, Block> blocks;
std::map<const void*, std::string> names;
std::string launches;
cudaError_t last = cudaSuccess;
long calls = 0, mallocs = 0, fail_call = -1, fail_malloc = -1, bad = 0;
int pattern = 0;

cudaError_t result(cudaError_t e) {
    if (e != cudaSuccess) last = e;
    return e;
}
bool fails() { return ++calls == fail_call; }
void check(const void* p, size_t n) {
    char* c = static_cast<char*>(const_cast<void*>(p));
    auto it = blocks.upper_bound(c);
    if (it == blocks.begin()) {
        ++bad;
        return;
    }
    --it;
    if (c + n > it->first + it->second.size) ++bad;
}
cudaError_t copy(void* d, const void* s, size_t n, cudaMemcpyKind k) {
    if (fails()) return result(cudaErrorInvalidValue);
    if (n == 0) return cudaSuccess;
    const long before = bad;
    if (k != cudaMemcpyDeviceToHost) check(d, n);
    if (k != cudaMemcpyHostToDevice) check(s, n);
    if (bad == before) memmove(d, s, n);
    return cudaSuccess;
}
cudaError_t fill(void* d, int v, size_t n) {
    if (fails()) return result(cudaErrorInvalidValue);
    const long before = bad;
    check(d, n);
    if (bad == before) memset(d, v, n);
    return cudaSuccess;
}
cudaError_t launch(const void* f) {
    if (fails()) return result(cudaErrorLaunchOutOfResources);
    launches += names.count(f) ? names[f] : "?";
    launches += "\n";
    return cudaSuccess;
}
}  // namespace

extern "C" {
// ------------------------------------------------------------ the tests' side
void fake_fail_call(long k) { fail_call = k < 0 ? -1 : calls + k; }       // the k-th call from now
void fake_fail_malloc(long k) { fail_malloc = k < 0 ? -1 : mallocs + k; }
void fake_pattern(int byte) { pattern = byte; }   // contents of new blocks
long fake_calls() { return calls; }
long fake_bad() { return bad; }
long fake_live() { return (long)blocks.size(); }
size_t fake_bytes() {
    size_t n = 0;
    for (auto& b : blocks) n += b.second.size;
    return n;
}
void fake_mark() {
    for (auto& b : blocks) b.second.old = true;
}
// FNV-1a over the blocks of the mark
unsigned long long fake_hash() {
    unsigned long long h = 1469598103934665603ull;
    for (auto& b : blocks)
        if (b.second.old)
            for (size_t i = 0; i < b.second.size; ++i) h = (h ^ (unsigned char)b.first[i]) * 1099511628211ull;
    return h;
}
const char* fake_launches() { return launches.c_str(); }
void fake_clear_launches() { launches.clear(); }

// -------------------------------------------------------------------- runtime
cudaError_t cudaMalloc(void** p, size_t n) {
    ++mallocs;
    if (mallocs == fail_malloc || fails()) return result(cudaErrorMemoryAllocation);
    char* c = static_cast<char*>(malloc(n ? n : 1));
    memset(c, pattern, n ? n : 1);
    blocks[c] = {n, false};
    *p = c;
    return cudaSuccess;
}
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { return cudaMalloc(p, n); }
cudaError_t cudaFree(void* p) {
    if (!p) return cudaSuccess;
    if (!blocks.erase(static_cast<char*>(p))) {
        ++bad;
        return cudaSuccess;
    }
    free(p);
    return cudaSuccess;
}
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { return cudaFree(p); }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) {
    if (fails()) return result(cudaErrorMemoryAllocation);
    *p = calloc(1, n ? n : 1);
    return cudaSuccess;
}
cudaError_t cudaMallocHost(void** p, size_t n) { return cudaHostAlloc(p, n, 0); }
cudaError_t cudaFreeHost(void* p) {
    free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind k) { return copy(d, s, n, k); }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t) { return copy(d, s, n, k); }
cudaError_t cudaMemset(void* d, int v, size_t n) { return fill(d, v, n); }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { return fill(d, v, n); }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return fails() ? result(cudaErrorUnknown) : cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* st, unsigned) {
    *st = nullptr;
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaGetLastError() {
    const cudaError_t e = last;
    last = cudaSuccess;
    return e;
}
cudaError_t cudaPeekAtLastError() { return last; }
const char* cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "an error of the stand-in"; }
cudaError_t cudaGetDevice(int* d) {
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) {
    *v = 152;
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
    *n = 1;
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void* f, void**) { return launch(f); }
cudaError_t cudaLaunchCooperativeKernel(const void* f, dim3, dim3, void**, size_t, cudaStream_t) { return launch(f); }
cudaError_t cudaLaunchKernel(const void* f, dim3, dim3, void**, size_t, cudaStream_t) { return launch(f); }
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
    *k = (cudaKernel_t)(f);
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t, cudaStream_t) { return launch((const void*)k); }
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void*) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaSuccess; }
void** __cudaRegisterFatBinary(void*) {
    static void* h;
    return &h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, void*, void*, void*, void*, int*) {
    names[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
}
