// A stand-in for the CUDA runtime that runs the library's host path without a GPU: device memory is
// host memory with a limit, kernels do nothing, streams run in order at once. The fake_* functions
// set the limit and read the counts of the calls that the host path is checked for.
#include <cstddef>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>

namespace {
size_t limit_bytes = ~(size_t)0, used_bytes = 0;
std::map<void*, size_t> blocks;
long n_malloc = 0, n_refused = 0, n_capture = 0, n_launch = 0, n_device_sync = 0;
char handle;  // what every opaque handle points to
}  // namespace

struct Dim3 { unsigned x, y, z; };

extern "C" {
void fake_limit(size_t bytes) { limit_bytes = bytes; }
size_t fake_used() { return used_bytes; }
long fake_count(int what) {
    const long v[] = {n_malloc, n_refused, n_capture, n_launch, n_device_sync};
    return v[what];
}

int cudaMalloc(void** p, size_t n) {
    ++n_malloc;
    if (used_bytes + n > limit_bytes) {
        ++n_refused;
        return 2;  // cudaErrorMemoryAllocation
    }
    if (posix_memalign(p, 256, n)) return 2;
    std::memset(*p, 0, n);
    blocks[*p] = n;
    used_bytes += n;
    return 0;
}
int cudaFree(void* p) {
    auto it = blocks.find(p);
    if (it == blocks.end()) return p ? 1 : 0;
    used_bytes -= it->second;
    blocks.erase(it);
    std::free(p);
    return 0;
}
int cudaMemcpy(void* d, const void* s, size_t n, int) { std::memcpy(d, s, n); return 0; }
int cudaMemcpyAsync(void* d, const void* s, size_t n, int, void*) { std::memcpy(d, s, n); return 0; }
int cudaMemset(void* d, int v, size_t n) { std::memset(d, v, n); return 0; }
int cudaMemsetAsync(void* d, int v, size_t n, void*) { std::memset(d, v, n); return 0; }
int cudaSetDevice(int) { return 0; }
int cudaGetDevice(int* d) { *d = 0; return 0; }
int cudaGetDeviceCount(int* n) { *n = 1; return 0; }
int cudaDeviceGetAttribute(int* v, int, int) { *v = 152; return 0; }
int cudaDeviceSynchronize() { ++n_device_sync; return 0; }
int cudaGetLastError() { return 0; }
const char* cudaGetErrorString(int) { return "fake"; }
int cudaEventCreate(void** e) { *e = &handle; return 0; }
int cudaEventCreateWithFlags(void** e, unsigned) { *e = &handle; return 0; }
int cudaEventDestroy(void*) { return 0; }
int cudaEventElapsedTime(float* ms, void*, void*) { *ms = 1.f; return 0; }
int cudaEventQuery(void*) { return 0; }
int cudaEventRecord(void*, void*) { return 0; }
int cudaEventRecordWithFlags(void*, void*, unsigned) { return 0; }
int cudaEventSynchronize(void*) { return 0; }
int cudaStreamCreateWithFlags(void** s, unsigned) { *s = &handle; return 0; }
int cudaStreamDestroy(void*) { return 0; }
int cudaStreamSynchronize(void*) { return 0; }
int cudaStreamWaitEvent(void*, void*, unsigned) { return 0; }
int cudaStreamBeginCapture(void*, int) { ++n_capture; return 0; }
int cudaStreamEndCapture(void*, void** g) { *g = &handle; return 0; }
int cudaGraphDestroy(void*) { return 0; }
int cudaGraphExecDestroy(void*) { return 0; }
int cudaGraphInstantiate(void** x, void*, unsigned long long) { *x = &handle; return 0; }
int cudaGraphLaunch(void*, void*) { ++n_launch; return 0; }
int cudaFuncSetAttribute(const void*, int, int) { return 0; }
int cudaLaunchKernelExC(const void*, const void*, void**) { return 0; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t) { *n = 4; return 0; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
    *n = 4;
    return 0;
}
int cudaGetSymbolAddress(void** p, const void*) { *p = nullptr; return 1; }
int cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long, int* q) {
    *f = nullptr;
    *q = 1;
    return 1;
}
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, void*, void*, void*, void*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(Dim3, Dim3, size_t, void*) { return 0; }
int __cudaPopCallConfiguration(Dim3* g, Dim3* b, size_t* n, void* s) {
    *g = *b = Dim3{1, 1, 1};
    *n = 0;
    *static_cast<void**>(s) = nullptr;
    return 0;
}
int __cudaGetKernel(void** k, const void* f) { *k = const_cast<void*>(f); return 0; }
int __cudaLaunchKernel(void*, Dim3, Dim3, void**, size_t, void*) { return 0; }

int cublasCreate_v2(void** h) { *h = &handle; return 0; }
int cublasDestroy_v2(void*) { return 0; }
int cublasSetStream_v2(void*, void*) { return 0; }
int cublasCgemm_v2(...) { return 0; }
int cublasZherk_v2(...) { return 0; }
int cusolverDnCreate(void** h) { *h = &handle; return 0; }
int cusolverDnDestroy(void*) { return 0; }
int cusolverDnSetStream(void*, void*) { return 0; }
int cusolverDnZheevd(...) { return 0; }
int cusolverDnZheevd_bufferSize(...) { return 1; }
}
