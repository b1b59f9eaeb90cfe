// A CUDA runtime without a GPU: memory is host memory, kernels are counted and not run, and the
// calls that a test names fail with an error code. Linked with the library's own objects, it runs
// the host side of every entry point on the CPU (tests/_fake_cuda.py). As on a device, a launch fails
// that asks for more than 48 KB of dynamic shared memory without the attribute having been set for
// the kernel on the device that is current.
#include <cuda.h>
#include <cuda_runtime_api.h>
#include <stdlib.h>
#include <string.h>

#include <map>
#include <string>
#include <utility>

#include "common.cuh"

typedef struct CUkern_st* Kernel;

namespace {
struct State {
    int dev = 0;
    std::map<std::pair<int, const void*>, int> smem;  // (device, kernel) -> attribute
    std::map<const void*, std::string> name;
    std::map<std::string, long> launches;
    std::string fail_name;
    long fail_after = 0;
    bool fail_encode = false;
    size_t limit = ~size_t(0), largest = 0;
    std::map<const char*, size_t> blocks;  // of cudaMallocAsync
    long outside = 0;                      // digit cuts and tensor maps that leave their block
    cudaError_t last = cudaSuccess;
    dim3 grid, block;
    size_t dyn = 0;
    cudaStream_t st = nullptr;
};
State& s() {
    static State* x = new State;  // registration runs before this file's own initialisers
    return *x;
}
cudaError_t note(cudaError_t e) {
    if (e != cudaSuccess) s().last = e;
    return e;
}
// [p, p + n) lies in one block
void check(const void* p, size_t n) {
    auto it = s().blocks.upper_bound((const char*)p);
    if (it == s().blocks.begin() || (const char*)p + n > (--it)->first + it->second) ++s().outside;
}
// the digit planes and exponents of `rows` rows of K values
void check_digits(const void* d, const void* e, size_t rows, size_t K) {
    check(d, (K + 127) / 128 * 8 * rows * 128 * 2);
    check(e, rows * 4);
}
CUresult encode(CUtensorMap*, CUtensorMapDataType type, cuuint32_t rank, void* base, const cuuint64_t* dims,
                const cuuint64_t* strides, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
    size_t n = dims[0] * (type == CU_TENSOR_MAP_DATA_TYPE_FLOAT32 ? 4 : 2);
    for (cuuint32_t i = 1; i < rank; ++i) n += (dims[i] - 1) * strides[i - 1];
    check(base, n);
    return s().fail_encode ? CUDA_ERROR_INVALID_VALUE : CUDA_SUCCESS;
}
}  // namespace

extern "C" {
// ---- the tests' side ----
void fake_reset() {
    s().launches.clear();
    s().fail_name.clear();
    s().fail_encode = false;
    s().limit = ~size_t(0);
    s().largest = 0;
    s().outside = 0;
    s().last = cudaSuccess;
    s().dev = 0;
}
void fake_device(int d) { s().dev = d; }
void fake_fail_launch(const char* name, long after) {  // launches of such kernels fail after `after` good ones
    s().fail_name = name;
    s().fail_after = after;
}
void fake_fail_encode(int on) { s().fail_encode = on; }
void fake_alloc_limit(size_t bytes) { s().limit = bytes; }
size_t fake_largest_alloc() { return s().largest; }  // of those that succeeded
long fake_outside() { return s().outside; }
long fake_launches(const char* name) {
    long n = 0;
    for (auto& k : s().launches)
        if (k.first.find(name) != std::string::npos) n += k.second;
    return n;
}

const char* fake_launched(int i) {  // name of the i-th kernel launched so far, null past the last
    for (auto& k : s().launches)
        if (i-- == 0) return k.first.c_str();
    return nullptr;
}

// ---- registration and launches ----
void** __cudaRegisterFatBinary(void*) {
    static void* h;
    return &h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
char __cudaInitModule(void**) { return 1; }
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterManagedVar(void**, void** host, char*, const char*, int, size_t size, int, int) {
    *host = calloc(1, size);
}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, void*, void*, void*, void*,
                            int*) {
    s().name[host] = name;
}
cudaError_t __cudaGetKernel(Kernel* k, const void* f) {
    *k = (Kernel)f;
    return cudaSuccess;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t dyn, cudaStream_t st) {
    s().grid = g;
    s().block = b;
    s().dyn = dyn;
    s().st = st;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* dyn, void* st) {
    *g = s().grid;
    *b = s().block;
    *dyn = s().dyn;
    *(cudaStream_t*)st = s().st;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(Kernel k, dim3 g, dim3 b, void** a, size_t dyn, cudaStream_t) {
    const std::string& n = s().name[k];
    if (!g.x || !g.y || !g.z || !b.x || g.y > 65535 || g.z > 65535 || b.x * b.y * b.z > 1024)
        return note(cudaErrorInvalidConfiguration);
    auto it = s().smem.find({s().dev, k});
    if (dyn > 48 * 1024 && (it == s().smem.end() || dyn > (size_t)it->second)) return note(cudaErrorInvalidValue);
    if (!s().fail_name.empty() && n.find(s().fail_name) != std::string::npos && s().fail_after-- <= 0)
        return note(cudaErrorLaunchOutOfResources);
    ++s().launches[n];
    auto num = [&](int i) { return (size_t) * (int*)a[i]; };
    auto ptr = [&](int i) { return *(void**)a[i]; };
    if (n.find("k_oz_split_rows") != std::string::npos) check_digits(ptr(4), ptr(5), num(2), num(3));
    if (n.find("k_oz_split_cols") != std::string::npos) check_digits(ptr(6), ptr(7), num(5), num(4));
    if (n.find("k_oz_split_ldl") != std::string::npos) {
        check_digits(ptr(7), ptr(8), num(2), num(4));
        check_digits(ptr(9), ptr(10), num(3), num(4));
    }
    return cudaSuccess;
}

// ---- devices, attributes, errors ----
cudaError_t cudaGetDevice(int* d) {
    *d = s().dev;
    return cudaSuccess;
}
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) {
    memset(p, 0, sizeof *p);
    p->major = 10;
    p->minor = 3;
    p->multiProcessorCount = 152;
    p->sharedMemPerBlockOptin = 232448;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) {
    *v = 152;
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute, int v) {
    s().smem[{s().dev, f}] = v;
    return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
    *f = (void*)encode;
    *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
cudaError_t cudaGetLastError() {
    const cudaError_t e = s().last;
    s().last = cudaSuccess;
    return e;
}
const char* cudaGetErrorString(cudaError_t) { return "failed on request"; }

// ---- memory ----
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) {
    if (n > s().limit) return note(cudaErrorMemoryAllocation);
    if (n > s().largest) s().largest = n;
    *p = calloc(1, n);
    if (!*p) return note(cudaErrorMemoryAllocation);
    s().blocks[(const char*)*p] = n;
    return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t n) {
    *p = calloc(1, n);
    return cudaSuccess;
}
cudaError_t cudaMallocHost(void** p, size_t n) { return cudaMalloc(p, n); }
cudaError_t cudaFreeAsync(void* p, cudaStream_t) {
    s().blocks.erase((const char*)p);
    free(p);
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) { return cudaFreeAsync(p, nullptr); }
cudaError_t cudaMemcpy(void* d, const void* a, size_t n, cudaMemcpyKind kind) {
    memcpy(d, a, n);
    // a run's scalars: ||G||^2, which no kernel has formed, is 1
    if (kind == cudaMemcpyDeviceToHost && n == sizeof(thc::DevScalars)) ((thc::DevScalars*)d)->normG2 = 1.0;
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* a, size_t n, cudaMemcpyKind k, cudaStream_t) {
    return cudaMemcpy(d, a, n, k);
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
    memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaMemset2DAsync(void* d, size_t pitch, int v, size_t w, size_t h, cudaStream_t) {
    for (size_t i = 0; i < h; ++i) memset((char*)d + i * pitch, v, w);
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
    static char block[1 << 20];
    *p = block;
    return cudaSuccess;
}

// ---- streams, events, graphs: everything has run when it is asked for ----
cudaError_t cudaEventCreate(cudaEvent_t* e) {
    *e = (cudaEvent_t)1;
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* t, cudaEvent_t, cudaEvent_t) {
    *t = 1.0f;
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
    *e = (cudaGraphExec_t)1;
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
    *g = (cudaGraph_t)1;
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* st, unsigned) {
    *st = (cudaStream_t)1;
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* c) {
    *c = cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
}
