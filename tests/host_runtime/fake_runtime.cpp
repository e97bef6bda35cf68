// A CUDA runtime for host tests: the library's own object files linked against it run every host path (allocation,
// copies, launches, synchronisation, error returns) without a GPU.  Kernels do nothing, device memory is host memory;
// calls fail where a test asks, and what is still queued on a stream is counted.
#include <cuda.h>
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

#include "modal_internal.cuh"


namespace {
std::map<const void*, std::string> names;   // host stub -> kernel
int fail_alloc = 0, fail_copy = 0;           // every allocation; the fail_copy-th asynchronous copy from now
long long pending = 0, live = 0;             // operations queued since the last wait; temporaries held
void queued() { ++pending; }
dim3 launch_grid;
struct Tiles {                               // an encoded tensor map of two dimensions
    long long base, cols, rows, pitch;
};
std::vector<Tiles> encoded;
struct Job {                                 // the second argument of k_cubic
    double* partial;
    int64_t npix, ppc;
    int nctas;
    int64_t nunits;
};
std::vector<long long> cubic_log;            // per launch of k_cubic: its two tensor maps and its job
CUresult encode(CUtensorMap*, CUtensorMapDataType, cuuint32_t rank, void* base, const cuuint64_t* dims, const cuuint64_t* strides,
                const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                CUtensorMapFloatOOBfill) {
    if (rank == 2) encoded.push_back({(long long)base, (long long)dims[0], (long long)dims[1], (long long)strides[0]});
    return CUDA_SUCCESS;
}
cudaError_t allocate(void** p, size_t n) {
    *p = nullptr;
    if (fail_alloc) return cudaErrorMemoryAllocation;
    *p = std::calloc(n ? n : 1, 1);
    return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
}  // namespace

extern "C" {
// what a test sets and reads
void fake_fail_alloc(int on) { fail_alloc = on; }
void fake_fail_copy(int nth) { fail_copy = nth; }
long long fake_pending() { return pending; }
long long fake_live() { return live; }
// The launches of the cubic sums of B maps at address `maps` (weights W, partial sums at `partial`): twelve values each into out.
int fake_cubic(long long npix, int P, int B, int ctas, long long maps, long long W, long long partial, long long* out, int max) {
    modal::Plan pl;
    pl.P = P;
    pl.npix = npix;
    pl.n_max = P * (P + 1) * (P + 2) / 6;
    pl.cubic_ctas = ctas;
    pl.cubic_groups = 1;
    pl.cubic_boxes = 1;
    pl.nsm = 152;
    pl.W = reinterpret_cast<float*>(W);
    cubic_log.clear();
    if (modal::launch_cubic(pl, reinterpret_cast<const float*>(maps), B, reinterpret_cast<double*>(partial), nullptr) != cudaSuccess) return -1;
    for (size_t i = 0; i < cubic_log.size() && i < (size_t)max; ++i) out[i] = cubic_log[i];
    return (int)cubic_log.size() / 12;
}

// registration and launches
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) { names[host] = name; }
unsigned __cudaPushCallConfiguration(dim3 grid, dim3, size_t, cudaStream_t) { launch_grid = grid; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3*, size_t*, void*) { *grid = launch_grid; return cudaSuccess; }
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* host) { *k = (cudaKernel_t)host; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3, void** args, size_t, cudaStream_t) {
    queued();
    if (names[k].find("7k_cubicILb") != std::string::npos && encoded.size() >= 2) {
        const Tiles &m = encoded[encoded.size() - 2], &w = encoded.back();
        const Job& j = *static_cast<const Job*>(args[1]);
        for (long long v : {m.base, m.cols, m.rows, m.pitch, w.base, w.cols, (long long)j.partial, (long long)j.npix, (long long)j.ppc,
                            (long long)j.nctas, (long long)j.nunits, (long long)grid.x})
            cubic_log.push_back(v);
    }
    return cudaSuccess;
}

cudaError_t cudaMalloc(void** p, size_t n) { return allocate(p, n); }
cudaError_t cudaFree(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { const cudaError_t e = allocate(p, n); live += e == cudaSuccess; return e; }
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { live -= p != nullptr; std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { std::memmove(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
    if (fail_copy > 0 && --fail_copy == 0) return cudaErrorInvalidValue;
    queued();
    std::memmove(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemset(void* d, int v, size_t n) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { queued(); std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { pending = 0; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { pending = 0; return cudaSuccess; }
cudaError_t cudaMemGetInfo(size_t* f, size_t* t) { *f = *t = (size_t)280 << 30; return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "failed on request"; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) { *p = nullptr; return cudaErrorInvalidValue; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** p, unsigned, unsigned long long, cudaDriverEntryPointQueryResult* q) {
    *p = (void*)&encode;
    *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}

// events, streams and graphs: nothing to do
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 0.f; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = nullptr; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaErrorNotSupported; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t*) { return cudaErrorNotSupported; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t*, cudaGraph_t, unsigned long long) { return cudaErrorNotSupported; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaErrorNotSupported; }
}
