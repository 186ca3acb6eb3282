// A stand-in for the CUDA runtime, for tests of the library's host code without a device: the library's
// objects are linked against it.  "Device" memory is host memory counted against a limit, copies are made
// at once, kernels are not run: a launch is recorded by the kernel's name.  Memory pools keep what is freed
// until the next synchronisation and then release what is above their threshold, as documented.
#include <cuda_runtime_api.h>

#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

namespace {
struct Block { size_t bytes; bool pooled; };
std::map<char *, Block> blocks;
std::map<void *, size_t> arrays;
std::map<const void *, std::string> kernels;
std::vector<std::string> launches;
size_t limit = ~size_t(0), used = 0, idle = 0, threshold = 0;
int surf_calls = 0, surf_fail = -1, surf_error = 0;
dim3 cfg_grid, cfg_block;
size_t cfg_smem;
void *cfg_stream;
int handle;                                  // what any opaque handle points at
cudaError_t last = cudaSuccess;

cudaError_t ret(cudaError_t e) { if (e != cudaSuccess) last = e; return e; }
void sync() { if (idle > threshold) idle = threshold; }
cudaError_t take(void **p, size_t n, bool pooled) {
    size_t have = pooled ? (idle < n ? idle : n) : 0;
    if (used + idle + (n - have) > limit) return ret(cudaErrorMemoryAllocation);
    idle -= have;
    used += n;
    *p = std::calloc(n ? n : 1, 1);
    blocks[static_cast<char *>(*p)] = Block{n, pooled};
    return cudaSuccess;
}
cudaError_t drop(void *p) {
    if (!p) return cudaSuccess;
    auto it = blocks.find(static_cast<char *>(p));
    if (it == blocks.end()) return ret(cudaErrorInvalidValue);
    used -= it->second.bytes;
    if (it->second.pooled) idle += it->second.bytes;
    blocks.erase(it);
    std::free(p);
    return cudaSuccess;
}
template <typename T> cudaError_t opaque(T *h) { *h = reinterpret_cast<T>(&handle); return cudaSuccess; }
cudaError_t launch(const void *f) { launches.push_back(kernels[f]); return cudaSuccess; }
// the driver's query of the allocation that an address lies in
int address_range(unsigned long long *base, size_t *size, unsigned long long p) {
    for (auto &b : blocks)
        if (reinterpret_cast<char *>(p) >= b.first && reinterpret_cast<char *>(p) < b.first + b.second.bytes) {
            *base = reinterpret_cast<unsigned long long>(b.first);
            *size = b.second.bytes;
            return 0;
        }
    return 1;
}
}  // namespace

#define API extern "C" __attribute__((visibility("default")))
// ---- what the tests ask for
API void fake_reset() { last = cudaSuccess; launches.clear(); limit = ~size_t(0); surf_calls = 0; surf_fail = -1; }
API void fake_limit(size_t bytes) { limit = bytes; }
API size_t fake_reserved() { return used + idle; }
API int fake_arrays() { return (int)arrays.size(); }
API int fake_surface_arrays_made() { return surf_calls; }
API void fake_fail_surface_array(int nth, int error) { surf_calls = 0; surf_fail = nth; surf_error = error; }
API void *fake_device_alloc(size_t n) { void *p = nullptr; take(&p, n, false); return p; }
API const char *fake_launches() {
    static std::string s;
    s.clear();
    for (auto &l : launches) s += l + "\n";
    launches.clear();
    return s.c_str();
}
// ---- memory
API cudaError_t cudaMalloc(void **p, size_t n) { return take(p, n, false); }
API cudaError_t cudaFree(void *p) { sync(); return drop(p); }
API cudaError_t cudaMallocHost(void **p, size_t n) { *p = std::malloc(n); return cudaSuccess; }
API cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { *p = std::malloc(n); return cudaSuccess; }
API cudaError_t cudaFreeHost(void *p) { std::free(p); return cudaSuccess; }
API cudaError_t cudaHostRegister(void *, size_t, unsigned) { return cudaSuccess; }
API cudaError_t cudaMemPoolCreate(cudaMemPool_t *p, const cudaMemPoolProps *) { return opaque(p); }
API cudaError_t cudaMemPoolDestroy(cudaMemPool_t) { idle = 0; return cudaSuccess; }
API cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *v) { threshold = *static_cast<uint64_t *>(v); return cudaSuccess; }
API cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t keep) { if (idle > keep) idle = keep; return cudaSuccess; }
API cudaError_t cudaMallocFromPoolAsync(void **p, size_t n, cudaMemPool_t, cudaStream_t) { return take(p, n, true); }
API cudaError_t cudaFreeAsync(void *p, cudaStream_t) { return drop(p); }
API cudaError_t cudaMallocArray(cudaArray_t *a, const cudaChannelFormatDesc *d, size_t w, size_t h, unsigned flags) {
    if ((flags & cudaArraySurfaceLoadStore) && surf_calls++ == surf_fail) return ret(static_cast<cudaError_t>(surf_error));
    const size_t n = w * h * ((d->x + d->y + d->z + d->w) / 8);
    if (used + idle + n > limit) return ret(cudaErrorMemoryAllocation);
    used += n;
    *a = static_cast<cudaArray_t>(std::malloc(1));
    arrays[*a] = n;
    return cudaSuccess;
}
API cudaError_t cudaFreeArray(cudaArray_t a) { used -= arrays[a]; arrays.erase(a); std::free(a); return cudaSuccess; }
API cudaChannelFormatDesc cudaCreateChannelDesc(int x, int y, int z, int w, cudaChannelFormatKind f) { return cudaChannelFormatDesc{x, y, z, w, f}; }
API cudaError_t cudaCreateSurfaceObject(cudaSurfaceObject_t *s, const cudaResourceDesc *) { *s = 7; return cudaSuccess; }
API cudaError_t cudaCreateTextureObject(cudaTextureObject_t *t, const cudaResourceDesc *, const cudaTextureDesc *, const cudaResourceViewDesc *) { *t = 9; return cudaSuccess; }
API cudaError_t cudaDestroySurfaceObject(cudaSurfaceObject_t) { return cudaSuccess; }
API cudaError_t cudaDestroyTextureObject(cudaTextureObject_t) { return cudaSuccess; }
API cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { std::memcpy(d, s, n); return cudaSuccess; }
API cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind k, cudaStream_t) {
    unsigned long long base;
    size_t size;
    launches.push_back("cudaMemcpyAsync");
    if (k == cudaMemcpyDeviceToDevice && !address_range(&base, &size, reinterpret_cast<unsigned long long>(s)) &&
        reinterpret_cast<unsigned long long>(s) + n > base + size)
        return ret(cudaErrorInvalidValue);
    std::memcpy(d, s, n);
    return cudaSuccess;
}
API cudaError_t cudaMemcpy3DAsync(const cudaMemcpy3DParms *, cudaStream_t) { launches.push_back("cudaMemcpy3DAsync"); return cudaSuccess; }
API cudaError_t cudaMemcpy2DToArrayAsync(cudaArray_t, size_t, size_t, const void *, size_t, size_t, size_t, cudaMemcpyKind, cudaStream_t) { launches.push_back("cudaMemcpy2DToArrayAsync"); return cudaSuccess; }
API cudaError_t cudaMemset(void *p, int v, size_t n) { std::memset(p, v, n); return cudaSuccess; }
API cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t) { return cudaSuccess; }
API cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *p) {
    unsigned long long base;
    size_t size;
    std::memset(a, 0, sizeof(*a));
    a->type = address_range(&base, &size, reinterpret_cast<unsigned long long>(p)) ? cudaMemoryTypeUnregistered : cudaMemoryTypeDevice;
    return cudaSuccess;
}
API cudaError_t cudaGetDriverEntryPointByVersion(const char *name, void **f, unsigned, unsigned long long, cudaDriverEntryPointQueryResult *r) {
    const bool known = !std::strcmp(name, "cuMemGetAddressRange");
    *f = known ? reinterpret_cast<void *>(&address_range) : nullptr;
    if (r) *r = known ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
    return cudaSuccess;
}
// ---- device, streams, events
API cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
API cudaError_t cudaSetDevice(int) { return cudaSuccess; }
API cudaError_t cudaGetDeviceCount(int *n) { *n = 1; return cudaSuccess; }
API cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMaxTexture2DGatherWidth || a == cudaDevAttrMaxTexture2DGatherHeight ? 32768
         : a == cudaDevAttrMaxSharedMemoryPerBlockOptin || a == cudaDevAttrMaxSharedMemoryPerMultiprocessor ? 227 << 10
         : a == cudaDevAttrMultiProcessorCount ? 152 : 1;
    return cudaSuccess;
}
API cudaError_t cudaDeviceSynchronize() { sync(); return cudaSuccess; }
API cudaError_t cudaStreamSynchronize(cudaStream_t) { sync(); return cudaSuccess; }
API cudaError_t cudaEventSynchronize(cudaEvent_t) { sync(); return cudaSuccess; }
API cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
API cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
API cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 0.0f; return cudaSuccess; }
API cudaError_t cudaEventCreate(cudaEvent_t *e) { return opaque(e); }
API cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return opaque(e); }
API cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
API cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { return opaque(s); }
API cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
API cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
API cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *c) { *c = cudaStreamCaptureStatusNone; return cudaSuccess; }
API cudaError_t cudaGetLastError() { const cudaError_t e = last; last = cudaSuccess; return e; }
API const char *cudaGetErrorName(cudaError_t) { return "error"; }
API const char *cudaGetErrorString(cudaError_t) { return "of the stand-in runtime"; }
API cudaError_t cudaGetSymbolAddress(void **, const void *) { return ret(cudaErrorInvalidSymbol); }
// ---- kernels
API cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *a, const void *) { std::memset(a, 0, sizeof(*a)); a->numRegs = 64; return cudaSuccess; }
API cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
API cudaError_t cudaLaunchKernel(const void *f, dim3, dim3, void **, size_t, cudaStream_t) { return launch(f); }
API cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *, const void *f, void **) { return launch(f); }
API cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void **, size_t, cudaStream_t) { return launch(reinterpret_cast<const void *>(k)); }
API cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) { *k = reinterpret_cast<cudaKernel_t>(const_cast<void *>(f)); return cudaSuccess; }
API unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t m, cudaStream_t s) { cfg_grid = g; cfg_block = b; cfg_smem = m; cfg_stream = s; return 0; }
API cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *m, void *s) { *g = cfg_grid; *b = cfg_block; *m = cfg_smem; *static_cast<void **>(s) = cfg_stream; return cudaSuccess; }
API void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
API void __cudaRegisterFatBinaryEnd(void **) {}
API void __cudaUnregisterFatBinary(void **) {}
API void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
API void __cudaRegisterFunction(void **, const char *f, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) { kernels[f] = name; }
