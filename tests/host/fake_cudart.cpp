// A stand-in for the CUDA runtime, linked with the library's own objects in place of the real one: the
// library's host code (checks, dispatch, launches) then runs without a GPU.  "Device" memory is host
// memory, nothing is computed, and every launch is recorded.  As the runtime does, it refuses a launch
// with more than 48 KB of dynamic shared memory that its kernel has not opted into on the current device.
#include "fake_cudart.h"

#include <cuda.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <map>

namespace fake {
int device = 0;
std::vector<Launch> launches;
std::function<bool(size_t)> alloc_fails = [](size_t) { return false; };
std::function<int(const std::string&)> registers = [](const std::string&) { return 168; };
std::function<int(int)> sms = [](int) { return 152; };

namespace {
std::map<const void*, std::string>& kernels() {
    static std::map<const void*, std::string> k;
    return k;
}
std::map<std::pair<int, const void*>, int> opted_in;      // dynamic shared memory, by device and kernel
cudaError_t last = cudaSuccess;
struct Config {
    dim3 grid, block;
    size_t smem;
    cudaStream_t stream;
};
std::vector<Config> pushed;

cudaError_t answer(cudaError_t e) {
    if (e != cudaSuccess) last = e;
    return e;
}
int allowed(const void* fn) {
    const auto it = opted_in.find({device, fn});
    return it == opted_in.end() ? 48 * 1024 : it->second;
}
cudaError_t launch(const void* fn, dim3 grid, dim3 block, size_t smem) {
    if (smem > (size_t)allowed(fn)) return answer(cudaErrorInvalidValue);
    launches.push_back({device, kernels()[fn], grid, block, smem});
    return cudaSuccess;
}
cudaError_t allocate(void** p, size_t bytes) {
    *p = nullptr;
    if (alloc_fails(bytes)) return answer(cudaErrorMemoryAllocation);
    *p = std::aligned_alloc(256, (bytes + 511) / 256 * 256);
    return cudaSuccess;
}
template <class T>
cudaError_t handle(T* out) {
    static char any[64];
    *out = reinterpret_cast<T>(any);
    return cudaSuccess;
}
CUresult encode_tiled(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                      const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                      CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
    return CUDA_SUCCESS;
}
}  // namespace

std::vector<std::string> kernel_names() {
    std::vector<std::string> names;
    for (const auto& k : kernels()) names.push_back(k.second);
    return names;
}
bool launched(const std::string& part) {
    for (const Launch& l : launches)
        if (l.kernel.find(part) != std::string::npos) return true;
    return false;
}
}  // namespace fake

using namespace fake;

extern "C" {
void** __cudaRegisterFatBinary(void*) {
    static void* any;
    return &any;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
    kernels()[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* fn) {
    *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(fn));
    return cudaSuccess;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, cudaStream_t s) {
    pushed.push_back({grid, block, smem, s});
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* s) {
    const Config c = pushed.back();
    pushed.pop_back();
    *grid = c.grid;
    *block = c.block;
    *smem = c.smem;
    *static_cast<cudaStream_t*>(s) = c.stream;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3 block, void**, size_t smem, cudaStream_t) {
    return launch(reinterpret_cast<const void*>(k), grid, block, smem);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* fn, void**) {
    return launch(fn, c->gridDim, c->blockDim, c->dynamicSmemBytes);
}
cudaError_t cudaFuncSetAttribute(const void* fn, cudaFuncAttribute a, int value) {
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) opted_in[{device, fn}] = value;
    return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void* fn) {
    *a = cudaFuncAttributes{};
    a->numRegs = registers(kernels()[fn]);
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void* fn, int, size_t smem) {
    *n = smem > (size_t)allowed(fn) ? 0 : (int)std::max<size_t>(1, 227 * 1024 / (smem + 1024));
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void* fn, const cudaLaunchConfig_t* c) {
    int blocks = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, fn, 0, c->dynamicSmemBytes);
    *n = sms(device) * blocks / (int)c->attrs[0].val.clusterDim.x;
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) {
    *d = device;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int d) {
    *v = a == cudaDevAttrMultiProcessorCount ? sms(d) : 1;
    return cudaSuccess;
}
cudaError_t cudaGetLastError() {
    const cudaError_t e = last;
    last = cudaSuccess;
    return e;
}
const char* cudaGetErrorString(cudaError_t) { return "fake runtime error"; }
cudaError_t cudaGetDriverEntryPointByVersion(const char* name, void** fn, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* r) {
    const bool known = std::strcmp(name, "cuTensorMapEncodeTiled") == 0;
    *fn = known ? reinterpret_cast<void*>(&encode_tiled) : nullptr;
    *r = known ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
    static char any[256];
    *p = any;
    return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
    *a = cudaPointerAttributes{};
    a->type = cudaMemoryTypeDevice;
    a->devicePointer = const_cast<void*>(p);
    return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t bytes) { return allocate(p, bytes); }
cudaError_t cudaFree(void* p) {
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaMallocFromPoolAsync(void** p, size_t bytes, cudaMemPool_t, cudaStream_t) { return allocate(p, bytes); }
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { return cudaFree(p); }
cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps*) { return handle(p); }
cudaError_t cudaMemPoolDestroy(cudaMemPool_t) { return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaMemcpy(void*, const void*, size_t, cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemcpy2DAsync(void*, size_t, const void*, size_t, size_t, size_t, cudaMemcpyKind, cudaStream_t) {
    return cudaSuccess;
}
cudaError_t cudaMemset(void*, int, size_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return handle(s); }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return handle(e); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return handle(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
    *ms = 0.f;
    return cudaSuccess;
}
}
