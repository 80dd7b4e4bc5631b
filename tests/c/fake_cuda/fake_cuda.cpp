#include "fake_cuda.h"

#include <cuda.h>
#include <cuda_runtime_api.h>

#include <cstring>
#include <map>
#include <utility>

namespace fake {
std::vector<Launch> launches;
std::vector<size_t> allocations;
std::vector<std::string> refuse;
bool launched(const char* part) {
  for (const Launch& l : launches)
    if (!l.refused && l.name.find(part) != std::string::npos) return true;
  return false;
}
}  // namespace fake

namespace {

constexpr int DEVICES = 2;
constexpr size_t SMEM_DEFAULT = 48 << 10, SMEM_MAX = 227 << 10;
int device = 0;
cudaError_t last = cudaSuccess;
std::map<const void*, std::string>& names() {
  static std::map<const void*, std::string> m;
  return m;
}
std::map<std::pair<int, const void*>, size_t> allowed;
char* next_address = reinterpret_cast<char*>(uintptr_t(1) << 40);
struct Config {
  dim3 grid, block;
  size_t smem;
  cudaStream_t stream;
} pushed;

cudaError_t set(cudaError_t e) {
  if (e != cudaSuccess) last = e;
  return e;
}

cudaError_t do_launch(const void* func, size_t smem, bool overlap = false) {
  const std::string& name = names()[func];
  const auto a = allowed.find({device, func});
  bool refused = smem > (a == allowed.end() ? SMEM_DEFAULT : a->second);
  for (const std::string& r : fake::refuse) refused |= name.find(r) != std::string::npos;
  fake::launches.push_back({name, device, smem, overlap, refused});
  return set(refused ? cudaErrorInvalidValue : cudaSuccess);
}

CUresult encode(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
  return CUDA_SUCCESS;
}

}  // namespace

extern "C" {

void** __cudaRegisterFatBinary(void*) {
  static void* handle;
  return &handle;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*,
                            dim3*, dim3*, int*) {
  names()[host] = name;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(f));
  return cudaSuccess;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, cudaStream_t s) {
  pushed = Config{g, b, smem, s};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* s) {
  *g = pushed.grid;
  *b = pushed.block;
  *smem = pushed.smem;
  *static_cast<cudaStream_t*>(s) = pushed.stream;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t smem, cudaStream_t) {
  return do_launch(reinterpret_cast<const void*>(k), smem);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* func, void**) {
  bool overlap = false;
  for (unsigned k = 0; k < c->numAttrs; ++k)
    overlap |= c->attrs[k].id == cudaLaunchAttributeProgrammaticStreamSerialization &&
               c->attrs[k].val.programmaticStreamSerializationAllowed;
  return do_launch(func, c->dynamicSmemBytes, overlap);
}
cudaError_t cudaFuncSetAttribute(const void* func, cudaFuncAttribute a, int v) {
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) {
    if (v < 0 || (size_t)v > SMEM_MAX) return set(cudaErrorInvalidValue);
    allowed[{device, func}] = (size_t)v;
  }
  return cudaSuccess;
}
cudaError_t cudaGetDeviceCount(int* n) {
  *n = DEVICES;
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) {
  *d = device;
  return cudaSuccess;
}
cudaError_t cudaSetDevice(int d) {
  if (d < 0 || d >= DEVICES) return set(cudaErrorInvalidDevice);
  device = d;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : 0;
  return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t bytes) {
  *p = next_address;
  next_address += (bytes + 511) / 512 * 512;
  fake::allocations.push_back(bytes);
  return cudaSuccess;
}
cudaError_t cudaFree(void*) { return cudaSuccess; }
cudaError_t cudaMemset(void*, int, size_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
// device memory reads as zeros
cudaError_t cudaMemcpy(void* dst, const void*, size_t n, cudaMemcpyKind k) {
  if (k == cudaMemcpyDeviceToHost) std::memset(dst, 0, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* dst, const void* src, size_t n, cudaMemcpyKind k, cudaStream_t) {
  return cudaMemcpy(dst, src, n, k);
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
  *p = reinterpret_cast<void*>((uintptr_t(1) << 36) * (device + 1));
  return cudaSuccess;
}
cudaError_t cudaGetLastError(void) {
  const cudaError_t e = last;
  last = cudaSuccess;
  return e;
}
cudaError_t cudaPeekAtLastError(void) { return last; }
const char* cudaGetErrorString(cudaError_t) { return "error"; }
cudaError_t cudaDeviceSynchronize(void) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  static uintptr_t n = 0x1000;
  *s = reinterpret_cast<cudaStream_t>(n += 16);
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* c) {
  *c = cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) {
  static uintptr_t n = 0x2000;
  *e = reinterpret_cast<cudaEvent_t>(n += 16);
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  *ms = 1.f;
  return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** p, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
  *p = reinterpret_cast<void*>(&encode);
  *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}

}  // extern "C"
