// A CUDA runtime without a GPU, for tests of the host side: the library's objects are linked against it
// instead of the real one.  "Device" memory is host memory, a kernel launch does nothing but check its
// dynamic shared memory against the kernel's attribute on the current device (48 KB unless raised, as on
// real devices a setting of each device) and note the kernel's name.
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <utility>

namespace {
std::map<const void *, std::string> &kernels() {
  static std::map<const void *, std::string> m;
  return m;
}
std::map<std::pair<int, const void *>, int> shared_limit;
std::string launched;                 // names of the kernels launched, one a line
int device = 0;
int allocations_left = -1;            // -1: never fails
std::string gives_up;                 // a launch of a kernel of this name runs out of its bounded waits ...
bool gave_up = false;                 // ... and leaves 2 in the context's flag, the one int the host reads
cudaError_t last = cudaSuccess;
struct { dim3 grid, block; size_t smem; cudaStream_t st; } pushed;

cudaError_t launch(const void *f, size_t smem) {
  auto it = shared_limit.find({device, f});
  const size_t limit = it == shared_limit.end() ? 48 * 1024 : (size_t)it->second;
  if (smem > limit) return last = cudaErrorInvalidValue;
  launched += kernels()[f] + "\n";
  if (!gives_up.empty() && kernels()[f].find(gives_up) != std::string::npos) gave_up = true;
  return cudaSuccess;
}

// cuTensorMapEncodeTiled: its checks of the base address and the strides
CUresult CUDAAPI encode(CUtensorMap *, CUtensorMapDataType, cuuint32_t rank, void *base, const cuuint64_t *,
                        const cuuint64_t *stride, const cuuint32_t *, const cuuint32_t *,
                        CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                        CUtensorMapFloatOOBfill) {
  if ((uintptr_t)base % 16) return CUDA_ERROR_INVALID_VALUE;
  for (cuuint32_t i = 0; i + 1 < rank; ++i)
    if (stride[i] % 16) return CUDA_ERROR_INVALID_VALUE;
  return CUDA_SUCCESS;
}
}  // namespace

extern "C" {

// what the tests set and read
void fake_set_device(int d) { device = d; }
void fake_fail_allocation(int after) { allocations_left = after; }
const char *fake_launched() { return launched.c_str(); }
void fake_clear() { launched.clear(); }
void fake_give_up(const char *kernel) { gives_up = kernel; gave_up = false; }

// registration and <<<>>>
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *,
                            dim3 *, dim3 *, int *) {
  kernels()[host] = name;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, struct CUstream_st *st) {
  pushed.grid = g; pushed.block = b; pushed.smem = smem; pushed.st = st;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *smem, void *st) {
  *g = pushed.grid; *b = pushed.block; *smem = pushed.smem;
  *(cudaStream_t *)st = pushed.st;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void **, size_t smem, cudaStream_t) {
  return launch((const void *)k, smem);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **) {
  return launch(f, c->dynamicSmemBytes);
}

// devices and attributes
cudaError_t cudaGetDevice(int *d) { *d = device; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute a, int v) {
  if (a != cudaFuncAttributeMaxDynamicSharedMemorySize || v > 227 * 1024) return last = cudaErrorInvalidValue;
  shared_limit[{device, f}] = v;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) {
  *n = 2;
  return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *q) {
  *f = (void *)encode;
  if (q) *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}

// memory and streams
cudaError_t cudaMallocAsync(void **p, size_t n, cudaStream_t) {
  if (allocations_left == 0) return last = cudaErrorMemoryAllocation;
  if (allocations_left > 0) --allocations_left;
  *p = aligned_alloc(256, (n + 255) / 256 * 256 + 256);
  return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaFreeAsync(void *p, cudaStream_t) { free(p); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind kind, cudaStream_t) {
  memmove(d, s, n);
  if (gave_up && kind == cudaMemcpyDeviceToHost && n == sizeof(int)) *(int *)d = 2;
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void **p, const void *s) { *p = const_cast<void *>(s); return cudaSuccess; }
cudaError_t cudaGetLastError() { cudaError_t e = last; last = cudaSuccess; return e; }
cudaError_t cudaPeekAtLastError() { return last; }
const char *cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "a fake error"; }

}  // extern "C"
