// A CUDA runtime without GPUs, for host-side tests of the launch sequences: device
// memory is host memory, kernels do not run, and a launch checks what the real one
// does: dynamic shared memory beyond 48 KB must have been allowed for this kernel on
// the current device.  Two devices.
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <utility>

namespace {
int device = 0, launches = 0;
cudaError_t last = cudaSuccess;
std::map<std::pair<int, const void *>, int> allowed;
cudaError_t launch(const void *f, size_t smem) {
  auto it = allowed.find({device, f});
  if (smem > 48 * 1024 && (it == allowed.end() || (size_t)it->second < smem))
    return last = cudaErrorInvalidValue;
  ++launches;
  return cudaSuccess;
}
}  // namespace

extern "C" {
void fake_set_device(int d) { device = d; }
int fake_launches() { return launches; }

void **__cudaRegisterFatBinary(void *) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, void *, void *, void *,
                            void *, int *) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
struct Call {
  dim3 grid, block;
  size_t smem;
  void *stream;
} pending;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, void *s) {
  pending = {g, b, smem, s};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *smem, void *s) {
  *g = pending.grid, *b = pending.block, *smem = pending.smem;
  *static_cast<void **>(s) = pending.stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void **, size_t smem, cudaStream_t) {
  return launch((const void *)k, smem);
}
cudaError_t cudaLaunchKernel(const void *f, dim3, dim3, void **, size_t smem, cudaStream_t) {
  return launch(f, smem);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **) {
  return launch(f, c->dynamicSmemBytes);
}
cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute, int v) {
  allowed[{device, f}] = v;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() {
  const cudaError_t e = last;
  last = cudaSuccess;
  return e;
}
cudaError_t cudaGetDevice(int *d) { return *d = device, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMalloc(void **p, size_t n) {
  *p = std::calloc(n ? n : 1, 1);
  return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaFree(void *p) { return std::free(p), cudaSuccess; }
cudaError_t cudaMemset(void *p, int v, size_t n) { return std::memset(p, v, n), cudaSuccess; }
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t) { return cudaMemset(p, v, n); }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) {
  return std::memmove(d, s, n), cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind k, cudaStream_t) {
  return cudaMemcpy(d, s, n, k);
}
cudaError_t cudaGetSymbolAddress(void **p, const void *) { return *p = nullptr, cudaSuccess; }
int cufftPlanMany(int *plan, int, int *, int *, int, int, int *, int, int, int, int) {
  return *plan = 1, 0;
}
int cufftSetStream(int, void *) { return 0; }
int cufftExecR2C(int, void *, void *) { return 0; }
int cufftDestroy(int) { return 0; }
}
