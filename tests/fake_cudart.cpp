// A CUDA runtime of two imaginary devices, linked with the library's objects
// in place of the real one: device memory is addresses that nothing reads,
// copies and launches do nothing.  As on a device, a launch that asks for more
// than 48 KB of dynamic shared memory is refused unless its kernel was given
// that much on the current device.  test_launch_forms.py reads the record.
#include <cuda_runtime_api.h>

#include <cstdint>
#include <cstdlib>
#include <map>
#include <utility>

#include "kernels.h"
#include "solver.h"

namespace {
int dev = 0;
const int kSms[2] = {152, 148};
std::map<std::pair<int, const void *>, int> opt_in;
long launches = 0, refused = 0;
unsigned last_grid = 0;
uintptr_t next_mem = (uintptr_t)1 << 40;

cudaError_t launched(const void *f, unsigned grid, size_t smem) {
  if (smem > 48 * 1024) {
    auto it = opt_in.find({dev, f});
    if (it == opt_in.end() || (size_t)it->second < smem) {
      ++refused;
      return cudaErrorInvalidValue;
    }
  }
  ++launches;
  last_grid = grid;
  return cudaSuccess;
}
cudaError_t any_handle(void **p) {
  *p = (void *)(next_mem += 256);
  return cudaSuccess;
}
}  // namespace

extern "C" {
long fake_launches() { return launches; }
long fake_refused() { return refused; }
unsigned fake_last_grid() { return last_grid; }
// launch_hop_dw_cg, launch_hop_dw_r and the fused low-precision hop on vh sites per parity
int fake_launch_cg(int which, int64_t vh) {
  using namespace jqcd;
  HopParams P = {};
  P.g.nxh = P.g.nx = P.g.ny = P.g.nz = P.g.nt = 2;
  P.g.vh = vh;
  switch (which) {
    case 0: return launch_hop_dw_cg(P, nullptr, nullptr, nullptr, nullptr, nullptr);
    case 1: return launch_hop_dw_r(P, nullptr, nullptr, nullptr, nullptr);
    case 2: return launch_hop_lp_cg(PREC_F32, P, nullptr, nullptr, nullptr);
    default: return launch_hop_lp_cg(PREC_F16N, P, nullptr, nullptr, nullptr);
  }
}

cudaError_t cudaGetDevice(int *d) { *d = dev; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { dev = d; return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int *n) { *n = 2; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int d) {
  *v = a == cudaDevAttrMultiProcessorCount ? kSms[d] : 0;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute, int v) {
  opt_in[{dev, f}] = v;
  return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **) {
  return launched(f, c->gridDim.x, c->dynamicSmemBytes);
}
static struct { dim3 grid, block; size_t smem; cudaStream_t s; } pushed;
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, cudaStream_t s) {
  pushed = {grid, block, smem, s};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *s) {
  *grid = pushed.grid;
  *block = pushed.block;
  *smem = pushed.smem;
  *(cudaStream_t *)s = pushed.s;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3, void **, size_t smem, cudaStream_t) {
  return launched((const void *)k, grid.x, smem);
}
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, void *, void *, dim3 *, dim3 *, int *) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}

cudaError_t cudaMalloc(void **p, size_t n) {
  *p = (void *)next_mem;
  next_mem += (n + 255) / 256 * 256;
  return cudaSuccess;
}
cudaError_t cudaFree(void *) { return cudaSuccess; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { *p = calloc(1, n); return cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void **p, const void *) { return any_handle(p); }
cudaError_t cudaMemcpyAsync(void *, const void *, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "refused by the fake runtime"; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { return any_handle((void **)s); }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { return any_handle((void **)e); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return any_handle((void **)e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }

// not used by the calls under test
#define ABSENT { return cudaErrorNotSupported; }
cudaError_t cudaDeviceGetStreamPriorityRange(int *, int *) ABSENT
cudaError_t cudaEventElapsedTime(float *, cudaEvent_t, cudaEvent_t) ABSENT
cudaError_t cudaEventQuery(cudaEvent_t) ABSENT
cudaError_t cudaEventSynchronize(cudaEvent_t) ABSENT
cudaError_t cudaGraphDestroy(cudaGraph_t) ABSENT
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) ABSENT
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *, cudaGraph_t, unsigned long long) ABSENT
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) ABSENT
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *, const void *, int, size_t, unsigned) ABSENT
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *, const void *) ABSENT
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) ABSENT
cudaError_t cudaStreamCreateWithPriority(cudaStream_t *, unsigned, int) ABSENT
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *) ABSENT
}  // extern "C"
