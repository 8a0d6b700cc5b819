// Two devices without a GPU: the parts of the CUDA runtime that the MLP's and
// the staged DIA kernel's launch code calls.  As on a GPU, a launch on a device
// fails while its dynamic shared memory is above the function's limit on that
// device.  The program runs both products on device 0, then on device 1.
#include <cuda_runtime_api.h>

#include <cstdio>
#include <cstring>
#include <map>
#include <utility>

#include "smat_internal.h"

static int g_device = 0, g_launches = 0;
static std::map<std::pair<int, const void *>, size_t> g_limit;

extern "C" {
cudaError_t cudaGetDevice(int *d) { *d = g_device; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448 : a == cudaDevAttrMultiProcessorCount ? 152 : 0;
  return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *a, const void *) { std::memset(a, 0, sizeof(*a)); return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute, int v) { g_limit[{g_device, f}] = (size_t)v; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaMemcpyFromSymbol(void *, const void *, size_t, size_t, cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **) {
  const auto it = g_limit.find({g_device, f});
  if (c->dynamicSmemBytes > (it == g_limit.end() ? (size_t)48 * 1024 : it->second)) {
    std::printf("device %d: %zu bytes of shared memory refused\n", g_device, c->dynamicSmemBytes);
    return cudaErrorInvalidValue;
  }
  ++g_launches;
  return cudaSuccess;
}
// registration of the kernels in the object files
void **__cudaRegisterFatBinary(void *) { static void *p; return &p; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, void *, void *, void *, void *, int *) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
int __cudaPopCallConfiguration(void *, void *, void *, void *) { return 0; }
int __cudaLaunchKernel(const void *, int, int, void **, size_t, void *) { return 0; }
int __cudaGetKernel(void **, const void *) { return 0; }
}

int main() {
  alignas(256) static float buf[1 << 16];
  smat_s h;
  h.m = h.n = 100000;
  h.P = h.m;
  h.dtype = SMAT_F64;
  h.esz = 8;
  h.dia_nd = 5;
  h.dia_val = buf;
  h.dia_off = (int32_t *)buf;
  const double one = 1.0, zero = 0.0;
  int bad = 0;
  for (g_device = 0; g_device < 2; ++g_device) {
    if (smat_mlp_loss_grad(buf, buf, buf, 32, buf, buf, buf, nullptr) != SMAT_OK) bad |= 1;
    if (smat::launch_mlp_forward(buf, buf, 32, buf, nullptr) != cudaSuccess) bad |= 2;
    const int before = g_launches;
    for (int k = 1; k <= smat::dia_staged_kernels(); ++k)
      smat::launch_dia_staged(&h, k, &one, buf, &zero, buf, nullptr);
    if (g_launches != before + smat::dia_staged_kernels()) bad |= 4;
  }
  std::printf("bad %d launches %d\n", bad, g_launches);
  return bad;
}
