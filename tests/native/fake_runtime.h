// Stand-ins for the CUDA runtime's launch and attribute calls, for programs that
// call the library's launchers without a GPU (a program's own definitions come
// first at load time).  A launch with more dynamic shared memory than the kernel
// has been allowed on the current device is refused, as the runtime would.
#pragma once

#include <cuda_runtime.h>
#include <stdio.h>
#include <string.h>

#include <map>
#include <utility>
#include <vector>

#include "cem_internal.h"

namespace cem {
cudaError_t launch_step_fp64(const DevState &d, int cur, bool first, bool energy, const StepStreams &ss,
                             cudaEvent_t *marks);
cudaError_t launch_step_fp32(const DevState &d, int cur, bool first, bool energy, const StepStreams &ss,
                             cudaEvent_t *marks);
cudaError_t launch_step_fp64_batch(const BatchDev &b, bool first, bool energy, int grid_main,
                                   const StepStreams &ss);
cudaError_t launch_step_fp32_batch(const BatchDev &b, bool first, bool energy, int tile_rows,
                                   int grid_main, const StepStreams &ss);
void tile64_shape(int nx, int ny, int &tx, int &ty);
}  // namespace cem

struct Launch {
  const void *f;
  dim3 grid, block;
};
static std::vector<Launch> g_log;
static int g_device = 0, g_refused = 0;
static cudaError_t g_last = cudaSuccess;
static std::map<std::pair<int, const void *>, int> g_most, g_split;

static cudaError_t launched(const void *f, dim3 grid, dim3 block, size_t smem) {
  g_log.push_back(Launch{f, grid, block});
  auto it = g_most.find({g_device, f});
  const size_t most = it == g_most.end() ? 48 * 1024 : (size_t)it->second;
  if (smem <= most) return cudaSuccess;
  printf("device %d: %zu bytes of dynamic shared memory, %zu allowed\n", g_device, smem, most);
  ++g_refused;
  return g_last = cudaErrorInvalidValue;
}

extern "C" {
cudaError_t cudaGetDevice(int *d) {
  *d = g_device;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute a, int v) {
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) g_most[{g_device, f}] = v;
  else g_split[{g_device, f}] = v;
  return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **) {
  return launched(f, c->gridDim, c->blockDim, c->dynamicSmemBytes);
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3 block, void **, size_t smem, cudaStream_t) {
  return launched((const void *)k, grid, block, smem);
}
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaGetLastError() {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
}
