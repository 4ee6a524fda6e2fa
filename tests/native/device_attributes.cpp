// Launches the steps of the library on two devices in turn with a stand-in
// for the CUDA runtime's launch and attribute calls (this program's own
// definitions come first at load time), which refuses a launch with more dynamic
// shared memory than the kernel has been allowed on the current device.
// Prints one line per launch that the stand-in refused; returns their number.
#include <cuda_runtime.h>
#include <stdio.h>
#include <string.h>

#include <map>
#include <utility>

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

static int g_device = 0, g_refused = 0, g_launches = 0;
static cudaError_t g_last = cudaSuccess;
static std::map<std::pair<int, const void *>, int> g_most, g_split;

static cudaError_t launched(const void *f, size_t smem) {
  ++g_launches;
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
  return launched(f, c->dynamicSmemBytes);
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void **, size_t smem, cudaStream_t) {
  return launched((const void *)k, smem);
}
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaGetLastError() {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
}

int main() {
  using namespace cem;
  int failed = 0;
  size_t splits[2] = {0, 0};
  for (g_device = 0; g_device < 2; ++g_device) {
    for (int precision = 0; precision < 2; ++precision) {
      static DevState d;
      memset(&d, 0, sizeof d);
      d.g.nx = 400;
      d.g.ny = 160;
      d.g.nn = 401 * 161;
      d.g.ne = 400 * 160;
      d.precision = precision;
      d.ph_cap = d.ck_cap = d.list_cap = 1000;
      tile64_shape(400, 160, d.t64x, d.t64y);
      StepStreams ss;
      memset(&ss, 0, sizeof ss);
      BatchDev b;
      memset(&b, 0, sizeof b);
      b.n = b.n_main = b.n_pieces = b.n_ph = b.n_eval = 1;
      for (int energy = 0; energy < 2; ++energy)
        if (precision) {
          failed += launch_step_fp32(d, 0, false, energy, ss, nullptr) != cudaSuccess;
          failed += launch_step_fp32_batch(b, false, energy, 16, 152, ss) != cudaSuccess;
        } else {
          failed += launch_step_fp64(d, 0, false, energy, ss, nullptr) != cudaSuccess;
          failed += launch_step_fp64_batch(b, false, energy, 152, ss) != cudaSuccess;
        }
    }
    for (auto &kv : g_split) splits[g_device] += kv.first.first == g_device;
  }
  printf("%d launches, %d refused, %d calls failed, shared-memory splits set: %zu and %zu\n", g_launches,
         g_refused, failed, splits[0], splits[1]);
  return g_launches == 0 || g_refused || failed || !splits[0] || splits[0] != splits[1];
}
