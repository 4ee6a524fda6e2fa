// Launches the steps of the library on two devices in turn.  Prints one line per
// launch that the stand-in runtime refused; returns 0 when there was none.
#include "fake_runtime.h"

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
  printf("%d launches, %d refused, %d calls failed, shared-memory splits set: %zu and %zu\n", (int)g_log.size(),
         g_refused, failed, splits[0], splits[1]);
  return g_log.empty() || g_refused || failed || !splits[0] || splits[0] != splits[1];
}
