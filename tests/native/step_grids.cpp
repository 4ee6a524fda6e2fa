// An FP32 step of n x n elements, all of which may split: "1" or "0" for whether the
// evaluation (the first launch) asks for a shared-memory split, then for each launch
// its threads of a block and blocks.
#include <stdlib.h>

#include "fake_runtime.h"

int main() {
  using namespace cem;
  const char *side = getenv("MESH_SIDE");
  const int n = side ? atoi(side) : 1024;
  static DevState d;
  memset(&d, 0, sizeof d);
  d.precision = 1;
  d.g.nx = d.g.ny = n;
  d.g.nn = (n + 1) * (n + 1);
  d.g.ne = n * n;
  d.ck_cap = d.ph_cap = d.list_cap = n * n;
  StepStreams ss;
  memset(&ss, 0, sizeof ss);
  if (launch_step_fp32(d, 0, false, false, ss, nullptr) != cudaSuccess || g_log.empty()) return 1;
  printf("%d\n", (int)g_split.count({g_device, g_log[0].f}));
  for (const Launch &l : g_log) printf("%u %u\n", l.block.x, l.grid.x);
  return 0;
}
