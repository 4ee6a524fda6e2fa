// Threads of each launch of an FP64 batch step with more work items of every kind
// than the GPU holds blocks.  Prints one line per launch: threads of a block, blocks.
#include "fake_runtime.h"

int main() {
  using namespace cem;
  StepStreams ss;
  memset(&ss, 0, sizeof ss);
  BatchDev b;
  memset(&b, 0, sizeof b);
  b.n = 64;
  b.n_main = b.n_pieces = b.n_ph = b.n_eval = 1 << 20;
  if (launch_step_fp64_batch(b, false, false, 16 * 152, ss) != cudaSuccess) return 1;
  for (const Launch &l : g_log) printf("%u %u\n", l.block.x, l.grid.x);
  return 0;
}
