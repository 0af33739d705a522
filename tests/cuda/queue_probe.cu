// Lengths of a context's queues after its last sub-step: retry queue, back-up
// list, Newton continuation queue, its finite-difference end
// (tests/test_gpu_queue_ends.py builds and loads this file).
#include "hr_ctx.h"

extern "C" int queue_counts(const harmrad_ctx* c, int* out) {
  if (cudaStreamSynchronize(c->stream) != cudaSuccess) return 1;
  return (int)cudaMemcpy(out, c->qcount, 4 * sizeof(int), cudaMemcpyDeviceToHost);
}
