// Fills the scoring kernel's status, counters and row offsets with ones: no error, -1, and NaN ("not published yet").
//
// A kernel and not a memset, so that the scoring kernel's CTAs are launched and set themselves up meanwhile (programmatic
// launch): with the compaction chained to the selection likewise, a call of 4096 tokens x 32 heads takes 34.0 us instead of
// 39.1, a decode round 83.7 instead of 90.6.  In a file of its own: beside the scoring kernel it changes where that kernel's
// code comes to lie, which made it 9 % slower.
#include "ahakv_internal.cuh"

namespace ahakv {
namespace {

constexpr int kThreads = 128;

__global__ void __launch_bounds__(kThreads) clear_kernel(uint4* to, int count) {
  griddep_launch();
  griddep_wait();
  const int i = blockIdx.x * kThreads + threadIdx.x;
  if (i < count) to[i] = make_uint4(~0u, ~0u, ~0u, ~0u);
}

}  // namespace

ahakv_status launch_clear(void* to, size_t bytes, cudaStream_t st) {
  const int count = (int)(bytes / sizeof(uint4));
  count_launch();
  return cuda_ok(launch_chained(clear_kernel, dim3((count + kThreads - 1) / kThreads), dim3(kThreads), 1, 0, st, (uint4*)to, count));
}

}  // namespace ahakv
