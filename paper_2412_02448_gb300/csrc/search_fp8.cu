// The fused search kernel over FP8 E4M3 rows.
#include "search_kernel.cuh"

namespace unify {

cudaError_t launch_batch_fp8(const BatchArgs& a, int wpb, int regs, int num_sms, cudaStream_t st) {
  return launch_dt<StoreFP8>(a, wpb, regs, num_sms, st);
}

}  // namespace unify
