// The fused search kernel over bfloat16 rows.
#include "search_kernel.cuh"

namespace unify {

cudaError_t launch_batch_bf16(const BatchArgs& a, int wpb, int regs, int num_sms, cudaStream_t st) {
  return launch_dt<StoreBF16>(a, wpb, regs, num_sms, st);
}

}  // namespace unify
