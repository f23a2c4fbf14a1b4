// The fused search kernel over float32 rows.
#include "search_kernel.cuh"

namespace unify {

cudaError_t launch_batch_f32(const BatchArgs& a, int wpb, int regs, int num_sms, cudaStream_t st) {
  return launch_dt<StoreF32>(a, wpb, regs, num_sms, st);
}

}  // namespace unify
