// Tables that are not aligned to pieces of memory columns or pairs of feature columns.
#include "k_attn_kernels.cuh"

namespace tgnn {
AttnKernel attn_kernel_words(int de, bool bf16, bool bwd) {
  if (de == 0) return pick_dir<1, 10, true, 2, 0, X_F32_SINGLE>(bwd);
  return bf16 ? pick_dir<1, 10, true, 2, 4, X_BF16_SINGLE>(bwd) : pick_dir<1, 10, true, 2, 4, X_F32_SINGLE>(bwd);
}
}  // namespace tgnn
