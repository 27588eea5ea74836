// 11 to 16 neighbors, d <= 128, even numbers of heads.
#include "k_attn_kernels.cuh"

namespace tgnn {
template AttnKernel attn_kernel<2, 16, false, 1>(int, bool, bool);
}
