// More than 16 neighbors, d <= 128, even numbers of heads.
#include "k_attn_kernels.cuh"

namespace tgnn {
template AttnKernel attn_kernel<2, 10, true, 1>(int, bool, bool);
}
