// Odd numbers of heads, d > 128.
#include "k_attn_kernels.cuh"

namespace tgnn {
template AttnKernel attn_kernel<1, 10, true, 2>(int, bool, bool);
}
