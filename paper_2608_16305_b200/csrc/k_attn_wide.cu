// d > 128, even numbers of heads.
#include "k_attn_kernels.cuh"

namespace tgnn {
template AttnKernel attn_kernel<2, 10, true, 2>(int, bool, bool);
}
