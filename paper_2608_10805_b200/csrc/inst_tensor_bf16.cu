// Instantiation unit: tensor-core kernels, bf16 activations.
#include "panel_host.cuh"
namespace wt {
namespace tensor {
WT_TENSOR_INSTANTIATE(__nv_bfloat16, )
WT_WIDE_INSTANTIATE(__nv_bfloat16, )
}  // namespace tensor
}  // namespace wt
