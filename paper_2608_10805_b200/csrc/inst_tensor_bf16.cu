// Instantiation unit: tensor-core kernels, bf16 activations.
#include "tensor_kernels.cuh"
namespace wt {
namespace tensor {
WT_TENSOR_INSTANTIATE(__nv_bfloat16, )
}  // namespace tensor
}  // namespace wt
