// Instantiation unit: tensor-core kernels, f16 activations.
#include "tensor_kernels.cuh"
namespace wt {
namespace tensor {
WT_TENSOR_INSTANTIATE(__half, )
}  // namespace tensor
}  // namespace wt
