// Instantiation unit: tensor-core kernels, f16 activations.
#include "panel_host.cuh"
namespace wt {
namespace tensor {
WT_TENSOR_INSTANTIATE(__half, )
WT_WIDE_INSTANTIATE(__half, )
}  // namespace tensor
}  // namespace wt
