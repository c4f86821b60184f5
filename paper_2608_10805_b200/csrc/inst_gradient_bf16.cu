// Instantiation unit: weight gradients of whole planes of several levels with tensor cores, bf16 activations.
#include "pyramid_gradient.cuh"
namespace wt {
namespace pyramid {
WT_PYRAMID_INSTANTIATE(__nv_bfloat16, extern)
WT_GRADIENT_INSTANTIATE(__nv_bfloat16, )
}  // namespace pyramid
}  // namespace wt
