// Instantiation unit: weight gradients of whole planes of several levels with tensor cores, f16 activations.
#include "pyramid_gradient.cuh"
namespace wt {
namespace pyramid {
WT_PYRAMID_INSTANTIATE(__half, extern)
WT_GRADIENT_INSTANTIATE(__half, )
}  // namespace pyramid
}  // namespace wt
