// Instantiation unit: whole-plane kernels of several levels with tensor cores, f16 activations.
#include "pyramid_kernels.cuh"
namespace wt {
namespace pyramid {
WT_PYRAMID_INSTANTIATE(__half, )
}  // namespace pyramid
}  // namespace wt
