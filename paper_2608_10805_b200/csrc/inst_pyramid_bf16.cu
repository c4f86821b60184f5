// Instantiation unit: whole-plane kernels of several levels with tensor cores, bf16 activations.
#include "pyramid_kernels.cuh"
namespace wt {
namespace pyramid {
WT_PYRAMID_INSTANTIATE(__nv_bfloat16, )
}  // namespace pyramid
}  // namespace wt
