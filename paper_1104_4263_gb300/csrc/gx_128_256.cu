// Complex64 product passes on any grid (gx_kernels.cuh): lengths 128, 192, 256.
#include "gx_kernels.cuh"

namespace die {

DIE_GX_INSTANTIATE(128)
DIE_GX_INSTANTIATE(192)
DIE_GX_INSTANTIATE(256)

}  // namespace die
