// Complex64 product passes on any grid (gx_kernels.cuh): lengths 16, 24, 32, 48, 64, 96.
#include "gx_kernels.cuh"

namespace die {

DIE_GX_INSTANTIATE(16)
DIE_GX_INSTANTIATE(24)
DIE_GX_INSTANTIATE(32)
DIE_GX_INSTANTIATE(48)
DIE_GX_INSTANTIATE(64)
DIE_GX_INSTANTIATE(96)

}  // namespace die
