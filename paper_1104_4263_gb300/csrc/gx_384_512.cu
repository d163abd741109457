// Complex64 product passes on any grid (gx_kernels.cuh): lengths 384, 512.
#include "gx_kernels.cuh"

namespace die {

DIE_GX_INSTANTIATE(384)
DIE_GX_INSTANTIATE(512)

}  // namespace die
