// Complex64 product passes on any grid (gx_kernels.cuh): lengths 1536, 2048.
#include "gx_kernels.cuh"

namespace die {

DIE_GX_INSTANTIATE(1536)
DIE_GX_INSTANTIATE(2048)

}  // namespace die
