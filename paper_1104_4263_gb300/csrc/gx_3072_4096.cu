// Complex64 product passes on any grid (gx_kernels.cuh): lengths 3072, 4096.
#include "gx_kernels.cuh"

namespace die {

DIE_GX_INSTANTIATE(3072)
DIE_GX_INSTANTIATE(4096)

}  // namespace die
