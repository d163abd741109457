// Complex64 product passes on any grid (gx_kernels.cuh): lengths 768, 1024.
#include "gx_kernels.cuh"

namespace die {

DIE_GX_INSTANTIATE(768)
DIE_GX_INSTANTIATE(1024)

}  // namespace die
