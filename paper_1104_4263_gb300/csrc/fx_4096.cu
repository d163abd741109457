// FP64 product passes (fx_kernels.cuh): length 4096.
#include "fx_kernels.cuh"

namespace die {

template struct FxLaunch<16, fx_plan(4096).r0, fx_plan(4096).r1, 4096>;

}  // namespace die
