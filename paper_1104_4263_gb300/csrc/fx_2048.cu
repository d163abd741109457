// FP64 product passes (fx_kernels.cuh): length 2048.
#include "fx_kernels.cuh"

namespace die {

template struct FxLaunch<fx_plan(2048).ept, fx_plan(2048).r0, fx_plan(2048).r1, 2048>;

}  // namespace die
