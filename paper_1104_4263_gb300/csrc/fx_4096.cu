// FP64 product passes (fx_kernels.cuh): length 4096.
#include "fx_kernels.cuh"

namespace die {

template struct FxLaunch<fx_plan(4096).ept, fx_plan(4096).r0, fx_plan(4096).r1, 4096>;

}  // namespace die
