// FP64 product passes (fx_kernels.cuh): lengths 128 and 256.
#include "fx_kernels.cuh"

namespace die {

template struct FxLaunch<fx_plan(128).ept, fx_plan(128).r0, fx_plan(128).r1, 128>;
template struct FxLaunch<fx_plan(256).ept, fx_plan(256).r0, fx_plan(256).r1, 256>;

}  // namespace die
