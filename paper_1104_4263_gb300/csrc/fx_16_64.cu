// FP64 product passes (fx_kernels.cuh): lengths 16, 32 and 64.
#include "fx_kernels.cuh"

namespace die {

template struct FxLaunch<fx_plan(16).ept, fx_plan(16).r0, fx_plan(16).r1, 16>;
template struct FxLaunch<fx_plan(32).ept, fx_plan(32).r0, fx_plan(32).r1, 32>;
template struct FxLaunch<fx_plan(64).ept, fx_plan(64).r0, fx_plan(64).r1, 64>;

}  // namespace die
