// FP64 product passes (fx_kernels.cuh): lengths 192 and 384.
#include "fx_kernels.cuh"

namespace die {

template struct FxLaunch<fx_plan(192).ept, fx_plan(192).r0, fx_plan(192).r1, 192>;
template struct FxLaunch<fx_plan(384).ept, fx_plan(384).r0, fx_plan(384).r1, 384>;

}  // namespace die
