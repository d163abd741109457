// FP64 product passes (fx_kernels.cuh): lengths 512 and 1024.
#include "fx_kernels.cuh"

namespace die {

template struct FxLaunch<fx_plan(512).ept, fx_plan(512).r0, fx_plan(512).r1, 512>;
template struct FxLaunch<fx_plan(1024).ept, fx_plan(1024).r0, fx_plan(1024).r1, 1024>;

}  // namespace die
