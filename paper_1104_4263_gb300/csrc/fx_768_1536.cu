// FP64 product passes (fx_kernels.cuh): lengths 768 and 1536.
#include "fx_kernels.cuh"

namespace die {

template struct FxLaunch<fx_plan(768).ept, fx_plan(768).r0, fx_plan(768).r1, 768>;
template struct FxLaunch<fx_plan(1536).ept, fx_plan(1536).r0, fx_plan(1536).r1, 1536>;

}  // namespace die
