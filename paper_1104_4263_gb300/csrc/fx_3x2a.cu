// FP64 product passes (fx_kernels.cuh): lengths 48, 96 and the runtime plan of the others of 3 * 2^a.
#include "fx_kernels.cuh"

namespace die {

template struct FxLaunch<12, 6, 4, 0>;
template struct FxLaunch<12, 12, 4, 0>;
template struct FxLaunch<fx_plan(48).ept, fx_plan(48).r0, fx_plan(48).r1, 48>;
template struct FxLaunch<fx_plan(96).ept, fx_plan(96).r0, fx_plan(96).r1, 96>;

}  // namespace die
