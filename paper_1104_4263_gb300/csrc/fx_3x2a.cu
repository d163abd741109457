// FP64 product passes (fx_kernels.cuh): lengths 3 * 2^a.
#include "fx_kernels.cuh"

namespace die {

template struct FxLaunch<12, 6, 4, 0>;
template struct FxLaunch<12, 12, 4, 0>;

}  // namespace die
