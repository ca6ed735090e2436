// Fused-epilogue mode products: the Krogstad stages (and the ETD2RK ones they share).
#include "b3_launch.cuh"

namespace fcgle {

template struct FusedLaunch<b3::EpiFhat>;
template struct FusedLaunch<b3::EpiStageD>;
template struct FusedLaunch<b3::EpiKrog2>;
template struct FusedLaunch<b3::EpiKrog3>;
template struct FusedLaunch<b3::EpiKrogFinal>;

}  // namespace fcgle
