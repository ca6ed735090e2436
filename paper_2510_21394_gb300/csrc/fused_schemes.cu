// Fused-epilogue mode products: ETD2RK, the one-operator schemes and LBDF2.
#include "b3_launch.cuh"

namespace fcgle {

template struct FusedLaunch<b3::EpiEtd2>;
template struct FusedLaunch<b3::EpiSpecStep>;
template struct FusedLaunch<b3::EpiLBDF2S>;
template struct FusedLaunch<b3::EpiExtrapG>;

}  // namespace fcgle
