// Fused-epilogue mode products: stores, spectral scaling and the state update.
#include "b3_launch.cuh"

namespace fcgle {

template struct FusedLaunch<b3::EpiStoreSplitGen>;
template struct FusedLaunch<b3::EpiStoreF32>;
template struct FusedLaunch<b3::EpiScaleF>;
template struct FusedLaunch<b3::EpiUpdateG>;

}  // namespace fcgle
