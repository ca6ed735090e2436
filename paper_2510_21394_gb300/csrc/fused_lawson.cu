// Fused-epilogue mode products: Lawson-RK2, Strang and the complex (Kronecker-product) products.
#include "b3_launch.cuh"

namespace fcgle {

template struct FusedLaunch<b3::EpiLRK2A>;
template struct FusedLaunch<b3::EpiLRK2B>;
template struct FusedLaunch<b3::EpiStrangB>;
template struct FusedLaunchCx<b3::EpiStoreF32>;
template struct FusedLaunchCx<b3::EpiStoreSplitGen>;
template struct FusedLaunchCx<b3::EpiUpdateG>;
template struct FusedLaunchCx<b3::EpiStrangKron>;
template struct FusedLaunchCx<b3::EpiLRK2Kron>;

}  // namespace fcgle
