// yz pass of the three-pass Poisson solve for some lengths (plane.hpp).
#include "plane_kernels.cuh"

namespace lgf {

template struct PlaneYZ<16>;
template struct PlaneYZ<32>;
template struct PlaneYZ<64>;
template struct PlaneYZ<80>;
template struct PlaneYZ<240>;

}  // namespace lgf
