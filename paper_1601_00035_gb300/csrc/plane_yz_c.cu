// yz pass of the three-pass Poisson solve for some lengths (plane.hpp).
#include "plane_kernels.cuh"

namespace lgf {

template struct PlaneYZ<112>;
template struct PlaneYZ<144>;
template struct PlaneYZ<176>;
template struct PlaneYZ<192>;
template struct PlaneYZ<224>;
template struct PlaneYZ<256>;

}  // namespace lgf
