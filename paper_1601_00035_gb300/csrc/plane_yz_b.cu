// yz pass of the three-pass Poisson solve for some lengths (plane.hpp).
#include "plane_kernels.cuh"

namespace lgf {

template struct PlaneYZ<48>;
template struct PlaneYZ<96>;
template struct PlaneYZ<128>;
template struct PlaneYZ<160>;
template struct PlaneYZ<208>;

}  // namespace lgf
