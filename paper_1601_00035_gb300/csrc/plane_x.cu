// x passes of the three-pass Poisson solve for some lengths (plane.hpp).
#include "plane_kernels.cuh"

namespace lgf {

template struct PlaneX<16>;
template struct PlaneX<32>;
template struct PlaneX<48>;
template struct PlaneX<64>;
template struct PlaneX<80>;
template struct PlaneX<96>;
template struct PlaneX<112>;
template struct PlaneX<128>;
template struct PlaneX<144>;
template struct PlaneX<160>;
template struct PlaneX<176>;
template struct PlaneX<192>;
template struct PlaneX<208>;
template struct PlaneX<224>;
template struct PlaneX<240>;
template struct PlaneX<256>;

}  // namespace lgf
