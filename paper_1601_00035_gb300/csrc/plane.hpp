// Three-pass FP32 form of the Poisson solve (kernels in plane_kernels.cuh):
//   x forward   gather, real transform along x, transposed store
//   yz          per (kx, residue of ky): transform along y, convolution along z,
//               inverse along y, all in one shared-memory plane
//   x inverse   recombination of the ky residues, real inverse along x, scatter
// against the five passes of poisson.cu (which FP64 plans and boxes beyond the lengths here keep).
#pragma once
#include "plan.hpp"
#include "plane_len.hpp"

namespace lgf {

struct PlaneTask {  // one unit of a grouped launch
    PlaneGeom g;
    cx<float> *wa, *wb;
    int solve, first;
};
constexpr int kPlaneMaxSolves = 128;
struct PlanePtrs {
    const float *src[kPlaneMaxSolves];
    float *dst[kPlaneMaxSolves];
};

// lengths for a solve (g: boxes and origins set; maxabs: largest |target - source| offset per
// axis); false where the five-pass form is the one to take
// units: (solve, component) pairs whose launches share the GPU
bool plane_pick(const Geom &g, const long maxabs[3], int units, PlaneGeom &out);
lgf_status plane_prepare();                 // per-device tables and kernel attributes
lgf_status plane_tables(PlaneGeom &g);      // fills st, w2 from the per-device tables
lgf_status plane_spectrum(const double *d_octant, int K, const PlaneGeom &g, float *d_Kt, cudaStream_t s);
inline size_t plane_spectrum_size(const PlaneGeom &g) { return (size_t)g.KX * g.Dy * (g.Mz + 1) * g.My; }
inline size_t plane_elems_a(const PlaneGeom &g) { return (size_t)g.KX * g.Es[1] * g.Es[2]; }          // per component
inline size_t plane_elems_b(const PlaneGeom &g) { return (size_t)g.KX * g.Et[1] * g.Et[2]; }
int plane_tiles(int pass, const PlaneGeom &g);  // thread blocks of one component (pass 0, 1, 2)
lgf_status plane_pass(int pass, const PlaneGeom &g, const float *src, float *dst, cx<float> *wa, cx<float> *wb,
                      cudaStream_t s);
lgf_status plane_pass_grouped(int pass, int M, size_t smem, int threads, int Dy, const PlaneTask *tasks, const int *cta, int ncta,
                              const PlanePtrs &ptrs, cudaStream_t s);
size_t plane_smem(int pass, const PlaneGeom &g);
lgf_status plane_launch(const PlaneGeom &g, const float *src, float *dst, cx<float> *wa, cx<float> *wb, cudaStream_t s,
                        Profiler *prof = nullptr, cudaEvent_t mark = nullptr, int mark_after = -1);

// per length M (multiple of 16): the launches, instantiated in the plane_*.cu units
template <int M>
struct PlaneX {
    static lgf_status prepare();
    static lgf_status fwd(const PlaneGeom &g, const float *src, cx<float> *a, cudaStream_t s);
    static lgf_status inv(const PlaneGeom &g, const cx<float> *b, float *dst, cudaStream_t s);
    static lgf_status fwd_grp(const PlaneTask *t, const int *cta, int ncta, const PlanePtrs &p, cudaStream_t s);
    static lgf_status inv_grp(const PlaneTask *t, const int *cta, int ncta, const PlanePtrs &p, cudaStream_t s);
};
template <int M>
struct PlaneYZ {
    static lgf_status prepare();
    static lgf_status run(const PlaneGeom &g, const cx<float> *a, cx<float> *b, cudaStream_t s);
    static lgf_status grp(const PlaneTask *t, const int *cta, int ncta, size_t smem, int threads, int Dy,
                          cudaStream_t s);
};

}  // namespace lgf
