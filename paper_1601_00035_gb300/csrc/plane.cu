// Host side of the three-pass Poisson solve (plane.hpp): choice of lengths, per-device
// tables, the kernel spectrum in the planes' order, and the dispatch over lengths.
#include <algorithm>
#include <cmath>
#include <map>
#include <mutex>
#include <vector>

#include "plane.hpp"

namespace lgf {
namespace {

// y lengths of a residue plane (the y stages are instantiated for these radices)
const int kPlaneY[] = {16, 32, 48, 64, 80, 96, 112, 128};

// Per length M: stage twiddles [R2][R1] w_M^(b q) of the x / y radices and of the z radices, and
// w_2M^n for n <= M.
struct Tables {
    float2 *d = nullptr;
    int st[kPlaneMax / 16 + 1] = {}, zt[kPlaneMax / 16 + 1] = {}, w2[kPlaneMax / 16 + 1] = {};
};
std::mutex g_mu;
std::map<int, Tables> g_tables;

lgf_status build_tables(Tables &t)
{
    const double tau = 6.28318530717958647692;
    std::vector<float2> h;
    for (int i = 0; i < 2 * (kPlaneMax / 16); i++) {
        const int M = 16 * (i / 2 + 1), R2 = i % 2 ? plane_z2(M) : plane_r2(M), R1 = M / R2;
        (i % 2 ? t.zt : t.st)[M / 16] = (int)h.size();
        for (int b = 0; b < R2; b++)
            for (int q = 0; q < R1; q++) {
                const double a = -tau * (b * q) / M;
                h.push_back(make_float2((float)std::cos(a), (float)std::sin(a)));
            }
        if (i % 2) continue;
        t.w2[M / 16] = (int)h.size();
        for (int n = 0; n <= M; n++) {
            const double a = -tau * n / (2 * M);
            h.push_back(make_float2((float)std::cos(a), (float)std::sin(a)));
        }
    }
    LGF_CUDA_TRY(cudaMalloc(&t.d, h.size() * sizeof(float2)));
    if (cudaMemcpy(t.d, h.data(), h.size() * sizeof(float2), cudaMemcpyHostToDevice) != cudaSuccess) {
        cudaFree(t.d);
        t.d = nullptr;
        set_error("upload of the transform tables failed");
        return LGF_ERR_CUDA;
    }
    return LGF_OK;
}

// the octant spectrum in the planes' order: Kt[kx][r][row][pos], row 0 .. Mz/2 the even z
// frequencies 2 row, the rest the odd ones 2 (row - Mz/2 - 1) + 1; position pos of the in-place
// order holds k = q + R1 k2 (pos = q R2 + k2), ky = Dy k + r
__global__ void k_plane_spectrum(const float *__restrict__ Kh, int KX, int Dy, int My, int R1, int R2, int Mz,
                                 float *__restrict__ Kt)
{
    const int Ny = Dy * My;
    const int64_t total = (int64_t)KX * Dy * (Mz + 1) * My;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int pos = (int)(i % My);
        const int row = (int)((i / My) % (Mz + 1));
        const int64_t kr = i / ((int64_t)My * (Mz + 1));
        const int r = (int)(kr % Dy), kx = (int)(kr / Dy);
        const int ky = Dy * (pos / R2 + R1 * (pos % R2)) + r;
        const int kyf = ky <= Ny / 2 ? ky : Ny - ky;
        const int kz = row <= Mz / 2 ? 2 * row : 2 * (row - Mz / 2 - 1) + 1;
        Kt[i] = Kh[((int64_t)kz * (Ny / 2 + 1) + kyf) * KX + kx];
    }
}

// plane, tables, and 16 columns of the odd half per group
inline size_t yz_smem(int My, int Mz, int threads)
{
    return ((size_t)(My + threads / plane_z2(Mz)) * (Mz + 1) + My + 3 * Mz) * sizeof(float2);
}
// Estimated time of the yz pass (arbitrary units): the columns that an SM of the 152 works through,
// at the issue rate of its resident warps.  The factors are fits to measured solves of 32^3 to 192^3
// boxes, one and three components: a single resident block hides less of its loads (1.25); clusters
// of three are placed badly, of four read more remote shared memory (1.3, 1.08; e.g. 96^3, three
// components: D = 2, M = 96 76 us, 4 x 48 80 us, 3 x 64 91 us).  threads: the block size that
// reaches it (whole column groups); 1e30 where no block fits.
double yz_cost(int KX, int D, int M, int Mz, int units, int &threads)
{
    const int gt = 16 * plane_z2(Mz), cap = plane_yz_threads(Mz);
    const double share = (double)KX * D * units / 152.0;  // thread blocks per SM
    double best = 1e30;
    for (int ng = 1; ng <= M / 16 && gt * ng <= cap; ng++) {
        const size_t sm = yz_smem(M, Mz, gt * ng) + 1024;
        if (sm > 228 * 1024) continue;
        const int fit = (int)std::min<size_t>(228 * 1024 / sm, cap / (gt * ng));
        const double warps = std::min<double>(fit, std::ceil(share)) * gt * ng / 32;
        const double rounds = (double)((M / 16 + ng - 1) / ng) * ng * 16 / M;  // idle groups in the last round
        const double waves = 0.7 * share + 0.3 * std::ceil(share);
        const double c = waves * (M * (0.5 + 0.5 * rounds) + 6.0) * (warps + 8.0) / warps * (fit == 1 ? 1.25 : 1.0) *
                         (D == 2 ? 1.0 : (D == 3 ? 1.3 : 1.08));
        if (c < best) {
            best = c;
            threads = gt * ng;
        }
    }
    return best;
}

inline int up16(long v) { return (int)((v + 15) / 16 * 16); }

}  // namespace

bool plane_pick(const Geom &g, const long maxabs[3], int units, PlaneGeom &o)
{
    // x: N >= 2 maxabs + 2 (the exact embedding) and N >= 2 Es (the zero half of the first stage)
    const long nx = std::max<long>(2 * maxabs[0] + 2, 2L * g.Es[0]);
    const long mz = std::max<long>(maxabs[2] + 1, std::max(g.Es[2], g.Et[2]));
    const long ny = 2 * maxabs[1] + 2;
    if (nx > 2 * kPlaneMax || mz > kPlaneMax || ny > 4 * 128) return false;
    o.Mx = up16((nx + 1) / 2);
    o.KX = o.Mx + 1;
    o.Mz = up16(mz);
    // y: Dy * My >= ny, by the geometry of one component alone, so that a solve's arithmetic does not
    // depend on what it is batched with; the threads per block by all units that run together
    double best = 1e30;
    o.My = 0;
    for (int D = 2; D <= kPlaneMaxD; D++)
        for (int M : kPlaneY) {
            int threads;
            const double c = (long)D * M >= ny ? yz_cost(o.KX, D, M, o.Mz, 1, threads) : 1e30;
            if (c < best) {
                best = c;
                o.My = M;
                o.Dy = D;
            }
        }
    if (!o.My) return false;
    yz_cost(o.KX, o.Dy, o.My, o.Mz, units, o.ntz);
    // A long target box around a short source (or the reverse) pads z to twice the longer: keep the
    // five passes where that costs more than the three save.  At equal padded points the three passes
    // take 0.7 to 0.9 of the five's time (96^3, three components: 77 against 103 us; 192^3 748 against
    // 1091), at 1.11 times the points 0.87 to 0.98, at 1.17 and 1.25 they lost (234 against 198 us, 312
    // against 280).  The 256-point y and z passes are the five's best (128^3: 192 against 183 us at
    // equal points, 151 against 174 at 0.88 of them).  Below 2^18 points the launches count: 64^3
    // 13 us against 18.
    const double vol = (double)o.Dy * o.My * 2 * o.Mz * o.KX, vol5 = (double)g.N[1] * g.N[2] * (g.N[0] / 2 + 1);
    if (vol > (1 << 18) && vol > (g.N[1] == 256 && g.N[2] == 256 ? 0.95 : 1.12) * vol5) return false;
    o.Ry1 = plane_r1(o.My);
    o.Ry2 = plane_r2(o.My);
    o.B = g.B;
    o.lB = g.lB;
    o.ncomp = g.ncomp;
    o.c0 = g.c0;
    o.nc = g.nc;
    for (int a = 0; a < 3; a++) {
        o.Es[a] = g.Es[a];
        o.Et[a] = g.Et[a];
        o.d0[a] = g.T0[a] - g.S0[a];
        o.nbS[a] = g.nbS[a];
        o.nbT[a] = g.nbT[a];
    }
    return true;
}

lgf_status plane_prepare()
{
    int dev = 0;
    LGF_CUDA_TRY(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lk(g_mu);
    Tables &t = g_tables[dev];
    if (t.d) return LGF_OK;
#define LGF_PREP(M)                    \
    LGF_TRY(PlaneX<M>::prepare());     \
    LGF_TRY(PlaneYZ<M>::prepare());
    LGF_PLANE_LENGTHS(LGF_PREP)
#undef LGF_PREP
    return build_tables(t);
}

lgf_status plane_tables(PlaneGeom &g)
{
    int dev = 0;
    LGF_CUDA_TRY(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lk(g_mu);
    const Tables &t = g_tables[dev];
    if (!t.d) {
        set_error("transform tables not built on this device");
        return LGF_ERR_STATE;
    }
    const int M[3] = {g.Mx, g.My, g.Mz};
    for (int a = 0; a < 3; a++) {
        g.st[a] = t.d + (a == 2 ? t.zt : t.st)[M[a] / 16];
        g.w2[a] = t.d + t.w2[M[a] / 16];
    }
    return LGF_OK;
}

lgf_status plane_spectrum(const double *d_octant, int K, const PlaneGeom &g, float *d_Kt, cudaStream_t s)
{
    const int N[3] = {2 * g.Mx, g.Dy * g.My, 2 * g.Mz};
    float *oct = nullptr;
    LGF_CUDA_TRY(cudaMalloc(&oct, (size_t)g.KX * (N[1] / 2 + 1) * (N[2] / 2 + 1) * sizeof(float)));
    lgf_status st = build_spectrum(d_octant, K, N, oct, nullptr, s);
    if (st == LGF_OK) {
        const int64_t total = (int64_t)plane_spectrum_size(g);
        k_plane_spectrum<<<(int)std::min<int64_t>((total + 255) / 256, 152 * 32), 256, 0, s>>>(oct, g.KX, g.Dy, g.My,
                                                                                             g.Ry1, g.Ry2, g.Mz, d_Kt);
        if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(s) != cudaSuccess) {
            set_error("spectrum reordering failed");
            st = LGF_ERR_CUDA;
        }
    }
    cudaFree(oct);
    return st;
}

size_t plane_smem(int pass, const PlaneGeom &g)
{
    return pass == 1 ? yz_smem(g.My, g.Mz, g.ntz) : 0;
}

int plane_tiles(int pass, const PlaneGeom &g)
{
    if (pass == 1) return g.KX * g.Dy;
    const int rows = pass == 0 ? g.Es[1] * g.Es[2] : g.Et[1] * g.Et[2];
    return (rows + 31) / 32;
}

#define LGF_PLANE_SWITCH(m, CALL)                                           \
    switch (m) {                                                            \
        LGF_PLANE_LENGTHS(CALL)                                             \
        default: set_error("unsupported plane length %d", m); return LGF_ERR_ARG; \
    }

lgf_status plane_pass(int pass, const PlaneGeom &g, const float *src, float *dst, cx<float> *wa, cx<float> *wb,
                      cudaStream_t s)
{
#define LGF_F(M) case M: return PlaneX<M>::fwd(g, src, wa, s);
#define LGF_Z(M) case M: return PlaneYZ<M>::run(g, wa, wb, s);
#define LGF_I(M) case M: return PlaneX<M>::inv(g, wb, dst, s);
    if (pass == 0) LGF_PLANE_SWITCH(g.Mx, LGF_F)
    if (pass == 1) LGF_PLANE_SWITCH(g.Mz, LGF_Z)
    LGF_PLANE_SWITCH(g.Mx, LGF_I)
#undef LGF_F
#undef LGF_Z
#undef LGF_I
}

lgf_status plane_pass_grouped(int pass, int M, size_t smem, int threads, int Dy, const PlaneTask *t, const int *cta, int n,
                              const PlanePtrs &p, cudaStream_t s)
{
#define LGF_F(L) case L: return PlaneX<L>::fwd_grp(t, cta, n, p, s);
#define LGF_Z(L) case L: return PlaneYZ<L>::grp(t, cta, n, smem, threads, Dy, s);
#define LGF_I(L) case L: return PlaneX<L>::inv_grp(t, cta, n, p, s);
    if (pass == 0) LGF_PLANE_SWITCH(M, LGF_F)
    if (pass == 1) LGF_PLANE_SWITCH(M, LGF_Z)
    LGF_PLANE_SWITCH(M, LGF_I)
#undef LGF_F
#undef LGF_Z
#undef LGF_I
}

lgf_status plane_launch(const PlaneGeom &g, const float *src, float *dst, cx<float> *wa, cx<float> *wb, cudaStream_t s,
                        Profiler *prof, cudaEvent_t mark, int mark_after)
{
    static const char *names[3] = {"x_fwd_gather_r2c", "yz_conv", "x_inv_c2r_scatter"};
    const bool P = prof && prof->on;
    for (int pass = 0; pass < 3; pass++) {
        if (P) prof->begin(s);
        LGF_TRY(plane_pass(pass, g, src, dst, wa, wb, s));
        if (P) prof->end(names[pass], s);
        if (mark && mark_after == pass) LGF_CUDA_TRY(cudaEventRecord(mark, s));
    }
    return LGF_OK;
}

}  // namespace lgf
