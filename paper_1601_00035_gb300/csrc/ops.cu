// Local operators of the staggered grid (App. A point forms) on a block set,
// with the mask semantics of Sec. 4.2: values outside the listed blocks are
// zero.  Axis map: component (1),(2),(3) = x, y, z; position index n = (i, j, k).
//
//   G^T f  (faces -> cells):   sum_q (f^q_{n-e_q} - f^q_n) / dx            (G^T = -Dbar)
//   G c    (cells -> faces):   (c_{n+e_q} - c_n) / dx
//   C f    (faces -> edges):   (f^r_n - f^r_{n+e_s} + f^s_{n+e_r} - f^s_n) / dx,  (q,r,s) cyclic
//   C^T e  (edges -> faces):   (e^r_{n-e_s} - e^r_n + e^s_n - e^s_{n-e_r}) / dx
//   N~(f)  (faces -> faces, eq. opr_def_nonlin, e = C f):
//     1/4 sum_{m in {-1,0}} [ e^r_{n+m e_s} (f^s + f^s_{+e_q})_{n+m e_s} - e^s_{n+m e_r} (f^r + f^r_{+e_q})_{n+m e_r} ]
//
// One thread block per block of the set; neighbour values come through the
// 27-neighbour table (L1/L2).  The operators overlap their predecessor's end (programmatic dependent
// launch: every operator once on the 256^3 ring 123 -> 113 us) and read its output by ordinary
// loads (__ldca), since loads through the read-only path may be taken before the wait for it.  The
// two that follow a Poisson solve, C^T and the projection tail, do not: started beside the solve's
// last pass they would run on its shared-memory carveout, with little L1 for the neighbours' rows
// (the ring's step 1534 against 1428 us, its velocity refresh 748 against 739).
#include <algorithm>

#include "plan.hpp"

namespace lgf {
namespace {

template <int B>
struct Fetch {
    const float *f;
    int ncomp;
    const int *nb;  // 27 neighbours of this block
    // value of component c at local position (x, y, z), which may lie in a neighbour
    __device__ __forceinline__ float operator()(int c, int x, int y, int z) const
    {
        const int dx = x < 0 ? -1 : (x >= B ? 1 : 0);
        const int dy = y < 0 ? -1 : (y >= B ? 1 : 0);
        const int dz = z < 0 ? -1 : (z >= B ? 1 : 0);
        const int n = nb[(dz + 1) * 9 + (dy + 1) * 3 + (dx + 1)];
        if (n < 0) return 0.f;
        return __ldg(f + ((size_t)(n * ncomp + c) * B + (z - dz * B)) * B * B + (y - dy * B) * B + (x - dx * B));
    }
};

// Four x-adjacent points per thread: thread (xq, y) of a z slab walks its planes, so that a row
// moves in 16-byte pieces, the z neighbours stay in registers from one plane to the next, and a
// neighbour block is selected once per four points.  (A thread per column with a neighbour
// selection per value took 55 us for the curl of the 256^3 ring's 1251 blocks, 123 MB, bound by
// the selections' integer instructions; this form is bound by memory, see op_launch.)
// V4: 16-byte accesses (both buffers aligned), else the same in scalar ones.
template <int B>
struct Slab {
    static constexpr int Q = B / 4;          // quads per row
    static constexpr int ZT = 4;             // slabs of a block
    static constexpr int ZP = B / ZT;        // planes of a slab
    static constexpr int threads = Q * B * ZT;
};

struct Quad {
    float v[4];
};
template <bool V4>
__device__ __forceinline__ Quad get(const float *p)
{
    if constexpr (V4) {
        const float4 w = __ldca(reinterpret_cast<const float4 *>(p));
        return {{w.x, w.y, w.z, w.w}};
    } else
        return {{__ldca(p), __ldca(p + 1), __ldca(p + 2), __ldca(p + 3)}};
}
template <int B, bool V4>
struct Rows {
    const float *f;
    int ncomp;
    const int *nb;  // 27 neighbours of this block (shared memory)
    // base of the row (y, z) of component c, which may lie one block off in y or z; null if absent
    __device__ __forceinline__ const float *row(int c, int y, int z, int dx = 0) const
    {
        const int dy = y < 0 ? -1 : (y >= B ? 1 : 0), dz = z < 0 ? -1 : (z >= B ? 1 : 0);
        const int n = nb[(dz + 1) * 9 + (dy + 1) * 3 + dx + 1];
        return n < 0 ? nullptr : f + ((size_t)(n * ncomp + c) * B + (z - dz * B)) * B * B + (y - dy * B) * B;
    }
    __device__ __forceinline__ Quad quad(int c, int xq, int y, int z) const
    {
        const float *p = row(c, y, z);
        return p ? get<V4>(p + 4 * xq) : Quad{{0.f, 0.f, 0.f, 0.f}};
    }
    // value at x = -1 .. B of row (y, z)
    __device__ __forceinline__ float at(int c, int x, int y, int z) const
    {
        const int dx = x < 0 ? -1 : (x >= B ? 1 : 0);
        const float *p = row(c, y, z, dx);
        return p ? __ldca(p + x - dx * B) : 0.f;
    }
    // the quad moved by one point along x
    __device__ __forceinline__ Quad next_x(const Quad &q, int c, int xq, int y, int z) const
    {
        return {{q.v[1], q.v[2], q.v[3], at(c, 4 * xq + 4, y, z)}};
    }
    __device__ __forceinline__ Quad prev_x(const Quad &q, int c, int xq, int y, int z) const
    {
        return {{at(c, 4 * xq - 1, y, z), q.v[0], q.v[1], q.v[2]}};
    }
};
template <bool V4>
__device__ __forceinline__ void put(float *p, const Quad &q)
{
    if constexpr (V4) *reinterpret_cast<float4 *>(p) = make_float4(q.v[0], q.v[1], q.v[2], q.v[3]);
    else
#pragma unroll
        for (int i = 0; i < 4; i++) p[i] = q.v[i];
}

// OP: 0 curl (faces->edges), 1 curl^T (edges->faces), 2 G^T (faces->cells), 3 G (cells->faces)
template <int B, int OP, bool V4>
__global__ void __launch_bounds__(Slab<B>::threads) k_op(const float *__restrict__ in, float *__restrict__ out,
                                                         const int *__restrict__ nbr27, float inv_dx)
{
    using S = Slab<B>;
    const int blk = blockIdx.x;
    __shared__ int nb[27];
    if (threadIdx.x < 27) nb[threadIdx.x] = nbr27[blk * 27 + threadIdx.x];
    __syncthreads();
    pdl_trigger();
    pdl_wait();  // the previous kernel's output
    const int xq = threadIdx.x % S::Q, y = (threadIdx.x / S::Q) % B, z0 = threadIdx.x / (S::Q * B) * S::ZP;
    constexpr int nin = OP == 3 ? 1 : 3, nout = OP == 2 ? 1 : 3;
    const Rows<B, V4> F{in, nin, nb};
    float *o = out + ((size_t)blk * nout * B + z0) * B * B + y * B + 4 * xq;
    constexpr size_t cs = (size_t)B * B * B;
    // lo: planes z - 1 (backward differences) or z (forward ones), rolling
    Quad lo[nin];
#pragma unroll
    for (int c = 0; c < nin; c++) lo[c] = F.quad(c, xq, y, OP == 1 || OP == 2 ? z0 - 1 : z0);
#pragma unroll
    for (int k = 0; k < S::ZP; k++, o += B * B) {
        const int z = z0 + k;
        Quad r[nout];
        if constexpr (OP == 0) {
            const Quad f0 = lo[0], f1 = lo[1], f2 = lo[2];
            const Quad z0q = F.quad(0, xq, y, z + 1), z1q = F.quad(1, xq, y, z + 1);
            const Quad y0q = F.quad(0, xq, y + 1, z), y2q = F.quad(2, xq, y + 1, z);
            const Quad x1q = F.next_x(f1, 1, xq, y, z), x2q = F.next_x(f2, 2, xq, y, z);
#pragma unroll
            for (int i = 0; i < 4; i++) {
                r[0].v[i] = (f1.v[i] - z1q.v[i] + y2q.v[i] - f2.v[i]) * inv_dx;
                r[1].v[i] = (f2.v[i] - x2q.v[i] + z0q.v[i] - f0.v[i]) * inv_dx;
                r[2].v[i] = (f0.v[i] - y0q.v[i] + x1q.v[i] - f1.v[i]) * inv_dx;
            }
            lo[0] = z0q;
            lo[1] = z1q;
            if (k + 1 < S::ZP) lo[2] = F.quad(2, xq, y, z + 1);
        } else if constexpr (OP == 1) {
            const Quad e0 = F.quad(0, xq, y, z), e1 = F.quad(1, xq, y, z), e2 = F.quad(2, xq, y, z);
            const Quad y0q = F.quad(0, xq, y - 1, z), y2q = F.quad(2, xq, y - 1, z);
            const Quad x1q = F.prev_x(e1, 1, xq, y, z), x2q = F.prev_x(e2, 2, xq, y, z);
#pragma unroll
            for (int i = 0; i < 4; i++) {
                r[0].v[i] = (lo[1].v[i] - e1.v[i] + e2.v[i] - y2q.v[i]) * inv_dx;
                r[1].v[i] = (x2q.v[i] - e2.v[i] + e0.v[i] - lo[0].v[i]) * inv_dx;
                r[2].v[i] = (y0q.v[i] - e0.v[i] + e1.v[i] - x1q.v[i]) * inv_dx;
            }
            lo[0] = e0;
            lo[1] = e1;
        } else if constexpr (OP == 2) {
            const Quad f0 = F.quad(0, xq, y, z), f1 = F.quad(1, xq, y, z), f2 = F.quad(2, xq, y, z);
            const Quad x0q = F.prev_x(f0, 0, xq, y, z), y1q = F.quad(1, xq, y - 1, z);
#pragma unroll
            for (int i = 0; i < 4; i++) {
                float v = x0q.v[i] - f0.v[i];
                v += y1q.v[i] - f1.v[i];
                v += lo[2].v[i] - f2.v[i];
                r[0].v[i] = v * inv_dx;
            }
            lo[2] = f2;
        } else {
            const Quad c0 = lo[0], zq = F.quad(0, xq, y, z + 1), yq = F.quad(0, xq, y + 1, z);
            const Quad xn = F.next_x(c0, 0, xq, y, z);
#pragma unroll
            for (int i = 0; i < 4; i++) {
                r[0].v[i] = (xn.v[i] - c0.v[i]) * inv_dx;
                r[1].v[i] = (yq.v[i] - c0.v[i]) * inv_dx;
                r[2].v[i] = (zq.v[i] - c0.v[i]) * inv_dx;
            }
            lo[0] = zq;
        }
#pragma unroll
        for (int c = 0; c < nout; c++) put<V4>(o + c * cs, r[c]);
    }
}

// N~(f) with shared-memory planes: thread (x, y) walks z; plane z' of f = M(u + u_inf) with a one-cell
// halo in x and y lives in a ring of five slots, and plane z' of e = C f at in-plane positions
// -1 .. B-1 in a ring of three, so every stencil value is one shared-memory read and a plane costs one
// barrier: what a thread overtaking the others writes next lies in slots they no longer read.  The
// planes are unrolled, so that slots are constants.  Same arithmetic as eq. opr_def_nonlin.
// The 256^3 ring's 1251 blocks, 123 MB (184 with rv): 41 -> 33 us (48 -> 43 with rv), all of it by the
// reads free of bank conflicts; one barrier instead of three, addresses kept, and values kept in
// registers from plane to plane each measured the same, so what is left is latency.
// rv (optional): also writes rv = u + out (the first stage's r = u + g without a separate
// linear combination; the same single FP32 addition).
template <int B>
__global__ void __launch_bounds__(B *B) k_nonlinear(const float *__restrict__ in, float *__restrict__ out,
                                                    const int *__restrict__ nbr27,
                                                    const unsigned char *__restrict__ out_keep, float inv_dx,
                                                    float coef, float u0, float u1, float u2, float *__restrict__ rv)
{
    constexpr int H = B + 2;  // f plane edge (halo -1 .. B)
    constexpr int HE = B + 1; // e plane edge (-1 .. B-1)
    __shared__ int nb[27];
    __shared__ float Fs[5][3][H * H];   // [slot][component][(y+1) H + (x+1)]
    __shared__ float Es[3][3][HE * H];  // [slot][component][(y+1) H + (x+1)], its last column unused
    // thread block (blk, zs) walks output planes z0 .. z0 + ZP - 1 of block blk; planes are numbered from z0
    constexpr int ZS = B >= 16 ? 2 : 1, ZP = B / ZS;
    constexpr size_t cs = (size_t)B * B * B;
    const int blk = blockIdx.x / ZS;
    const int z0 = (blockIdx.x % ZS) * ZP;
    // a warp takes rows y and y + 8 of a 16^3 block: 8 H = 16 mod 32, so its halves read different banks
    // (adjacent rows, 18 apart, share two and cost every read a second pass)
    const int x = threadIdx.x % B, y = B == 16 ? threadIdx.x / 32 + threadIdx.x / 16 % 2 * 8 : threadIdx.x / B;
    const bool keep = out_keep == nullptr || out_keep[blk];
    const size_t o0 = ((size_t)blk * 3 * B + z0) * B * B + y * B + x;
    pdl_trigger();
    pdl_wait();  // the previous kernel's output
    if (!keep) {
        for (int z = 0; z < ZP; z++)
#pragma unroll
            for (int q = 0; q < 3; q++) {
                const size_t o = o0 + q * cs + z * B * B;
                out[o] = 0.f;
                if (rv) rv[o] = __ldca(in + o);
            }
        return;
    }
    if (threadIdx.x < 27) nb[threadIdx.x] = nbr27[blk * 27 + threadIdx.x];
    __syncthreads();
    const float uinf[3] = {u0, u1, u2};
    // f plane zp (-1 .. ZP): fetch_f reads it from global memory into registers
    // (each thread holds at most 2 points x 3 components: (B + 2)^2 < 2 B^2),
    // commit_f stores it into its slot, so a plane's loads can be in flight
    // while the previous plane is computed
    constexpr int PT = (H * H + B * B - 1) / (B * B);
    static_assert(PT <= 2, "halo plane points per thread");
    int row[PT], at[PT];  // of a thread's points: neighbour (dy, dx), place in that block's plane
#pragma unroll
    for (int t = 0; t < PT; t++) {
        const int idx = threadIdx.x + t * B * B;
        const int hx = idx % H - 1, hy = idx / H - 1;
        const int dx = hx < 0 ? -1 : (hx >= B ? 1 : 0), dy = hy < 0 ? -1 : (hy >= B ? 1 : 0);
        row[t] = idx < H * H ? (dy + 1) * 3 + dx + 1 : -1;
        at[t] = (hy - dy * B) * B + hx - dx * B;
    }
    float pre[PT][3];
    auto fetch_f = [&](int zp) {
        const int z = z0 + zp, dz = z < 0 ? -1 : (z >= B ? 1 : 0);
#pragma unroll
        for (int t = 0; t < PT; t++) {
            const int n = row[t] >= 0 ? nb[(dz + 1) * 9 + row[t]] : -1;
            const float *p = in + ((size_t)n * 3 * B + (z - dz * B)) * (B * B) + at[t];
#pragma unroll
            for (int c = 0; c < 3; c++) pre[t][c] = n >= 0 ? __ldca(p + c * cs) + uinf[c] : 0.f;
        }
    };
    auto commit_f = [&](int zp) {
        float *dst = &Fs[(zp + 1) % 5][0][threadIdx.x];
#pragma unroll
        for (int t = 0; t < PT; t++)
            if (row[t] >= 0)
#pragma unroll
                for (int c = 0; c < 3; c++) dst[c * H * H + t * B * B] = pre[t][c];
    };
    // e plane zp (-1 .. ZP - 1): e^c(p) = f^r(p) - f^r(p + e_s) + f^s(p + e_r) - f^s(p), (c, r, s) cyclic
    constexpr int ET = (HE * H + B * B - 1) / (B * B);
    auto make_e = [&](int zp) {
        const float(*f)[H * H] = Fs[(zp + 1) % 5], (*g)[H * H] = Fs[(zp + 2) % 5];  // planes zp, zp + 1
        float(*e)[HE * H] = Es[(zp + 1) % 3];
#pragma unroll
        for (int t = 0; t < ET; t++) {
            const int p = threadIdx.x + t * B * B;
            if (p >= HE * H) continue;
            const float f0 = f[0][p], f1 = f[1][p], f2 = f[2][p];
            // c = 0 (r = y, s = z); c = 1 (r = z, s = x); c = 2 (r = x, s = y)
            e[0][p] = (f1 - g[1][p] + f[2][p + H] - f2) * inv_dx;
            e[1][p] = (f2 - f[2][p + 1] + g[0][p] - f0) * inv_dx;
            e[2][p] = (f0 - f[0][p + H] + f[1][p + 1] - f1) * inv_dx;
        }
    };
    const int pf = (y + 1) * H + x + 1;
    auto F = [&](int c, int dx, int dy, int zp) -> float { return Fs[(zp + 1) % 5][c][pf + dy * H + dx]; };
    auto Ev = [&](int c, int dx, int dy, int zp) -> float { return Es[(zp + 1) % 3][c][pf + dy * H + dx]; };
    fetch_f(-1);
    commit_f(-1);
    fetch_f(0);
    commit_f(0);
    fetch_f(1);
    commit_f(1);
    __syncthreads();
    make_e(-1);
    fetch_f(2);  // ZP >= 2
#pragma unroll
    for (int z = 0; z < ZP; z++) {
        if (z + 2 <= ZP) commit_f(z + 2);  // the slot of plane z - 3
        if (z + 3 <= ZP) fetch_f(z + 3);   // in flight during this plane
        make_e(z);                         // reads f planes z, z + 1; the slot of plane z - 3
        __syncthreads();
        const int o[3][3] = {{1, 0, 0}, {0, 1, 0}, {0, 0, 1}};  // unit offsets e_q
#pragma unroll
        for (int q = 0; q < 3; q++) {
            const int r = (q + 1) % 3, s2 = (q + 2) % 3;
            float v = 0.f;
#pragma unroll
            for (int m = -1; m <= 0; m++) {
                const int ax = m * o[s2][0], ay = m * o[s2][1], az = z + m * o[s2][2];
                v += Ev(r, ax, ay, az) * (F(s2, ax, ay, az) + F(s2, ax + o[q][0], ay + o[q][1], az + o[q][2]));
                const int bx = m * o[r][0], by = m * o[r][1], bz = z + m * o[r][2];
                v -= Ev(s2, bx, by, bz) * (F(r, bx, by, bz) + F(r, bx + o[q][0], by + o[q][1], bz + o[q][2]));
            }
            const size_t i = o0 + q * cs + z * B * B;
            const float gv = v * 0.25f * coef;
            out[i] = gv;
            if (rv) rv[i] = __ldca(in + i) + gv;
        }
    }
}

// Projection tail fused with the gradient: gd_q(n) = (dhat(n + e_q) - dhat(n)) / dx
// on faces (App. A, G), then out1 = rv - gd and optionally out2 = c2 (g - gd);
// gd itself is never stored.  Threads as in k_op: 57 -> 39 us on the 256^3 ring's 1251 blocks, 266
// MB with both outputs (6.8 TB/s, some of it from L2).
template <int B, bool V4>
__global__ void __launch_bounds__(Slab<B>::threads) k_grad_combine(const float *__restrict__ dhat,
                                                                   const float *__restrict__ rv,
                                                                   const float *__restrict__ g,
                                                                   float *__restrict__ out1, float *__restrict__ out2,
                                                                   const int *__restrict__ nbr27, float inv_dx, float c2)
{
    using S = Slab<B>;
    const int blk = blockIdx.x;
    __shared__ int nb[27];
    if (threadIdx.x < 27) nb[threadIdx.x] = nbr27[blk * 27 + threadIdx.x];
    __syncthreads();
    pdl_trigger();
    pdl_wait();  // the previous kernel's output
    const int xq = threadIdx.x % S::Q, y = (threadIdx.x / S::Q) % B, z0 = threadIdx.x / (S::Q * B) * S::ZP;
    const Rows<B, V4> D{dhat, 1, nb};
    constexpr size_t cs = (size_t)B * B * B;
    size_t o = ((size_t)blk * 3 * B + z0) * B * B + y * B + 4 * xq;
    Quad d0 = D.quad(0, xq, y, z0);
#pragma unroll
    for (int k = 0; k < S::ZP; k++, o += B * B) {
        const int z = z0 + k;
        const Quad zq = D.quad(0, xq, y, z + 1), yq = D.quad(0, xq, y + 1, z), xn = D.next_x(d0, 0, xq, y, z);
        Quad gq[3];
#pragma unroll
        for (int i = 0; i < 4; i++) {
            gq[0].v[i] = (xn.v[i] - d0.v[i]) * inv_dx;
            gq[1].v[i] = (yq.v[i] - d0.v[i]) * inv_dx;
            gq[2].v[i] = (zq.v[i] - d0.v[i]) * inv_dx;
        }
#pragma unroll
        for (int q = 0; q < 3; q++) {
            const Quad a = get<V4>(rv + o + q * cs);
            Quad r;
#pragma unroll
            for (int i = 0; i < 4; i++) r.v[i] = a.v[i] - gq[q].v[i];
            put<V4>(out1 + o + q * cs, r);
            if (out2) {
                const Quad b = get<V4>(g + o + q * cs);
#pragma unroll
                for (int i = 0; i < 4; i++) r.v[i] = c2 * (b.v[i] - gq[q].v[i]);
                put<V4>(out2 + o + q * cs, r);
            }
        }
        d0 = zq;
    }
}

// Ring diagnostics (Sec. 6 eq. int_quantities) over the first n_soln blocks of
// the set (D_soln): 15 FP64 sums, acc[0..2] = sum (x cross w) / 2, acc[3] = sum
// u . (x cross w) at cell centres, acc[4] = sum |w|^2 / 2, acc[5] = sum u . w at
// cell centres, acc[6 + 3a + b] = sum (x cross w)_a x_b / 2 (all without dx^3).
// w = C u on edges (computed here in FP64 from u), counted only on D_soln edges;
// edge (q) of cell index n sits at n - e_q / 2, cell n at n - (1,1,1)/2 (units
// of dx); cell values average the 2 faces / 4 edges around the cell.
template <int B>
__global__ void __launch_bounds__(B *B) k_diag(const float *__restrict__ u, const float *__restrict__ w,
                                               const int *__restrict__ nbr27, const int *__restrict__ coords,
                                               int n_soln, double dx, double *__restrict__ acc)
{
    const int blk = blockIdx.x;
    __shared__ int nb[27];
    __shared__ double red[15][B * B / 32];
    if (threadIdx.x < 27) {
        const int n = nbr27[blk * 27 + threadIdx.x];
        nb[threadIdx.x] = n < n_soln ? n : -1;  // w counts on D_soln only
    }
    __syncthreads();
    const int x = threadIdx.x % B, y = threadIdx.x / B;
    Fetch<B> U{u, 3, nbr27 + blk * 27};  // u: the whole set (global table)
    // w = C u at edge (q) of index (px, py, pz) in FP64 (App. A), zero off D_soln
    const double idx = 1.0 / dx;
    auto W = [&](int q, int px, int py, int pz) -> double {
        const int bx = px < 0 ? -1 : (px >= B ? 1 : 0);
        const int by = py < 0 ? -1 : (py >= B ? 1 : 0);
        const int bz = pz < 0 ? -1 : (pz >= B ? 1 : 0);
        if (nb[(bz + 1) * 9 + (by + 1) * 3 + (bx + 1)] < 0) return 0.0;
        const int r = (q + 1) % 3, s2 = (q + 2) % 3;
        const int o[3][3] = {{1, 0, 0}, {0, 1, 0}, {0, 0, 1}};
        return ((double)U(r, px, py, pz) - U(r, px + o[s2][0], py + o[s2][1], pz + o[s2][2]) +
                U(s2, px + o[r][0], py + o[r][1], pz + o[r][2]) - U(s2, px, py, pz)) * idx;
    };
    (void)w;
    const double ox = (double)coords[3 * blk] * B, oy = (double)coords[3 * blk + 1] * B,
                 oz = (double)coords[3 * blk + 2] * B;
    double a[15];
#pragma unroll
    for (int k = 0; k < 15; k++) a[k] = 0.0;
    for (int z = 0; z < B; z++) {
        const double vx = (ox + x) * dx, vy = (oy + y) * dx, vz = (oz + z) * dx;  // vertex of index n
        const double h = 0.5 * dx;
        // own-block edges
        const double w0 = W(0, x, y, z), w1 = W(1, x, y, z), w2 = W(2, x, y, z);
        // edge (q) positions: coordinate q shifted by -1/2
        const double e[3][3] = {{vx - h, vy, vz}, {vx, vy - h, vz}, {vx, vy, vz - h}};  // e[q][a]
        const double wv[3] = {w0, w1, w2};
#pragma unroll
        for (int ai = 0; ai < 3; ai++) {
            const int bi = (ai + 1) % 3, ci = (ai + 2) % 3;
            const double t1 = e[ci][bi] * wv[ci], t2 = e[bi][ci] * wv[bi];  // (x cross w)_a = x_b w_c - x_c w_b
            a[ai] += 0.5 * (t1 - t2);
#pragma unroll
            for (int bb = 0; bb < 3; bb++) a[6 + 3 * ai + bb] += 0.5 * (t1 * e[ci][bb] - t2 * e[bi][bb]);
        }
        a[4] += 0.5 * (w0 * w0 + w1 * w1 + w2 * w2);
        // cell-centred u and w
        const double uc[3] = {0.5 * ((double)U(0, x, y, z) + U(0, x - 1, y, z)),
                              0.5 * ((double)U(1, x, y, z) + U(1, x, y - 1, z)),
                              0.5 * ((double)U(2, x, y, z) + U(2, x, y, z - 1))};
        const double wc[3] = {
            0.25 * ((double)w0 + W(0, x, y - 1, z) + W(0, x, y, z - 1) + W(0, x, y - 1, z - 1)),
            0.25 * ((double)w1 + W(1, x, y, z - 1) + W(1, x - 1, y, z) + W(1, x - 1, y, z - 1)),
            0.25 * ((double)w2 + W(2, x - 1, y, z) + W(2, x, y - 1, z) + W(2, x - 1, y - 1, z))};
        const double px = vx - h, py = vy - h, pz = vz - h;
        const double xw[3] = {py * wc[2] - pz * wc[1], pz * wc[0] - px * wc[2], px * wc[1] - py * wc[0]};
        a[3] += uc[0] * xw[0] + uc[1] * xw[1] + uc[2] * xw[2];
        a[5] += uc[0] * wc[0] + uc[1] * wc[1] + uc[2] * wc[2];
    }
    // block reduction: warp shuffles, then one partial per warp in shared memory
    const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
#pragma unroll
    for (int k = 0; k < 15; k++) {
        double v = a[k];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (lane == 0) red[k][warp] = v;
    }
    __syncthreads();
    if (threadIdx.x < 15) {
        double v = 0.0;
        for (int i = 0; i < B * B / 32; i++) v += red[threadIdx.x][i];
        atomicAdd(acc + threadIdx.x, v);
    }
}

// Regrid weights' raw maxima (Sec. 5 eq. weight_fun): mu[b] = max |w| (3 edge
// components) and nu[b] = max |q| (cells) over block b, leaving out the cells within
// RIM = 3 cells of a block outside the set: the masked curl is spurious on the last
// layer, and N~ and G^T carry that one cell further each.
template <int B>
__global__ void __launch_bounds__(B *B) k_block_max(const float *__restrict__ w, const float *__restrict__ q,
                                                    const int *__restrict__ nbr27, float *__restrict__ mu,
                                                    float *__restrict__ nu)
{
    const int blk = blockIdx.x;
    __shared__ int nb[27];
    __shared__ float red[2][B * B / 32];
    if (threadIdx.x < 27) nb[threadIdx.x] = nbr27[blk * 27 + threadIdx.x];
    __syncthreads();
    const int x = threadIdx.x % B, y = threadIdx.x / B;
    const size_t b3 = (size_t)B * B * B;
    float m1 = 0.f, m2 = 0.f;
    for (int z = 0; z < B; z++) {
        bool inner = true;
        constexpr int RIM = 3;
        for (int oz = (z < RIM ? -1 : 0); oz <= (z >= B - RIM ? 1 : 0); oz++)
            for (int oy = (y < RIM ? -1 : 0); oy <= (y >= B - RIM ? 1 : 0); oy++)
                for (int ox = (x < RIM ? -1 : 0); ox <= (x >= B - RIM ? 1 : 0); ox++)
                    if (nb[(oz + 1) * 9 + (oy + 1) * 3 + (ox + 1)] < 0) inner = false;
        if (!inner) continue;
        const size_t o = (size_t)z * B * B + y * B + x;
#pragma unroll
        for (int c = 0; c < 3; c++) m1 = fmaxf(m1, fabsf(__ldg(w + ((size_t)blk * 3 + c) * b3 + o)));
        m2 = fmaxf(m2, fabsf(__ldg(q + (size_t)blk * b3 + o)));
    }
    for (int off = 16; off > 0; off >>= 1) {
        m1 = fmaxf(m1, __shfl_down_sync(0xffffffffu, m1, off));
        m2 = fmaxf(m2, __shfl_down_sync(0xffffffffu, m2, off));
    }
    const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
    if (lane == 0) {
        red[0][warp] = m1;
        red[1][warp] = m2;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        float m = 0.f;
        for (int i = 0; i < B * B / 32; i++) m = fmaxf(m, red[threadIdx.x][i]);
        (threadIdx.x == 0 ? mu : nu)[blk] = m;
    }
}

// Zero a vector field on the cells within RIM = 3 cells of a block outside the set
// (the mask edge's contaminated layer; the same cells the regrid weights leave out).
template <int B>
__global__ void __launch_bounds__(B *B) k_zero_rim(float *__restrict__ f, const int *__restrict__ nbr27)
{
    const int blk = blockIdx.x;
    __shared__ int nb[27];
    if (threadIdx.x < 27) nb[threadIdx.x] = nbr27[blk * 27 + threadIdx.x];
    __syncthreads();
    const int x = threadIdx.x % B, y = threadIdx.x / B;
    const size_t b3 = (size_t)B * B * B;
    constexpr int RIM = 3;
    for (int z = 0; z < B; z++) {
        bool inner = true;
        for (int oz = (z < RIM ? -1 : 0); oz <= (z >= B - RIM ? 1 : 0); oz++)
            for (int oy = (y < RIM ? -1 : 0); oy <= (y >= B - RIM ? 1 : 0); oy++)
                for (int ox = (x < RIM ? -1 : 0); ox <= (x >= B - RIM ? 1 : 0); ox++)
                    if (nb[(oz + 1) * 9 + (oy + 1) * 3 + (ox + 1)] < 0) inner = false;
        if (inner) continue;
        const size_t o = (size_t)z * B * B + y * B + x;
#pragma unroll
        for (int c = 0; c < 3; c++) f[((size_t)blk * 3 + c) * b3 + o] = 0.f;
    }
}

// out = sum_t c_t x_t over n floats (up to 4 terms; null x_t skipped).  out may
// alias an input (each element is read and written by the same thread), so no
// __restrict__ and no read-only-cache loads here.
__global__ void k_lincomb(float *out, int64_t n, const float *x0, float c0, const float *x1, float c1,
                          const float *x2, float c2, const float *x3, float c3)
{
    const int64_t n4 = n / 4;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n4; i += (int64_t)gridDim.x * blockDim.x) {
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
        auto acc = [&](const float *x, float c) {
            if (!x) return;
            const float4 v = reinterpret_cast<const float4 *>(x)[i];
            a.x = fmaf(c, v.x, a.x);
            a.y = fmaf(c, v.y, a.y);
            a.z = fmaf(c, v.z, a.z);
            a.w = fmaf(c, v.w, a.w);
        };
        acc(x0, c0);
        acc(x1, c1);
        acc(x2, c2);
        acc(x3, c3);
        reinterpret_cast<float4 *>(out)[i] = a;
    }
}

// out[i] = in[idx[i]] block by block ([n][ncomp][B^3] each)
__global__ void k_gather_blocks(const float *__restrict__ in, float *__restrict__ out, const int *__restrict__ idx,
                                int block_floats)
{
    const int i = blockIdx.x;
    const float4 *src = reinterpret_cast<const float4 *>(in + (size_t)__ldg(idx + i) * block_floats);
    float4 *dst = reinterpret_cast<float4 *>(out + (size_t)i * block_floats);
    for (int t = threadIdx.x; t < block_floats / 4; t += blockDim.x) dst[t] = __ldg(src + t);
}

}  // namespace

lgf_status op_launch(int op, int B, int nblk, const int *d_nbr27, const unsigned char *d_keep, const float *in,
                     float *out, double dx, double coef, const double uinf[3], cudaStream_t s, float *out2)
{
    if (out2 && op != 4) {
        set_error("a second output is only for the nonlinear term");
        return LGF_ERR_ARG;
    }
    const float inv_dx = (float)(1.0 / dx);
    const float u0 = uinf ? (float)uinf[0] : 0.f, u1 = uinf ? (float)uinf[1] : 0.f, u2 = uinf ? (float)uinf[2] : 0.f;
    const float cf = (float)coef;
    // 1251 blocks of 16^3 (the 256^3 ring): curl 55 -> 23 us and curl^T 58 -> 23 us for 123 MB (5.3
    // TB/s), G^T 22 -> 10-17 us and G 12 us for 82 MB, against the thread-per-column form
    const bool v4 = (((uintptr_t)in | (uintptr_t)out) & 15) == 0;
#define LGF_OPCASE(BB, OPV)                                                                                   \
    case OPV:                                                                                                 \
        if (OPV != 1)                                                                                         \
            LGF_CUDA_TRY(launch_pdl(v4 ? k_op<BB, OPV, true> : k_op<BB, OPV, false>, dim3(nblk),              \
                                    dim3(Slab<BB>::threads), s, in, out, d_nbr27, inv_dx));                  \
        else if (v4) k_op<BB, OPV, true><<<nblk, Slab<BB>::threads, 0, s>>>(in, out, d_nbr27, inv_dx);        \
        else k_op<BB, OPV, false><<<nblk, Slab<BB>::threads, 0, s>>>(in, out, d_nbr27, inv_dx);               \
        break;
#define LGF_OPSWITCH(BB)                                                                                      \
    switch (op) {                                                                                             \
        LGF_OPCASE(BB, 0)                                                                                     \
        LGF_OPCASE(BB, 1)                                                                                     \
        LGF_OPCASE(BB, 2)                                                                                     \
        LGF_OPCASE(BB, 3)                                                                                     \
        case 4:                                                                                               \
            LGF_CUDA_TRY(launch_pdl(k_nonlinear<BB>, dim3(nblk * (BB >= 16 ? 2 : 1)), dim3(BB * BB), s, in,   \
                                    out, d_nbr27, d_keep, inv_dx, cf, u0, u1, u2, out2));                     \
            break;                                                                                            \
        default: set_error("unknown operator %d", op); return LGF_ERR_ARG;                                    \
    }
    if (B == 8) {
        LGF_OPSWITCH(8)
    } else if (B == 16) {
        LGF_OPSWITCH(16)
    } else {
        set_error("operators support B in {8, 16} (got %d)", B);
        return LGF_ERR_ARG;
    }
#undef LGF_OPSWITCH
#undef LGF_OPCASE
    LGF_LAUNCH_CHECK("local operator");
    return LGF_OK;
}

lgf_status lincomb_launch(float *out, int64_t n, const float *x0, double c0, const float *x1, double c1, const float *x2,
                          double c2, const float *x3, double c3, cudaStream_t s)
{
    if (n % 4 != 0) {
        set_error("lincomb length %lld not a multiple of 4", (long long)n);
        return LGF_ERR_ARG;
    }
    const int threads = 256;
    const int blocks = (int)std::min<int64_t>((n / 4 + threads - 1) / threads, 152 * 16);
    k_lincomb<<<blocks, threads, 0, s>>>(out, n, x0, (float)c0, x1, (float)c1, x2, (float)c2, x3, (float)c3);
    LGF_LAUNCH_CHECK("lincomb");
    return LGF_OK;
}

lgf_status diag_launch(int B, int n_soln, const int *d_nbr27, const int *d_coords, const float *u, const float *w,
                       double dx, double *d_acc, cudaStream_t s)
{
    if (B == 8)
        k_diag<8><<<n_soln, 64, 0, s>>>(u, w, d_nbr27, d_coords, n_soln, dx, d_acc);
    else if (B == 16)
        k_diag<16><<<n_soln, 256, 0, s>>>(u, w, d_nbr27, d_coords, n_soln, dx, d_acc);
    else {
        set_error("operators support B in {8, 16} (got %d)", B);
        return LGF_ERR_ARG;
    }
    LGF_LAUNCH_CHECK("diagnostics");
    return LGF_OK;
}

lgf_status block_max_launch(int B, int nblk, const int *d_nbr27, const float *w, const float *q, float *mu, float *nu,
                            cudaStream_t s)
{
    if (B == 8)
        k_block_max<8><<<nblk, 64, 0, s>>>(w, q, d_nbr27, mu, nu);
    else if (B == 16)
        k_block_max<16><<<nblk, 256, 0, s>>>(w, q, d_nbr27, mu, nu);
    else {
        set_error("operators support B in {8, 16} (got %d)", B);
        return LGF_ERR_ARG;
    }
    LGF_LAUNCH_CHECK("block_max");
    return LGF_OK;
}

lgf_status zero_rim_launch(int B, int nblk, const int *d_nbr27, float *f, cudaStream_t s)
{
    if (B == 8)
        k_zero_rim<8><<<nblk, 64, 0, s>>>(f, d_nbr27);
    else if (B == 16)
        k_zero_rim<16><<<nblk, 256, 0, s>>>(f, d_nbr27);
    else {
        set_error("operators support B in {8, 16} (got %d)", B);
        return LGF_ERR_ARG;
    }
    LGF_LAUNCH_CHECK("zero_rim");
    return LGF_OK;
}

lgf_status grad_combine_launch(int B, int nblk, const int *d_nbr27, const float *dhat, const float *rv, const float *g,
                               float *out1, float *out2, double c2, double dx, cudaStream_t s)
{
    const float inv_dx = (float)(1.0 / dx);
    const bool v4 = (((uintptr_t)dhat | (uintptr_t)rv | (uintptr_t)g | (uintptr_t)out1 | (uintptr_t)out2) & 15) == 0;
#define LGF_GC(BB, V)                                                                                             \
    k_grad_combine<BB, V><<<nblk, Slab<BB>::threads, 0, s>>>(dhat, rv, g, out1, out2, d_nbr27, inv_dx, (float)c2)
    if (B == 8) {
        if (v4) LGF_GC(8, true);
        else LGF_GC(8, false);
    } else if (B == 16) {
        if (v4) LGF_GC(16, true);
        else LGF_GC(16, false);
    } else {
        set_error("operators support B in {8, 16} (got %d)", B);
        return LGF_ERR_ARG;
    }
#undef LGF_GC
    LGF_LAUNCH_CHECK("grad_combine");
    return LGF_OK;
}

lgf_status gather_launch(const float *in, float *out, const int *d_idx, int n, int block_floats, cudaStream_t s)
{
    if (n == 0) return LGF_OK;
    k_gather_blocks<<<n, 256, 0, s>>>(in, out, d_idx, block_floats);
    LGF_LAUNCH_CHECK("gather");
    return LGF_OK;
}

}  // namespace lgf
