// Kernels of the three-pass Poisson solve (plane.hpp).
//
// Lengths.  Every transform is an in-place two-factor DFT of length M = R1 * R2 in shared
// memory: a radix-R1 stage over elements b + m R2 (b < R2), twiddles w_M^(b q), a radix-R2
// stage over the R2 neighbours q R2 + k2.  Frequency q + R1 k2 ends at position q R2 + k2; the
// inverse runs the stages in reverse and returns to natural order, so nothing is permuted
// and a stage's reads and writes are the same slots of the same thread.  The padded lengths
// are multiples of M:
//   x  Nx = 2 Mx: a real row of Nx points as Mx complex ones (even, odd), split by w_Nx^k.
//   y  Ny = Dy My: thread blocks take the frequencies ky = Dy k + r of one residue r.  Their
//      transform has length My on the folded, twisted row sum_j x[n + j My] w_Ny^(r (n + j My)),
//      so a residue's plane [My][z] fits shared memory; the inverse gives My values v_r[n mod My]
//      per row, and the residues' thread blocks, a cluster, sum conj(w_Ny^(r p)) v_r[p mod My]
//      through distributed shared memory.
//   z  Nz = 2 Mz with Mz >= both boxes' extents: even and odd frequencies one after the other
//      (the odd ones on the row twisted by w_Nz^n), each a length-Mz transform, times the
//      spectrum, inverse; the two results add up in registers.
// One launch therefore holds what took three passes over [z][ky][kx] arrays of twice the
// volume: it reads the x-transformed rows Dy times (from L2) and writes the target rows once.
#pragma once
#include "fft.cuh"
#include "plane.hpp"

namespace lgf {
namespace {

using C = cx<float>;

// A complex value as one packed register pair (re, im): a complex sum, difference or real
// multiple is one .f32x2 instruction, which takes a third off the arithmetic of the in-register
// DFTs; rotations by -i and general twiddles work on the halves.
using V = fft::f32x2;
__device__ __forceinline__ V v_of(C a) { return fft::pk2(a.x, a.y); }
__device__ __forceinline__ C c_of(V a)
{
    C c;
    fft::unpk2(a, c.x, c.y);
    return c;
}
__device__ __forceinline__ V v_ld(const C *p) { return V{*reinterpret_cast<const unsigned long long *>(p)}; }
__device__ __forceinline__ void v_st(C *p, V a) { *reinterpret_cast<unsigned long long *>(p) = a.r; }
constexpr unsigned long long kZero = 0;
// u -+ i v
__device__ __forceinline__ V sub_i(V u, V v)
{
    const C a = c_of(u), b = c_of(v);
    return fft::pk2(a.x + b.y, a.y - b.x);
}
__device__ __forceinline__ V add_i(V u, V v)
{
    const C a = c_of(u), b = c_of(v);
    return fft::pk2(a.x - b.y, a.y + b.x);
}
// a w, a conj(w), the fused products spelled out: which of the two products is rounded must not
// depend on the kernel it is inlined in (grouped and single launches agree bitwise)
__device__ __forceinline__ C mul(C a, C w) { return {fmaf(a.x, w.x, -(a.y * w.y)), fmaf(a.x, w.y, a.y * w.x)}; }
__device__ __forceinline__ C mulc(C a, C w) { return {fmaf(a.x, w.x, a.y * w.y), fmaf(a.y, w.x, -(a.x * w.y))}; }
__device__ __forceinline__ V v_mul(V a, C w) { return v_of(mul(c_of(a), w)); }
__device__ __forceinline__ V v_mulc(V a, C w) { return v_of(mulc(c_of(a), w)); }
__device__ __forceinline__ V v_mul(V a, float2 w) { return v_mul(a, C{w.x, w.y}); }
__device__ __forceinline__ V v_mulc(V a, float2 w) { return v_mulc(a, C{w.x, w.y}); }
__device__ __forceinline__ C ld(const float2 *p) { return {p->x, p->y}; }
// data of an earlier pass: through L2, since under programmatic dependent launch this SM's L1 may
// still hold a line from before that pass wrote it
__device__ __forceinline__ C ld_l2(const C *p)
{
    const float2 v = __ldcg(reinterpret_cast<const float2 *>(p));
    return {v.x, v.y};
}

// ---------------------------------------------------------------------------
// in-register DFTs of length R <= 16
// ---------------------------------------------------------------------------
// cos and sin of 2 pi j / Q, j < Q, at compile time (Taylor series of the reduced angle)
constexpr double ct_cos(double x)
{
    double t = 1.0, s = 1.0;
    for (int k = 1; k < 24; k++) {
        t *= -x * x / ((2 * k - 1) * (2 * k));
        s += t;
    }
    return s;
}
constexpr double ct_sin(double x)
{
    double t = x, s = x;
    for (int k = 1; k < 24; k++) {
        t *= -x * x / ((2 * k) * (2 * k + 1));
        s += t;
    }
    return s;
}
template <int Q>
struct Roots {
    double c[Q] = {}, s[Q] = {};
    constexpr Roots()
    {
        for (int j = 0; j < Q; j++) {
            const double x = 2.0 * 3.14159265358979323846 * (2 * j <= Q ? j : j - Q) / Q;
            c[j] = ct_cos(x);
            s[j] = ct_sin(x);
        }
    }
};

// Odd length Q by the symmetric sums x_m + x_(Q-m), x_m - x_(Q-m).  A smooth field's spectrum lies in
// the lowest frequencies, in an inverse transform x_0 and x_(+-1) and, behind the index map of a
// prime-factor product (UP), x_0 and x_(+-H).  Those come last, so that the partial sums that are
// rounded stay small: from x_0 on, the point differences along x of a 200 x 16 x 16 solve (13-point
// sums) were off by 5.9e-6 relative, in this order by 5.1e-6 (the five passes: 4.8e-6); same time.
template <int Q, bool INV, bool UP = false>
__device__ __forceinline__ void dft_sym(V (&x)[Q])
{
    constexpr Roots<Q> W{};
    constexpr int H = (Q - 1) / 2;
    V t[H], d[H];
#pragma unroll
    for (int m = 0; m < H; m++) {
        t[m] = x[m + 1] + x[Q - 1 - m];
        d[m] = x[m + 1] - x[Q - 1 - m];
    }
    const V x0 = x[0];
    V s = t[UP ? 0 : H - 1];
#pragma unroll
    for (int i = 1; i < H; i++) s = s + t[UP ? i : H - 1 - i];
    x[0] = s + x0;
#pragma unroll
    for (int k = 1; k <= H; k++) {
        V a, b;
#pragma unroll
        for (int i = 0; i < H; i++) {
            const int m = UP ? i + 1 : H - i;
            const V c = fft::bc2((float)W.c[(k * m) % Q]), sn = fft::bc2((float)W.s[(k * m) % Q]);
            a = i == 0 ? c * t[m - 1] : fft::fma(c, t[m - 1], a);
            b = i == 0 ? sn * d[m - 1] : fft::fma(sn, d[m - 1], b);
        }
        a = a + x0;
        x[k] = INV ? add_i(a, b) : sub_i(a, b);
        x[Q - k] = INV ? sub_i(a, b) : add_i(a, b);
    }
}

// length 4 of (a, b, c, d) in place; HALF: c = d = 0
template <bool INV, bool HALF = false>
__device__ __forceinline__ void dft4(V &a, V &b, V &c, V &d)
{
    const V t0 = HALF ? a : a + c, t1 = HALF ? a : a - c, t2 = HALF ? b : b + d, t3 = HALF ? b : b - d;
    a = t0 + t2;
    c = t0 - t2;
    b = INV ? add_i(t1, t3) : sub_i(t1, t3);
    d = INV ? sub_i(t1, t3) : add_i(t1, t3);
}

// v times w_16^J (its conjugate for the inverse)
template <int J, bool INV>
__device__ __forceinline__ V twiddle16(V v)
{
    constexpr float h = 0.70710678118654752440f;
    const C a = c_of(v);
    if constexpr (J == 0) return v;
    else if constexpr (J == 4) return INV ? fft::pk2(-a.y, a.x) : fft::pk2(a.y, -a.x);
    else if constexpr (J == 2)
        return fft::bc2(h) * (INV ? fft::pk2(a.x - a.y, a.y + a.x) : fft::pk2(a.x + a.y, a.y - a.x));
    else if constexpr (J == 6)
        return fft::bc2(h) * (INV ? fft::pk2(-a.x - a.y, a.x - a.y) : fft::pk2(a.y - a.x, -a.x - a.y));
    else {
        constexpr Roots<16> W{};
        constexpr float c = (float)W.c[J], sn = INV ? (float)W.s[J] : -(float)W.s[J];
        return fft::pk2(fmaf(a.x, c, -(a.y * sn)), fmaf(a.x, sn, a.y * c));
    }
}

// Length R of a[0 .. R).  16 = 4 x 4; 8 = 4 + 4; 6, 10, 12, 14, 15 as prime-factor products
// (index maps by the Chinese remainder theorem, no twiddles); odd lengths by symmetric sums.
// HALF: a[m] = 0 for m >= (R + 1) / 2.
template <int R, bool INV, bool HALF = false>
__device__ __forceinline__ void dft(V (&a)[R])
{
    if constexpr (R == 4) {
        dft4<INV, HALF>(a[0], a[1], a[2], a[3]);
    } else if constexpr (R == 8) {
        V e[4] = {a[0], a[2], a[4], a[6]}, o[4] = {a[1], a[3], a[5], a[7]};
        dft4<INV, HALF>(e[0], e[1], e[2], e[3]);
        dft4<INV, HALF>(o[0], o[1], o[2], o[3]);
        a[0] = e[0] + o[0];
        a[4] = e[0] - o[0];
        a[2] = INV ? add_i(e[2], o[2]) : sub_i(e[2], o[2]);
        a[6] = INV ? sub_i(e[2], o[2]) : add_i(e[2], o[2]);
        // w_8 o_1 = h (s - i) o: the scale joins the sum
        const C p = c_of(o[1]), q = c_of(o[3]);
        const V t1 = INV ? fft::pk2(p.x - p.y, p.y + p.x) : fft::pk2(p.x + p.y, p.y - p.x);
        const V t3 = INV ? fft::pk2(q.x + q.y, q.y - q.x) : fft::pk2(q.x - q.y, q.y + q.x);  // -w_8^3 o_3 / h
        const V h = fft::bc2(0.70710678118654752440f), nh = fft::bc2(-0.70710678118654752440f);
        a[1] = fft::fma(h, t1, e[1]);
        a[5] = fft::fma(nh, t1, e[1]);
        a[3] = fft::fma(nh, t3, e[3]);
        a[7] = fft::fma(h, t3, e[3]);
    } else if constexpr (R == 16) {
#pragma unroll
        for (int n = 0; n < 4; n++) dft4<INV, HALF>(a[n], a[n + 4], a[n + 8], a[n + 12]);
        // a[n2 + 4 k1]: twiddles w_16^(n2 k1), then length 4 over n2
        a[5] = twiddle16<1, INV>(a[5]);
        a[6] = twiddle16<2, INV>(a[6]);
        a[7] = twiddle16<3, INV>(a[7]);
        a[9] = twiddle16<2, INV>(a[9]);
        a[10] = twiddle16<4, INV>(a[10]);
        a[11] = twiddle16<6, INV>(a[11]);
        a[13] = twiddle16<3, INV>(a[13]);
        a[14] = twiddle16<6, INV>(a[14]);
        a[15] = twiddle16<9, INV>(a[15]);
#pragma unroll
        for (int k = 0; k < 4; k++) dft4<INV>(a[4 * k], a[4 * k + 1], a[4 * k + 2], a[4 * k + 3]);
        // X[k1 + 4 k2] is at 4 k1 + k2
#pragma unroll
        for (int i = 0; i < 4; i++)
#pragma unroll
            for (int k = i + 1; k < 4; k++) {
                const V t = a[4 * i + k];
                a[4 * i + k] = a[4 * k + i];
                a[4 * k + i] = t;
            }
    } else if constexpr (R == 12) {
        V u[3][4];
#pragma unroll
        for (int n2 = 0; n2 < 4; n2++) {
            V x[3] = {a[(3 * n2) % 12], a[(4 + 3 * n2) % 12], a[(8 + 3 * n2) % 12]};
            dft_sym<3, INV>(x);
#pragma unroll
            for (int k = 0; k < 3; k++) u[k][n2] = x[k];
        }
#pragma unroll
        for (int k1 = 0; k1 < 3; k1++) {
            dft4<INV>(u[k1][0], u[k1][1], u[k1][2], u[k1][3]);
#pragma unroll
            for (int k2 = 0; k2 < 4; k2++) a[(4 * k1 + 9 * k2) % 12] = u[k1][k2];
        }
    } else if constexpr (R == 6 || R == 10 || R == 14) {
        constexpr int Q = R / 2;
        V u[2][Q];
#pragma unroll
        for (int n2 = 0; n2 < Q; n2++) {
            const V p = a[(2 * n2) % R], q = a[(Q + 2 * n2) % R];
            u[0][n2] = p + q;
            u[1][n2] = p - q;
        }
        dft_sym<Q, INV, true>(u[0]);
        dft_sym<Q, INV, true>(u[1]);
#pragma unroll
        for (int k1 = 0; k1 < 2; k1++)
#pragma unroll
            for (int k2 = 0; k2 < Q; k2++) a[(Q * k1 + (Q + 1) * k2) % R] = u[k1][k2];
    } else if constexpr (R == 15) {
        V u[3][5];
#pragma unroll
        for (int n2 = 0; n2 < 5; n2++) {
            V x[3] = {a[(3 * n2) % 15], a[(5 + 3 * n2) % 15], a[(10 + 3 * n2) % 15]};
            dft_sym<3, INV>(x);
#pragma unroll
            for (int k = 0; k < 3; k++) u[k][n2] = x[k];
        }
#pragma unroll
        for (int k1 = 0; k1 < 3; k1++) {
            dft_sym<5, INV, true>(u[k1]);
#pragma unroll
            for (int k2 = 0; k2 < 5; k2++) a[(10 * k1 + 6 * k2) % 15] = u[k1][k2];
        }
    } else {
        dft_sym<R, INV>(a);
    }
}

// One in-place butterfly of radix R on p[i * stride]: DFT, then element i times tw[i * ts]
// (TW = 1) or its conjugate (TW = 2).
template <int R, bool INV, int TW>
__device__ __forceinline__ void butterfly_at(C *p, int stride, const float2 *tw, int ts)
{
    V a[R];
#pragma unroll
    for (int i = 0; i < R; i++) a[i] = v_ld(p + i * stride);
    dft<R, INV>(a);
#pragma unroll
    for (int i = 0; i < R; i++) {
        if (TW == 1 && i > 0) a[i] = v_mul(a[i], ld(tw + i * ts));
        if (TW == 2 && i > 0) a[i] = v_mulc(a[i], ld(tw + i * ts));
        v_st(p + i * stride, a[i]);
    }
}

// copy n float2 of a table to shared memory
__device__ __forceinline__ void table_to_smem(float2 *s, const float2 *g, int n)
{
    for (int i = threadIdx.x; i < n; i += blockDim.x) s[i] = __ldg(g + i);
}

// ---------------------------------------------------------------------------
// x passes: 32 rows per thread block, lane = row, warps over butterflies.  The rows run along z, so
// that the transposed arrays [kx][y][z] move in 256-byte pieces; the block rows move in 64-byte
// ones.  Latency-bound (50 % issue): 31 and 36 us on the 256^3 ring's scalar solve against 32 and
// 47 us for the lane-per-element passes, 21 and 25 us on the 128^3 ring (three components).
// ---------------------------------------------------------------------------
// (pitch 34: rows of 32 consecutive entries for the stages, and 8 entries of 2 rows apart for the
// gather and the scatter, both conflict-free)
constexpr int PX_ROWS = 32, PX_THREADS = 256, PX_PITCH = 34;

template <int M>
__host__ __device__ constexpr size_t px_smem()
{
    return (size_t)(M * PX_PITCH + M + M / 2 + 1 + 1) * sizeof(float2) + (size_t)PX_ROWS * (M / 4) * sizeof(int);
}

// position of frequency k in the in-place order
template <int M>
__device__ __forceinline__ int pos_of(int k)
{
    constexpr int R1 = plane_r1(M), R2 = plane_r2(M);
    return (k % R1) * R2 + k / R1;
}

template <int M>
__device__ __forceinline__ void px_fwd_body(const PlaneGeom &g, const float *__restrict__ src, C *__restrict__ out,
                                            int tile, int c)
{
    constexpr int R1 = plane_r1(M), R2 = plane_r2(M), NW = PX_THREADS / 32;
    extern __shared__ float2 sm_px[];
    C *buf = reinterpret_cast<C *>(sm_px);
    float2 *tw = sm_px + M * PX_PITCH, *w2 = tw + M;
    int *lut = reinterpret_cast<int *>(w2 + M / 2 + 2);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nrows = g.Es[1] * g.Es[2], nbx = g.nbS[0], lB = g.lB, mB = g.B - 1;
    table_to_smem(tw, g.st[0], M);
    table_to_smem(w2, g.w2[0], M / 2 + 1);
    int mine = 0;
    for (int q = threadIdx.x; q < PX_ROWS * nbx; q += PX_THREADS) {
        const int l = q / nbx, xb = q - l * nbx, row = tile * PX_ROWS + l;
        int b = -1;
        if (row < nrows) {
            const int y = row / g.Es[2], z = row - y * g.Es[2];
            b = __ldg(g.src_lut + ((z >> lB) * g.nbS[1] + (y >> lB)) * nbx + xb);
            // offset of the row's first cell in the source array, or -1
            if (b >= 0) b = (b << 10) | ((z & mB) * g.B + (y & mB));
        }
        lut[q] = b;
        mine |= b >= 0;
    }
    pdl_trigger();
    pdl_wait();  // the producer of src is complete
    const int row = tile * PX_ROWS + lane;
    C *o = out + (size_t)c * g.KX * nrows + row;
    if (!__syncthreads_or(mine)) {  // no source block meets these rows
        if (row < nrows)
            for (int k = warp; k <= M; k += NW) o[(size_t)k * nrows] = {0.f, 0.f};
        return;
    }
    const int hx = g.Es[0] / 2;  // complex points of a row, <= M / 2
    const bool al = (reinterpret_cast<size_t>(src) & 7) == 0;
    const int cc = g.c0 + c;
    // 8 lanes per row: 64-byte pieces of the block rows
    const int l = threadIdx.x >> 3;
#pragma unroll 4
    for (int m = threadIdx.x & 7; m < hx; m += 8) {
        const int b = lut[l * nbx + ((2 * m) >> lB)];
        C v = {0.f, 0.f};
        if (b >= 0) {
            const float *p = src + ((size_t)((b >> 10) * g.ncomp + cc) << (3 * lB)) + ((b & 1023) << lB) + ((2 * m) & mB);
            if (al) v = ld_l2(reinterpret_cast<const C *>(p));
            else v = {__ldcg(p), __ldcg(p + 1)};
        }
        buf[m * PX_PITCH + l] = v;
    }
    __syncthreads();
    C *col = buf + lane;
    for (int b = warp; b < R2; b += NW) {
        V a[R1];
#pragma unroll
        for (int m = 0; m < R1; m++) {
            a[m] = V{kZero};
            if (m < (R1 + 1) / 2 && b + m * R2 < hx) a[m] = v_ld(col + (b + m * R2) * PX_PITCH);
        }
        dft<R1, false, true>(a);
#pragma unroll
        for (int q = 0; q < R1; q++) {
            if (q > 0) a[q] = v_mul(a[q], ld(tw + b * R1 + q));
            v_st(col + (b + q * R2) * PX_PITCH, a[q]);
        }
    }
    __syncthreads();
    for (int q = warp; q < R1; q += NW) butterfly_at<R2, false, 0>(col + q * R2 * PX_PITCH, PX_PITCH, nullptr, 0);
    __syncthreads();
    if (row >= nrows) return;
    // F_k = E + w^k O, F_(M-k) = conj(E - w^k O) from the transform of (even, odd) pairs
    for (int k = warp; k <= M / 2; k += NW) {
        const C u = col[pos_of<M>(k) * PX_PITCH], v = col[pos_of<M>(k == 0 ? 0 : M - k) * PX_PITCH];
        const C e = {0.5f * (u.x + v.x), 0.5f * (u.y - v.y)};
        const C od = {0.5f * (u.y + v.y), 0.5f * (v.x - u.x)};
        const C t = mul(od, ld(w2 + k));
        o[(size_t)k * nrows] = e + t;
        o[(size_t)(M - k) * nrows] = {e.x - t.x, t.y - e.y};
    }
}

template <int M>
__device__ __forceinline__ void px_inv_body(const PlaneGeom &g, const C *__restrict__ in, float *__restrict__ dst,
                                            int tile, int c)
{
    constexpr int R1 = plane_r1(M), R2 = plane_r2(M), NW = PX_THREADS / 32;
    extern __shared__ float2 sm_px[];
    C *buf = reinterpret_cast<C *>(sm_px);
    float2 *tw = sm_px + M * PX_PITCH, *w2 = tw + M;
    int *lut = reinterpret_cast<int *>(w2 + M / 2 + 2);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nrows = g.Et[1] * g.Et[2], nbx = g.nbT[0], lB = g.lB, mB = g.B - 1;
    table_to_smem(tw, g.st[0], M);
    table_to_smem(w2, g.w2[0], M / 2 + 1);
    int mine = 0;
    for (int q = threadIdx.x; q < PX_ROWS * nbx; q += PX_THREADS) {
        const int l = q / nbx, xb = q - l * nbx, r = tile * PX_ROWS + l;
        int b = -1;
        if (r < nrows) {
            const int y = r / g.Et[2], z = r - y * g.Et[2];
            b = __ldg(g.dst_lut + ((z >> lB) * g.nbT[1] + (y >> lB)) * nbx + xb);
            if (b >= 0) b = (b << 10) | ((z & mB) * g.B + (y & mB));
        }
        lut[q] = b;
        mine |= b >= 0;
    }
    if (!__syncthreads_or(mine)) return;  // no target block meets these rows
    const int row = tile * PX_ROWS + lane;
    const bool ok = row < nrows;
    pdl_trigger();
    pdl_wait();  // the yz pass is complete
    const C *p = in + (size_t)c * g.KX * nrows + (ok ? row : 0);
    C *col = buf + lane;
#pragma unroll 4
    for (int k = warp; k <= M / 2; k += NW) {
        const C u = ld_l2(p + (size_t)k * nrows), v = ld_l2(p + (size_t)(M - k) * nrows);
        const C e = {0.5f * (u.x + v.x), 0.5f * (u.y - v.y)};
        const C t = {0.5f * (u.x - v.x), 0.5f * (u.y + v.y)};
        const C od = mulc(t, ld(w2 + k));
        col[pos_of<M>(k) * PX_PITCH] = {e.x - od.y, e.y + od.x};
        if (k > 0) col[pos_of<M>(M - k) * PX_PITCH] = {e.x + od.y, od.x - e.y};
    }
    __syncthreads();
    for (int q = warp; q < R1; q += NW) butterfly_at<R2, true, 2>(col + q * R2 * PX_PITCH, PX_PITCH, tw + q, R1);
    __syncthreads();
    for (int b = warp; b < R2; b += NW) butterfly_at<R1, true, 0>(col + b * PX_PITCH, R2 * PX_PITCH, nullptr, 0);
    __syncthreads();
    const int hx = g.Et[0] / 2;
    const bool al = (reinterpret_cast<size_t>(dst) & 7) == 0;
    const int cc = g.c0 + c;
    const int l = threadIdx.x >> 3;
#pragma unroll 4
    for (int xh = threadIdx.x & 7; xh < hx; xh += 8) {
        const int b = lut[l * nbx + ((2 * xh) >> lB)];
        if (b < 0) continue;
        int m = xh + g.d0[0] / 2;  // d0 is a multiple of B; |position| < Nx / 2
        if (m < 0) m += M;
        const C v = buf[m * PX_PITCH + l];
        float *q = dst + ((size_t)((b >> 10) * g.ncomp + cc) << (3 * lB)) + ((b & 1023) << lB) + ((2 * xh) & mB);
        if (al) *reinterpret_cast<float2 *>(q) = make_float2(g.mul * v.x, g.mul * v.y);
        else {
            q[0] = g.mul * v.x;
            q[1] = g.mul * v.y;
        }
    }
}

template <int M>
__global__ void __launch_bounds__(PX_THREADS) k_px_fwd(PlaneGeom g, const float *__restrict__ src, C *__restrict__ out)
{
    px_fwd_body<M>(g, src, out, blockIdx.x, blockIdx.y);
}
template <int M>
__global__ void __launch_bounds__(PX_THREADS) k_px_inv(PlaneGeom g, const C *__restrict__ in, float *__restrict__ dst)
{
    px_inv_body<M>(g, in, dst, blockIdx.x, blockIdx.y);
}
template <int M>
__global__ void __launch_bounds__(PX_THREADS) k_px_fwd_grp(const PlaneTask *__restrict__ tasks,
                                                           const int *__restrict__ cta, PlanePtrs ptrs)
{
    const PlaneTask &t = tasks[__ldg(cta + blockIdx.x)];
    const PlaneGeom g = t.g;
    px_fwd_body<M>(g, ptrs.src[t.solve], t.wa, blockIdx.x - t.first, 0);
}
template <int M>
__global__ void __launch_bounds__(PX_THREADS) k_px_inv_grp(const PlaneTask *__restrict__ tasks,
                                                           const int *__restrict__ cta, PlanePtrs ptrs)
{
    const PlaneTask &t = tasks[__ldg(cta + blockIdx.x)];
    const PlaneGeom g = t.g;
    px_inv_body<M>(g, t.wb, ptrs.dst[t.solve], blockIdx.x - t.first, 0);
}

// ---------------------------------------------------------------------------
// yz pass
//
// Bound by instruction issue in its transforms (about 2.9 a cycle and SM) and, 38 % of its time,
// by the latency of its loads and the cluster's sum, which only a second resident block hides.
// GB300: the 256^3 ring's scalar solve (432 x 384 x 384 points before, 416 x 384 x 384 here) 195 us
// against 68 + 179 + 70 us for the y, z and y passes it replaces, the solve 246 against 409 us; the
// 128^3 ring, three components, 117 us against 47 + 96 + 49 (run one after another), the solve
// 151-158 against 174.  Choices measured there: both halves of z per barrier with the odd one in a
// scratch (157 -> 132 us), packed (re, im) DFTs (123 -> 114), the fold's loads eight in flight
// (141 -> 123), the cluster reading its peers along z (180 -> 141) and each plane row once (the
// 256^3 ring 230 -> 205).  The cluster's sum costs 25 us there and saves the x inverse pass, which
// would read every residue, the same; on planes of 192 rows it saves 50 of 100 us.
// ---------------------------------------------------------------------------
// Threads: column groups of 16 lanes (half a warp, so a 64-bit access of 16 lanes is one
// conflict-free 128-byte row at the plane's odd pitch) times the R2 butterflies of the first
// z stage; a thread block has one or more groups, as many as the plane leaves room for
// (plane_pick).  The radices keep R1 small: a thread holds R1 rows, R1 accumulated results and
// an R2-point butterfly at once.
template <int MZ>
struct YZ {
    static constexpr int R2 = plane_z2(MZ), R1 = MZ / R2;
    static constexpr int GT = 16 * R2;
    static constexpr int maxt = plane_yz_threads(MZ);  // threads per SM the register cap allows
    static constexpr int P = MZ + 1;                   // plane pitch (complex)
};

// Transforms along y of `lines` plane rows (slot of line l: (l + off) mod MZ), in place.
template <int MY, int MZ, bool INV>
__device__ __forceinline__ void y_transform(C *plane, int lines, int off, const float2 *tw)
{
    constexpr int R1 = plane_r1(MY), R2 = plane_r2(MY), P = YZ<MZ>::P;
    const int hw = threadIdx.x >> 4, l16 = threadIdx.x & 15, nh = blockDim.x >> 4;
    const int units = (lines + 15) >> 4;
#pragma unroll
    for (int st = 0; st < 2; st++) {
        const bool first = (st == 0) != INV;  // the radix-R1 stage
        const int nb = first ? R2 : R1;
        for (int u = hw; u < units * nb; u += nh) {
            const int b = u % nb, l = (u / nb) * 16 + l16;
            if (l < lines) {
                int slot = l + off;
                if (slot >= MZ) slot -= MZ;
                if (first) butterfly_at<R1, INV, INV ? 0 : 1>(plane + b * P + slot, R2 * P, tw + b * R1, 1);
                else butterfly_at<R2, INV, INV ? 2 : 0>(plane + b * R2 * P + slot, P, tw + b, R1);
            }
        }
        __syncthreads();
    }
}
template <int MZ, bool INV>
__device__ __forceinline__ void y_transform_any(int My, C *plane, int lines, int off, const float2 *tw)
{
    switch (My) {
        case 16: y_transform<16, MZ, INV>(plane, lines, off, tw); break;
        case 32: y_transform<32, MZ, INV>(plane, lines, off, tw); break;
        case 48: y_transform<48, MZ, INV>(plane, lines, off, tw); break;
        case 64: y_transform<64, MZ, INV>(plane, lines, off, tw); break;
        case 80: y_transform<80, MZ, INV>(plane, lines, off, tw); break;
        case 96: y_transform<96, MZ, INV>(plane, lines, off, tw); break;
        case 112: y_transform<112, MZ, INV>(plane, lines, off, tw); break;
        default: y_transform<128, MZ, INV>(plane, lines, off, tw); break;
    }
}

// thread-block clusters: barrier, a peer's shared-memory address, a read there
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_addr(const C *p, int rank)
{
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return a;
}
__device__ __forceinline__ C ld_cluster(uint32_t a)
{
    C v;
    asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a));
    return v;
}

template <int MZ>
__device__ __forceinline__ void group_sync(int grp)
{
    asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "n"(YZ<MZ>::GT) : "memory");
}

// The radix-R2 middle of the z convolution: butterfly q of one half (ZP: odd frequencies), in
// place at p[0 .. R2): DFT, spectrum kv, inverse DFT, stage twiddles of the inverse.
template <int MZ>
__device__ __forceinline__ void z_mid(C *p, const float (&kv)[YZ<MZ>::R2], const float2 *tw, int q)
{
    constexpr int R1 = YZ<MZ>::R1, R2 = YZ<MZ>::R2;
    V a[R2];
#pragma unroll
    for (int k2 = 0; k2 < R2; k2++) a[k2] = v_ld(p + k2);
    dft<R2, false>(a);
#pragma unroll
    for (int k2 = 0; k2 < R2; k2++) a[k2] = a[k2] * fft::bc2(kv[k2]);
    dft<R2, true>(a);
#pragma unroll
    for (int k2 = 0; k2 < R2; k2++) {
        if (k2 > 0) a[k2] = v_mulc(a[k2], ld(tw + k2 * R1 + q));
        v_st(p + k2, a[k2]);
    }
}
// its spectrum values (rows: plane_len.hpp).  K: the spectrum of the thread block's plane, col: the
// column's place in its rows of My.
template <int MZ>
__device__ __forceinline__ void z_spectrum(float (&kv)[YZ<MZ>::R2], const float *K, unsigned col, unsigned My, bool odd,
                                           int q)
{
    constexpr int R1 = YZ<MZ>::R1, R2 = YZ<MZ>::R2;
    const unsigned lo = col + plane_row_lo(MZ, odd, q) * My;
    const unsigned hi = col + plane_row_hi(MZ, odd, q) * My;
#pragma unroll
    for (int k2 = 0; k2 < R2; k2++) kv[k2] = k2 < R2 / 2 ? __ldg(K + (lo + k2 * R1 * My)) : __ldg(K + (hi - k2 * R1 * My));
}

// Fold and twist: plane[n][z] = sum_(j < NJ) A[n + j My][z] w_Ny^(r (n + j My)), zero outside the
// source box; half a warp takes 16 z of a row n, eight loads in flight per thread.
template <int MZ, int NJ>
__device__ __forceinline__ void fold_rows(C *plane, const C *__restrict__ a, const float2 *__restrict__ wf, int My,
                                          int Ey, int Ez)
{
    constexpr int U = 8 / NJ, P = YZ<MZ>::P;
    const int l16 = threadIdx.x & 15, nh = blockDim.x >> 4;
    for (int n = threadIdx.x >> 4; n < My; n += nh) {
        C w[NJ];
#pragma unroll
        for (int j = 0; j < NJ; j++) w[j] = n + j * My < Ey ? ld(wf + n + j * My) : C{0.f, 0.f};
        const C *p = a + n * Ez;
#pragma unroll
        for (int z0 = 0; z0 < MZ; z0 += 16 * U) {
            C v[U][NJ];
#pragma unroll
            for (int u = 0; u < U; u++)
#pragma unroll
                for (int j = 0; j < NJ; j++) {
                    const int z = z0 + 16 * u + l16;
                    v[u][j] = z < Ez && n + j * My < Ey ? ld_l2(p + j * My * Ez + z) : C{0.f, 0.f};
                }
#pragma unroll
            for (int u = 0; u < U; u++) {
                C s = mul(v[u][0], w[0]);
#pragma unroll
                for (int j = 1; j < NJ; j++) s = s + mul(v[u][j], w[j]);
                if (z0 + 16 * u < MZ) plane[n * P + z0 + 16 * u + l16] = s;
            }
        }
    }
}

// This thread block's share of the target rows: o[yt][zt] = sum_r conj(w_Ny^(r p)) v_r[p mod My][zt]
// over the cluster's planes.  It takes the rows p with p mod My in its My / DY of the plane rows, so
// each plane row is read once for all its targets p = n + j My; half a warp along zt.
template <int MZ, int DY>
__device__ __forceinline__ void sum_rows(C *plane, C *__restrict__ o, const PlaneGeom &g, int rank, int off)
{
    constexpr int U = 8 / DY, P = YZ<MZ>::P;
    const int l16 = threadIdx.x & 15, nh = blockDim.x >> 4, My = g.My, Ety = g.Et[1], Etz = g.Et[2];
    const int nc = (My + DY - 1) / DY, nb = rank * nc, ne = min(My, nb + nc);
    for (int n = nb + (threadIdx.x >> 4); n < ne; n += nh) {
        int y0 = (n - g.d0[1]) % My;  // first target row of this plane row
        if (y0 < 0) y0 += My;
        uint32_t base[DY];
#pragma unroll
        for (int q = 0; q < DY; q++) base[q] = cluster_addr(plane + n * P, q);
        for (int z0 = l16; z0 < Etz; z0 += 16 * U) {
            C v[U][DY];
#pragma unroll
            for (int u = 0; u < U; u++) {
                int slot = min(z0 + 16 * u, Etz - 1) + off;
                if (slot >= MZ) slot -= MZ;
#pragma unroll
                for (int q = 0; q < DY; q++) v[u][q] = ld_cluster(base[q] + slot * 8);
            }
            for (int yt = y0; yt < Ety; yt += My) {
                C w[DY];
#pragma unroll
                for (int q = 1; q < DY; q++) w[q] = ld(g.twi + q * Ety + yt);
                C *row = o + (size_t)yt * Etz;
#pragma unroll
                for (int u = 0; u < U; u++) {
                    C s = v[u][0];  // residue 0: factor 1
#pragma unroll
                    for (int q = 1; q < DY; q++) s = s + mul(v[u][q], w[q]);
                    if (z0 + 16 * u < Etz) row[z0 + 16 * u] = s;
                }
            }
        }
    }
}

template <int MZ>
__device__ __forceinline__ void yz_body(const PlaneGeom &g, const C *__restrict__ A, C *__restrict__ Bo, int item, int nc)
{
    using Y = YZ<MZ>;
    constexpr int R1 = Y::R1, R2 = Y::R2, P = Y::P;
    extern __shared__ float2 sm_yz[];
    C *plane = reinterpret_cast<C *>(sm_yz);
    const int My = g.My, NT = blockDim.x;
    float2 *twy = sm_yz + My * P, *twz = twy + My, *w2 = twz + MZ, *w2o = w2 + MZ;
    C *scratch = reinterpret_cast<C *>(w2o + MZ);  // [NT / GT][16][P]
    // the Dy residues of a (kx, component) are neighbours (a cluster)
    const int r = item % g.Dy, kc = item / g.Dy, c = kc % nc, kx = kc / nc, kr = kx * g.Dy + r;
    table_to_smem(twy, g.st[1], My);
    for (int i = threadIdx.x; i < MZ; i += NT) {
        // stage twiddles, the twist w_Nz^n of the odd half, and its conjugate at the target position
        // p = n, or n - Mz < 0, where it changes sign
        twz[i] = __ldg(g.st[2] + i);
        const float2 w = __ldg(g.w2[2] + i);
        w2[i] = w;
        w2o[i] = i - g.d0[2] >= MZ ? make_float2(-w.x, -w.y) : w;
    }
    const int Ey = g.Es[1], Ez = g.Es[2];
    pdl_trigger();
    pdl_wait();  // the x pass is complete
    {
        const C *a = A + ((size_t)c * g.KX + kx) * Ey * Ez;
        const float2 *wf = g.twf + r * Ey;
        if (Ey <= My) fold_rows<MZ, 1>(plane, a, wf, My, Ey, Ez);
        else if (Ey <= 2 * My) fold_rows<MZ, 2>(plane, a, wf, My, Ey, Ez);
        else fold_rows<MZ, 4>(plane, a, wf, My, Ey, Ez);
    }
    __syncthreads();
    y_transform_any<MZ, false>(My, plane, Ez, 0, twy);
    {
        const int grp = threadIdx.x / Y::GT, t = threadIdx.x % Y::GT, b = t >> 4, ng = NT / Y::GT;
        const float *Kp = g.Kt + (size_t)kr * (MZ + 1) * My;
        C *odd = scratch + (grp * 16 + (t & 15)) * P;  // the odd half of this thread's column
        for (int cg = grp; cg * 16 < My; cg += ng) {
            const int col = cg * 16 + (t & 15);
            C *colp = plane + col * P;
            float kv[R2];
            // the first middle butterfly's spectrum, in flight during the first stage
            const int ahead = plane_mid_ahead(MZ, b);
            z_spectrum<MZ>(kv, Kp, col, My, ahead >= R1, ahead >= R1 ? ahead - R1 : ahead);
            {
                V x[R1], v[R1];
#pragma unroll
                for (int m = 0; m < R1; m++) v[m] = x[m] = v_ld(colp + b + m * R2);
                dft<R1, false>(v);
#pragma unroll
                for (int q = 0; q < R1; q++) {
                    if (q > 0) v[q] = v_mul(v[q], ld(twz + b * R1 + q));
                    v_st(colp + b + q * R2, v[q]);
                }
#pragma unroll
                for (int m = 0; m < R1; m++) v[m] = v_mul(x[m], ld(w2 + b + m * R2));
                dft<R1, false>(v);
#pragma unroll
                for (int q = 0; q < R1; q++) {
                    if (q > 0) v[q] = v_mul(v[q], ld(twz + b * R1 + q));
                    v_st(odd + b + q * R2, v[q]);
                }
            }
            group_sync<MZ>(grp);
#pragma unroll
            for (int u0 = 0; u0 < 2 * R1; u0 += R2) {
                const int u = u0 + b;
                if ((2 * R1) % R2 == 0 || u < 2 * R1) {
                    const bool od = u >= R1;
                    const int q = od ? u - R1 : u;
                    if (u0 > 0) z_spectrum<MZ>(kv, Kp, col, My, od, q);
                    z_mid<MZ>((od ? odd : colp) + q * R2, kv, twz, q);
                }
            }
            group_sync<MZ>(grp);
            {
                V acc[R1], v[R1];
#pragma unroll
                for (int q = 0; q < R1; q++) acc[q] = v_ld(colp + b + q * R2);
                dft<R1, true>(acc);
#pragma unroll
                for (int q = 0; q < R1; q++) v[q] = v_ld(odd + b + q * R2);
                dft<R1, true>(v);
#pragma unroll
                for (int m = 0; m < R1; m++) v_st(colp + b + m * R2, acc[m] + v_mulc(v[m], ld(w2o + b + m * R2)));
            }
        }
    }
    __syncthreads();
    const int Etz = g.Et[2];
    int off = g.d0[2] % MZ;
    if (off < 0) off += MZ;
    y_transform_any<MZ, true>(My, plane, Etz, off, twy);
    // sum over the residues, conj(w_Ny^(r p)) v_r[p mod My] at target position p: the Dy thread blocks
    // of one (kx, component) form a cluster and each takes a share of the target rows, reading
    // the others' shared memory
    cluster_sync();
    {
        C *o = Bo + ((size_t)c * g.KX + kx) * Etz * g.Et[1];
        if (g.Dy == 2) sum_rows<MZ, 2>(plane, o, g, r, off);
        else if (g.Dy == 3) sum_rows<MZ, 3>(plane, o, g, r, off);
        else sum_rows<MZ, 4>(plane, o, g, r, off);
    }
    cluster_sync();  // the other blocks have read this one's plane
}

template <int MZ>
__global__ void __launch_bounds__(YZ<MZ>::maxt, 1) k_yz(PlaneGeom g, const C *__restrict__ A, C *__restrict__ Bo)
{
    yz_body<MZ>(g, A, Bo, blockIdx.x, g.nc);
}
template <int MZ>
__global__ void __launch_bounds__(YZ<MZ>::maxt, 1) k_yz_grp(const PlaneTask *__restrict__ tasks,
                                                                     const int *__restrict__ cta)
{
    const PlaneTask &t = tasks[__ldg(cta + blockIdx.x)];
    const PlaneGeom g = t.g;
    yz_body<MZ>(g, t.wa, t.wb, blockIdx.x - t.first, 1);
}

// dynamic shared memory up to the limit, and the same carveout for the three passes (an SM
// drains before it changes its carveout)
template <typename F>
lgf_status plane_attr(F *f, size_t smem)
{
    LGF_CUDA_TRY(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    LGF_CUDA_TRY(cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared));
    return LGF_OK;
}

}  // namespace

template <int M>
lgf_status PlaneX<M>::prepare()
{
    LGF_TRY(plane_attr(k_px_fwd<M>, px_smem<M>()));
    LGF_TRY(plane_attr(k_px_inv<M>, px_smem<M>()));
    LGF_TRY(plane_attr(k_px_fwd_grp<M>, px_smem<M>()));
    return plane_attr(k_px_inv_grp<M>, px_smem<M>());
}
template <int M>
lgf_status PlaneX<M>::fwd(const PlaneGeom &g, const float *src, cx<float> *a, cudaStream_t s)
{
    LGF_CUDA_TRY(launch_pdl_smem(k_px_fwd<M>, dim3(plane_tiles(0, g), g.nc), dim3(PX_THREADS), px_smem<M>(), s, g, src, a));
    return LGF_OK;
}
template <int M>
lgf_status PlaneX<M>::inv(const PlaneGeom &g, const cx<float> *b, float *dst, cudaStream_t s)
{
    LGF_CUDA_TRY(launch_pdl_smem(k_px_inv<M>, dim3(plane_tiles(2, g), g.nc), dim3(PX_THREADS), px_smem<M>(), s, g, b, dst));
    return LGF_OK;
}
template <int M>
lgf_status PlaneX<M>::fwd_grp(const PlaneTask *t, const int *cta, int ncta, const PlanePtrs &p, cudaStream_t s)
{
    LGF_CUDA_TRY(launch_pdl_smem(k_px_fwd_grp<M>, dim3(ncta), dim3(PX_THREADS), px_smem<M>(), s, t, cta, p));
    return LGF_OK;
}
template <int M>
lgf_status PlaneX<M>::inv_grp(const PlaneTask *t, const int *cta, int ncta, const PlanePtrs &p, cudaStream_t s)
{
    LGF_CUDA_TRY(launch_pdl_smem(k_px_inv_grp<M>, dim3(ncta), dim3(PX_THREADS), px_smem<M>(), s, t, cta, p));
    return LGF_OK;
}
template <int M>
lgf_status PlaneYZ<M>::prepare()
{
    LGF_TRY(plane_attr(k_yz<M>, 227 * 1024));
    return plane_attr(k_yz_grp<M>, 227 * 1024);
}
template <int M>
lgf_status PlaneYZ<M>::run(const PlaneGeom &g, const cx<float> *a, cx<float> *b, cudaStream_t s)
{
    LGF_CUDA_TRY(launch_pdl_cluster(k_yz<M>, dim3(plane_tiles(1, g) * g.nc), dim3(g.ntz), plane_smem(1, g), g.Dy, s, g, a, b));
    return LGF_OK;
}
template <int M>
lgf_status PlaneYZ<M>::grp(const PlaneTask *t, const int *cta, int ncta, size_t smem, int threads, int Dy,
                            cudaStream_t s)
{
    LGF_CUDA_TRY(launch_pdl_cluster(k_yz_grp<M>, dim3(ncta), dim3(threads), smem, Dy, s, t, cta));
    return LGF_OK;
}

}  // namespace lgf
