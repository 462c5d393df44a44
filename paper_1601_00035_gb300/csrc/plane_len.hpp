// Lengths of the three-pass Poisson solve and the index arithmetic that depends on them alone.
// Plain C++, so that a host compiler can check it over every length.
#pragma once

#if defined(__CUDACC__)
#define LGF_LEN __host__ __device__ constexpr
#else
#define LGF_LEN constexpr
#endif

namespace lgf {

// radices of M = R1 * R2 (R2 even)
LGF_LEN int plane_r2(int M)
{
    return M <= 32 ? 4 : M == 48 ? 6 : M <= 128 ? 8 : M == 144 ? 12 : M == 160 ? 10 : M == 192 ? 12 : M == 224 ? 14 : 16;
}
LGF_LEN int plane_r1(int M) { return M / plane_r2(M); }
// the z transform's second radix (even), and the threads per SM its registers leave room for
LGF_LEN int plane_z2(int M)
{
    return M == 16 ? 4 : (M <= 80 ? 8 : 16);
}
LGF_LEN int plane_yz_threads(int M) { return M <= 128 ? 1024 : M <= 192 ? 768 : 512; }

#define LGF_PLANE_LENGTHS(X) \
    X(16) X(32) X(48) X(64) X(80) X(96) X(112) X(128) X(144) X(160) X(176) X(192) X(208) X(224) X(240) X(256)

// The middle of the z convolution.  A column has 2 R1 butterflies of R2 points, u < R1 those of the
// even frequencies (q = u) and the rest those of the odd ones (q = u - R1); its R2 threads take
// butterfly b, then b + R2 and so on.  Threads b >= 2 R1 (lengths 96 and 112, where R1 is 6 and 7
// and R2 is 16) have none: the spectrum that every thread loads ahead is then the last butterfly's,
// and is dropped (64 ragged solves 1361 us; with a branch around the load 1369).
LGF_LEN int plane_mid_ahead(int M, int b)
{
    const int last = 2 * (M / plane_z2(M)) - 1;
    return last >= plane_z2(M) - 1 || b < last ? b : last;  // (the first folds at compile time)
}
// Spectrum row (0 .. M, plane.cu's order: even frequencies, then odd ones) of element k2 of butterfly
// q: frequency kk = q + R1 k2 of its half is row plane_row_lo + R1 k2 below M / 2 (k2 < R2 / 2), and
// folds to M - kk (even half) or M - 1 - kk (odd) above, row plane_row_hi - R1 k2.
LGF_LEN int plane_row_lo(int M, bool odd, int q) { return (odd ? M / 2 + 1 : 0) + q; }
LGF_LEN int plane_row_hi(int M, bool odd, int q) { return (odd ? M / 2 + M : M) - q; }

}  // namespace lgf
