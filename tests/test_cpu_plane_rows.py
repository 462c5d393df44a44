"""Which rows of the kernel spectrum the yz pass of the three-pass Poisson solve reads, for every z
length: the kernel's own index functions (plane_len.hpp), compiled for the host.  Every load of
every thread has to lie in the Mz + 1 rows of its plane, the first butterfly's early loads included,
and element k2 of butterfly q has to get the row that holds its frequency."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1601_00035_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "plane_len.hpp"
using namespace lgf;
int bad = 0;
void load(int M, int b, int u)  // thread b loads the spectrum of butterfly u
{
    const int R2 = plane_z2(M), R1 = M / R2;
    const bool odd = u >= R1;
    const int q = odd ? u - R1 : u;
    for (int k2 = 0; k2 < R2; k2++) {
        const int row = k2 < R2 / 2 ? plane_row_lo(M, odd, q) + k2 * R1 : plane_row_hi(M, odd, q) - k2 * R1;
        const int kz = 2 * (q + R1 * k2) + odd, f = kz <= M ? kz : 2 * M - kz;
        const int want = odd ? M / 2 + 1 + f / 2 : f / 2;
        if (row >= 0 && row <= M && row == want) continue;
        if (!bad++) printf("length %d, thread %d, k2 %d: row %d of %d, frequency in %d\n", M, b, k2, row, M + 1, want);
    }
}
void length(int M)
{
    const int R2 = plane_z2(M), R1 = M / R2;
    for (int b = 0; b < R2; b++) {
        const int ahead = plane_mid_ahead(M, b);
        load(M, b, ahead);
        if (b < 2 * R1 && ahead != b) bad++, printf("length %d: thread %d loads butterfly %d ahead\n", M, b, ahead);
        for (int u = b + R2; u < 2 * R1; u += R2) load(M, b, u);
    }
}
int main()
{
#define CHECK(M) length(M);
    LGF_PLANE_LENGTHS(CHECK)
    return bad != 0;
}
"""


def test_spectrum_rows(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "rows.cpp", tmp_path / "rows"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True, capture_output=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
