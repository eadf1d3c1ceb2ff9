"""The form in which FP64 links lie in memory for the integer Dslash
(csrc/fix_link.cuh): every number comes back bit for bit, the limbs are the
number rounded to a multiple of 2^-57 (0 below 2^-57), links that do not fit are
refused.

A host program includes the header itself (as test_fastdiv does).  Numbers:
uniform, with random powers of two down to the subnormals, exact 0, -0 and +-1,
just above 1 in size.  Random SU(3) rows must all fit.  No GPU.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1111_0125_gb300", "csrc")

PROGRAM = r"""
#include <math.h>
#include <stdio.h>
#include "fix_link.cuh"
using namespace stg;

static unsigned long long state = 88172645463325252ull;
static unsigned long long rnd(void)
{
    state ^= state << 13; state ^= state >> 7; state ^= state << 17;
    return state;
}

template <int N> static int run(void)
{
    long fit[6] = {0}, refused[6] = {0}, bad = 0;
    for (long t = 0; t < 1200000; ++t) {
        const int kind = t % 6;
        double u[N], v[N];
        int2 w[N];
        for (int r = 0; r < N; ++r) {
            double x = ldexp((double)(rnd() >> 11), -52) - 1.0;
            if (kind == 1) x = ldexp(x, -(int)(rnd() % 8));
            if (kind == 2 && rnd() % 18 == 0) x = ldexp(x, -(int)(rnd() % 60));
            if (kind == 3) x = rnd() % 3 ? (rnd() & 1 ? 0.0 : -0.0) : (rnd() & 1 ? 1.0 : -1.0);
            if (kind == 4 && r == 5) x = ldexp(x, -(int)(rnd() % 1074));
            if (kind == 5 && rnd() % 4 == 0) x = rnd() & 1 ? 1.0005 : -1.0005;
            if (kind == 1 && rnd() % 8 == 0)  // around a power of two: carries of the rounding
                x = ldexp(1.0 + ((int)(rnd() % 9) - 4) * ldexp(1.0, -52), -(int)(rnd() % 12));
            u[r] = x;
        }
        const unsigned row = rnd() & 15, col = rnd() & 15;
        if (!fix_encode<N>(u, row, col, w)) {
            ++refused[kind];
            continue;
        }
        ++fit[kind];
        fix_decode<N>(w, v);
        bad += (w[0].y & 15) != (int)row || (w[1].y & 15) != (int)col;
        for (int r = 0; r < N; ++r) {
            const long long x = ((long long)(w[r].x >> 1) << 28) + (w[r].y >> 4);
            const int l = w[r].y >> 4;
            const double y = ldexp(u[r], 57);  // llround: half away from zero
            bad += fix_bits(u[r]) != fix_bits(v[r]) || l < -(1 << 27) || l >= (1 << 27) ||
                   x != (fabs(y) < 1 ? 0 : llround(y));
        }
    }
    printf("N %d bad %ld", N, bad);
    for (int k = 0; k < 6; ++k) printf(" %ld/%ld", fit[k], refused[k]);
    printf("\n");
    // uniform numbers, and exact zeros and ones (at most 2 of the bits each): all fit
    return bad != 0 || (N == 18 && (refused[0] || refused[3] || refused[5])) || fit[4] == 0 || refused[4] == 0;
}

int main(void)
{
    return run<18>() | run<12>();
}
"""


def _nvcc():
    return shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc"
                                    if os.path.exists("/usr/local/cuda/bin/nvcc") else None)


def test_links_come_back_bit_for_bit(tmp_path):
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not available")
    src = tmp_path / "fix_link_check.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "fix_link_check"
    subprocess.run([nvcc, "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True,
                   capture_output=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-2000:]
