"""The mixed CG's scalars (csrc/stg_common.cuh): the state's doubles reach its
kernels in FP32 numbers with all their bits, an iteration stops by exactly
those, and quotients are rounded once.  No GPU: a host program includes the
headers.

A quotient's rounding to FP32 may differ from that of the double quotient only
where that lies within 2^-45 of a midpoint, 2^-20 of the cases.
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
#include <string.h>
#include "stg_internal.h"
using namespace stg;

static unsigned long long state = 88172645463325252ull;
static unsigned long long rnd(void)
{
    state ^= state << 13; state ^= state >> 7; state ^= state << 17;
    return state;
}
static double positive(int span) { return ldexp(1.0 + ldexp((double)(rnd() >> 12), -52), (int)(rnd() % (2 * span + 1)) - span); }
static FF pair(double v)
{
    const float hi = (float)v;
    return FF{hi, (float)(v - (double)hi)};
}
static double value(FF a) { return (double)a.hi + (double)a.lo; }
static int sign(double a, double b) { return a < b ? -1 : a > b ? 1 : 0; }

int main(void)
{
    long bad = 0, off = 0;
    for (int t = 0; t < 300000; ++t) {
        CGState h;
        memset(&h, 0, sizeof(h));
        h.delta_new = positive(60);
        h.delta_old = positive(60);
        h.rmax2 = positive(60);
        h.stop_r2 = positive(60);
        h.trig2 = 0.01;
        CGState g = h;
        state_put(&g, P32);
        bad += f3_double(g.f_stop) != h.stop_r2 || f3_double(g.f_trig) != 0.01 * h.rmax2;
        g.delta_new = g.delta_old = g.rmax2 = 0.0;
        state_got(&g);
        bad += g.delta_new != h.delta_new || g.delta_old != h.delta_old || g.rmax2 != h.rmax2;

        // sums around a stopping value, by its own ulps and by those of a pair
        const FF a = pair(positive(60));
        const double v = value(a), near[] = {v, nextafter(v, INFINITY), nextafter(v, 0.0), v * (1 + ldexp(1.0, -47)),
                                             v * (1 - ldexp(1.0, -47)), v * 1.5, v * 0.6, positive(60)};
        for (const double b : near) {
            const F3 s = f3_split(b), none = f3_split(0.0);
            bad += f3_cmp(a, s) != sign(v, b);
            bad += f3_stop(a, s, none) != (v <= b ? FLAG_CONVERGED : FLAG_RUN);
            bad += f3_stop(a, none, s) != (v < b ? FLAG_UPDATE : FLAG_RUN);
        }
        const FF loose = {a.hi, a.lo + a.hi * 0x1p-23f}, n = ff_norm(loose);
        bad += value(n) != value(loose) || n.hi != (float)value(loose);
    }
    const F3 one = f3_split(1.0), none = f3_split(0.0);
    bad += f3_stop(FF{INFINITY, 0.f}, one, none) != FLAG_BREAKDOWN || f3_stop(FF{NAN, 0.f}, one, none) != FLAG_BREAKDOWN ||
           f3_stop(FF{0.f, 0.f}, none, none) != FLAG_CONVERGED;
    for (int t = 0; t < 4000000; ++t) {
        const FF a = pair(positive(60)), b = pair(positive(60));
        const double q = value(a) / value(b);
        if (ff_div(a, b) != (float)q) {
            ++off;
            bad += fabs((double)ff_div(a, b) - q) > ldexp(q, -24) * (1 + ldexp(1.0, -18));
        }
    }
    printf("bad %ld off %ld\n", bad, off);
    return bad != 0 || off > 3 * 4;  // 4e6 2^-20 = 4 expected
}
"""


def test_scalars(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src = tmp_path / "scalars_check.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "scalars_check"
    subprocess.run([nvcc, "-O2", "-std=c++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"), str(src), "-o", str(exe)],
                   check=True, capture_output=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout
