"""Distance of the fixed-point transforms' values from overflow (csrc/fixed.cuh,
host build): the deviations inside every pass of every plan."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1903_08741_gb300", "csrc")
SRC = r"""
#include "fixed.cuh"
using namespace rich_fx;
static double acc;
static long cnt;
// a forward pass from bit b0 on, in place; the sum of squares of the values that
// its twiddles and shifts meet
template <int R> static void pass(fx2* a, int logn, int b0, int bits) {
    const int lq = logn - b0 - bits, n = 1 << logn, sh = ((b0 + bits) >> 1) - (b0 >> 1);
    for (int g = 0; g < n >> bits; ++g) {
        const int k = g & ((1 << lq) - 1), base = ((g >> lq) << (lq + bits)) + k;
        fx2 v[R];
        for (int j = 0; j < R; ++j) v[j] = a[base + (j << lq)];
        dft_fwd<R>(v);
        for (int j = 0; j < R; ++j) {
            acc += (double)v[j].re * v[j].re + (double)v[j].im * v[j].im;
            cnt += 2;
            a[base + (j << lq)] = cmul(v[j], circle_point(-((long long)(k * revr<R>(j)) << b0), n), sh);
        }
    }
}
// deviations (units of 2^55) inside the passes; returns their number
extern "C" int t_passes(int logn, int lines, const double* x, double* inside) {
    const int n = 1 << logn;
    fx2* a = new fx2[(long)n * lines];
    for (long i = 0; i < (long)n * lines; ++i)
        a[i] = fx2{llrint(ldexp(x[2 * i], FX_BITS)), llrint(ldexp(x[2 * i + 1], FX_BITS))};
    int np = 0;
    for (int b = 0; b < logn; ++np) {
        const int w = pass_bits(logn, b);
        acc = 0; cnt = 0;
        for (int l = 0; l < lines; ++l) {
            if (w == 3) pass<8>(a + (long)l * n, logn, b, w);
            else if (w == 2) pass<4>(a + (long)l * n, logn, b, w);
            else pass<2>(a + (long)l * n, logn, b, w);
        }
        inside[np] = ldexp(sqrt(acc / cnt), -FX_BITS);
        b += w;
    }
    delete[] a;
    return np;
}
"""


@pytest.mark.parametrize("logn", range(1, 14))
def test_values_stay_away_from_overflow(tmp_path, logn):
    """Rows start at 2^55 and columns behind rows of an odd power of two at 2^55.5;
    overflow is at 2^61 = 64 of the deviations' units.  65 536 values or more put
    the measured deviation within 1.5 % of the true one."""
    (tmp_path / "t.cpp").write_text(SRC)
    subprocess.run(["g++", "-O1", "-std=gnu++17", "-shared", "-fPIC", "-I", CSRC, "-o", str(tmp_path / "t.so"),
                    str(tmp_path / "t.cpp")], check=True)
    lib = C.CDLL(str(tmp_path / "t.so"))
    lines = max(1, 32768 >> logn)
    for start, least in ((1.0, 16.0), (2 ** 0.5, 16.0 / 2 ** 0.5)):
        x = np.random.default_rng(logn).standard_normal((lines << logn, 2)) * start
        inside = np.zeros(8)
        k = lib.t_passes(logn, lines, x.ctypes.data_as(C.c_void_p), inside.ctypes.data_as(C.c_void_p))
        assert k >= 1 and 64.0 / inside[:k].max() >= least / 1.015
        assert inside[:k].min() >= start           # nothing shrinks
