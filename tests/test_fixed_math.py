"""Host build of the fixed-point functions (csrc/fixed.cuh) against the library's:
the closures' exponential and van Genuchten functions over the forms they accept
and the ones they hand back, and the normals of the fields."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1903_08741_gb300", "csrc")
SRC = r"""
#include "fixed.cuh"
using namespace rich_fx;
extern "C" void t_exp(int n, const double* x, double* y) { for (int i = 0; i < n; ++i) y[i] = fx_exp(x[i]); }
extern "C" void t_div(int n, const double* a, const double* b, double* q) { for (int i = 0; i < n; ++i) q[i] = fx_div(a[i], b[i]); }
extern "C" void t_vg(int k, const double* ap, const double* n, const double* m, int* ok, double* s, double* kr, double* d) {
    for (int i = 0; i < k; ++i) { VgLog o; ok[i] = vg_log(ap[i], n[i], m[i], o); if (ok[i]) { s[i] = vg_s(o); vg_k(o, kr[i], d[i]); } }
}
extern "C" void t_cdf(int n, const double* x, double* y) {
    static NormTab t; make_norm_tab(t);
    for (int i = 0; i < n; ++i) y[i] = normal_cdf(x[i], t.phi);
}
extern "C" void t_normal(int k, const unsigned* c, double* y) {
    static NormTab t; make_norm_tab(t);
    for (int i = 0; i < k; ++i) { long long a, b; normal_pair(c[4*i], c[4*i+1], c[4*i+2], c[4*i+3], &t, a, b);
        y[2*i] = ldexp((double)a, -FX_BITS); y[2*i+1] = ldexp((double)b, -FX_BITS); }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed")
    (d / "t.cpp").write_text(SRC)
    subprocess.run(["g++", "-O1", "-std=gnu++17", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "t.so"), str(d / "t.cpp")],
                   check=True)
    return C.CDLL(str(d / "t.so"))


def dp(a):
    return a.ctypes.data_as(C.c_void_p)


def test_exp_is_within_six_tenths_of_a_unit(lib):
    """All magnitudes to the overflow, both signs, zeros and non-finite values:
    the rounding (0.5) and a working precision of 2^-57."""
    g = np.random.default_rng(0)
    s = np.where(g.random(60000) < 0.5, -1.0, 1.0)
    x = np.concatenate([s[:20000] * 2.0 ** g.uniform(-70, 9.4, 20000), s[20000:40000] * g.uniform(0, 700, 20000),
                        -g.uniform(0, 20, 20000), [0.0, -0.0, -800.0, 800.0, -np.inf, np.inf, np.nan, -511.99, -512.0, -740.0]])
    y = np.empty_like(x)
    lib.t_exp(len(x), dp(x), dp(y))
    with np.errstate(over="ignore", invalid="ignore", under="ignore"):
        want = np.exp(x.astype(np.longdouble))
        rounded = want.astype(np.float64)
        assert np.array_equal(np.isnan(y), np.isnan(rounded)) and np.array_equal(np.isinf(y), np.isinf(rounded))
        f = np.isfinite(rounded) & (rounded > 1e-300)
        assert (np.abs(y[f] - want[f]) / np.spacing(rounded[f])).max() < 0.6
        assert np.array_equal(y[x == 0], np.ones(2)) and y[x == -800.0] == 0


def test_division_is_within_six_tenths_of_a_unit(lib):
    """Mantissas at both ends and throughout, quotients over the whole range;
    what is not positive, normal or in range gives the division's own bits."""
    g = np.random.default_rng(3)
    k = 60000
    a, b = (1 + g.random(k)) * 2.0 ** g.integers(-400, 400, k), (1 + g.random(k)) * 2.0 ** g.integers(-400, 400, k)
    b[:1000] = np.nextafter(2.0, 0) * 2.0 ** g.integers(-9, 9, 1000)
    b[1000:2000] = 1 + 2.0 ** -52 * g.integers(0, 9, 1000)
    a[2000:3000] = b[2000:3000]
    special = np.array([0.0, -0.0, 1.0, -3.0, np.inf, -np.inf, np.nan, 5e-324, 2e-308, 1.7e308])
    sa, sb = (v.ravel() for v in np.meshgrid(special, special))
    q, sq = np.empty(k), np.empty(len(sa))
    lib.t_div(k, dp(a), dp(b), dp(q))
    want = a.astype(np.longdouble) / b.astype(np.longdouble)
    assert (np.abs(q - want) / np.spacing(a / b)).max() < 0.6
    assert np.array_equal(q[2000:3000], np.ones(1000))
    lib.t_div(len(sa), dp(sa), dp(sb), dp(sq))
    with np.errstate(all="ignore"):
        assert np.allclose(sq, sa / sb, rtol=2.3e-16, atol=0, equal_nan=True)


def test_van_genuchten_matches_the_library_functions(lib):
    """s, k_rw and its derivative where the ranges accept, against 64-bit
    mantissas: logarithms good to 2^-57, times n < 16 and two more roundings,
    1e-14 relative (k_rw: absolute, its 1 - x cancels)."""
    g = np.random.default_rng(1)
    k = 40000
    n = np.where(g.random(k) < 0.5, g.uniform(1.02, 2, k), g.uniform(2, 12, k))
    m = 1 - 1 / n
    ap = np.exp(g.uniform(-30, 8, k))
    ok, s, kr, d = np.zeros(k, np.int32), np.zeros(k), np.zeros(k), np.zeros(k)
    lib.t_vg(k, dp(ap), dp(n), dp(m), dp(ok), dp(s), dp(kr), dp(d))
    a = ok.astype(bool)
    assert a[(n * np.abs(np.log(ap)) < 40)].all()
    q, ql, qm = (v[a].astype(np.longdouble) for v in (ap, n, m))
    an = np.exp(ql * np.log(q))
    S = np.exp(-qm * np.log1p(an))
    b = 1 - S * (an / q)
    assert (np.abs(s[a] - S) / S).max() < 1e-14
    assert np.abs(kr[a] - np.sqrt(S) * b * b).max() < 1e-14
    D = S * an / ((1 + an) * q)
    assert (np.abs(d[a] - D) / D).max() < 1e-14


def test_van_genuchten_hands_back_what_leaves_its_ranges(lib):
    bad = [(-1.0, 2.0, 0.5), (0.0, 2.0, 0.5), (np.nan, 2.0, 0.5), (np.inf, 2.0, 0.5), (5e-324, 2.0, 0.5), (1e30, 2.0, 0.5),
           (1.0, 17.0, 0.9), (1.0, np.nan, 0.5), (1.0, -2.0, 0.5), (1.0, 2.0, 1.0), (1.0, 2.0, 0.0), (1.0, 2.0, -0.5),
           (1.0, 2.0, np.nan), (1e9, 12.0, 0.9), (1e-17, 15.0, 0.9)]
    ap, n, m = (np.array(v) for v in zip(*bad))
    ok, z = np.ones(len(bad), np.int32), np.zeros(len(bad))
    lib.t_vg(len(bad), dp(ap), dp(n), dp(m), dp(ok), dp(z), dp(z.copy()), dp(z.copy()))
    assert not ok.any()


def test_normals_match_box_muller(lib):
    """Box-Muller in FP64 is off by the rounding of its angle, 2^-51 times a
    radius of up to 8.6, and of its functions: 5e-15 in all."""
    g = np.random.default_rng(2)
    c = g.integers(0, 2 ** 32, (50000, 4), dtype=np.uint64).astype(np.uint32)
    c[0], c[1], c[2] = 0, 0xFFFFFFFF, (0xFFFFFFFF, 0xFFFFF000, 0, 0)
    y = np.empty((len(c), 2))
    lib.t_normal(len(c), dp(np.ascontiguousarray(c)), dp(y))
    w = c.astype(np.uint64)
    u = [((((w[:, k] << np.uint64(32)) | w[:, k + 1]) >> np.uint64(11)).astype(np.float64) + 0.5) * 2.0 ** -53 for k in (0, 2)]
    r = np.sqrt(-2.0 * np.log(u[0]))
    assert np.abs(y[:, 0] - r * np.cos(2 * np.pi * u[1])).max() < 5e-15
    assert np.abs(y[:, 1] - r * np.sin(2 * np.pi * u[1])).max() < 5e-15


def test_normal_cdf_matches_erfc(lib):
    """Against erfc in FP64 (2e-15 near -4, from the rounding of its argument);
    both sides of the table's range, points midway between entries, tiny and
    special values."""
    import math
    g = np.random.default_rng(4)
    x = np.concatenate([g.standard_normal(20000), g.uniform(-5, 5, 20000), 2.0 ** g.uniform(-80, 0, 500) * g.choice([-1, 1], 500),
                        np.arange(-520, 521) / 128.0, [0.0, -0.0, -30.0, 30.0, np.inf, -np.inf, np.nan, -4.0, 4.0]])
    y = np.empty_like(x)
    lib.t_cdf(len(x), dp(x), dp(y))
    want = np.array([0.5 * math.erfc(-v / math.sqrt(2.0)) for v in x])
    assert np.allclose(y, want, rtol=5e-15, atol=0, equal_nan=True)
    assert (y[x == 0] == 0.5).all()
