"""The fixed-point division (csrc/fixed.cuh, host build) gives the bits of the FP64
division, which it stands in for."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1903_08741_gb300", "csrc")
SRC = r"""
#include "fixed.cuh"
extern "C" void t_div(int n, const double* a, const double* b, double* q) { for (int i = 0; i < n; ++i) q[i] = rich_fx::fx_div(a[i], b[i]); }
"""


@pytest.fixture(scope="module")
def div(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed")
    (d / "t.cpp").write_text(SRC)
    subprocess.run(["g++", "-O1", "-std=gnu++17", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "t.so"), str(d / "t.cpp")],
                   check=True)
    lib = C.CDLL(str(d / "t.so"))

    def call(a, b):
        a, b = np.ascontiguousarray(a, dtype=np.float64), np.ascontiguousarray(b, dtype=np.float64)
        q = np.empty_like(a)
        lib.t_div(len(a), *(v.ctypes.data_as(C.c_void_p) for v in (a, b, q)))
        return q
    return call


def mantissas(g, k):
    """Random, and both ends of the binade and its middle to a few units."""
    near = np.array([1.0, 1.5, 2.0])[g.integers(0, 3, k)] + g.integers(-40, 41, k) * 2.0 ** -52
    return np.where(g.random(k) < 0.5, 1 + g.random(k), np.clip(near, 1.0, np.nextafter(2.0, 0.0)))


@pytest.mark.parametrize("kind", ["quotients", "reciprocals", "near_one", "near_midpoints"])
def test_quotients_are_correctly_rounded(div, kind):
    g = np.random.default_rng(["quotients", "reciprocals", "near_one", "near_midpoints"].index(kind))
    k = 1_000_000
    b = mantissas(g, k) * 2.0 ** g.integers(-450, 450, k)
    if kind == "reciprocals":
        a = np.ones(k)
    elif kind == "near_one":                        # both sides of a power of two
        a = b * (1 + g.integers(-3, 4, k) * 2.0 ** -52)
    elif kind == "near_midpoints":                  # a is b times a 53-bit number, to a unit
        a = np.nextafter(b * mantissas(g, k), np.where(g.random(k) < 0.5, 0.0, np.inf))
    else:
        a = mantissas(g, k) * 2.0 ** g.integers(-450, 450, k)
    assert np.array_equal(div(a, b), a / b)


def test_every_exponent_of_the_quotient(div):
    """The whole range, over the line where the FP64 division takes over."""
    e = np.arange(-1080, 1080)
    for m, n in ((1.0, np.nextafter(2.0, 1.0)), (np.nextafter(2.0, 1.0), 1.0), (1.7, 1.3), (1.3, 1.7)):
        h = e // 2
        a, b = np.ldexp(m, e - h), np.ldexp(n, -h)
        with np.errstate(all="ignore"):
            assert np.array_equal(div(a, b), a / b)
