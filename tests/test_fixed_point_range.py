"""Products of a shape function with a fixed-point separation at the edges of their range (csrc/otm_fix.cuh, the
functions the kernels call, compiled for the host), against exact fractions."""
import ctypes as C
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2206_08772_gb300", "csrc")

SRC = r'''
#include <cmath>
#include "otm_fix.cuh"
using namespace otm;
extern "C" void nd(double N, const i64 *d, int fb, double *e)
{
    fix_nd(N, d[0], d[1], d[2], fb, std::ldexp(1.0, -fb), e[0], e[1], e[2]);
}
extern "C" int force(const double *Q, double N, const i64 *d, int fb, double *f)
{
    double q[9];
    for (int i = 0; i < 9; i++) q[i] = Q[i];
    FixRows R;
    fix_rows(q, fb, R);
    return force_fix(R, N, d[0], d[1], d[2], f[0], f[1], f[2]);
}
'''


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("fixr")
    (d / "r.cpp").write_text(SRC)
    so = str(d / "r.so")
    subprocess.run([gxx, "-O2", "-std=gnu++17", "-shared", "-fPIC", "-I", CSRC, str(d / "r.cpp"), "-o", so], check=True)
    L = C.CDLL(so)
    L.nd.argtypes = [C.c_double, C.c_void_p, C.c_int, C.c_void_p]
    L.nd.restype = None
    L.force.argtypes = [C.c_void_p, C.c_double, C.c_void_p, C.c_int, C.c_void_p]
    return L


def ptr(a):
    return a.ctypes.data_as(C.c_void_p)


WEIGHTS = [1.0, 0.5, 0.5 * (1 + 2.0 ** -52), 1 - 2.0 ** -53, 2.0 ** -31 * 1.3, 1e-120, 2.0 ** -423, 2.0 ** -422 * 1.9, 1e-150,
           1e-290, 1e-300, 2.3e-308, 1e-310]


def edges():
    out = {0, 1, -1, 12345}
    for b in (32, 33, 34, 35, 47, 62):
        for k in (0, 1, 2, 3, 5, 1000, 2 ** 30, 2 ** 31 + 7):
            for s in (1, -1):
                out |= {s * (2 ** b + k), s * (2 ** b - k), s * (3 * 2 ** (b - 1) + k)}
    return sorted(d for d in out if abs(d) < 2 ** 63)


@pytest.mark.parametrize("fb", [71, 119, -59])
@pytest.mark.parametrize("N", WEIGHTS)
def test_shape_function_times_separation(lib, N, fb):
    """Two roundings (2^-53 of the value each, 2^-1075 below the normal range, times N there), and one unit of the
    separation."""
    rng = np.random.default_rng(1)
    e = np.zeros(3)
    for D in edges():
        for other in (2 ** 61 + 12345, 2 ** 33 - 1):
            d = np.array([D, other, -other], np.int64)[rng.permutation(3)]
            lib.nd(N, ptr(d), fb, ptr(e))
            for i in range(3):
                ref = Fraction(N) * int(d[i]) / Fraction(2) ** fb
                tol = abs(ref) / 2 ** 52 + Fraction(N) / Fraction(2) ** fb + Fraction(1, 2 ** 1074)
                assert abs(Fraction(float(e[i])) - ref) <= tol, (int(d[i]), float(e[i]), float(ref))


@pytest.mark.parametrize("fb", [71, 119])
@pytest.mark.parametrize("N", WEIGHTS)
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -420, 2.0 ** 420])
def test_force_products_at_the_edges(lib, N, fb, scale):
    """In range or refused, never wrong: Q selects one component a row, so that F takes each edge value (times 2^-3,
    the units of the rows). Bound as of the general rows: half an ulp, and 2^-56 of the row's entry times N and 2^62
    units."""
    Q = np.ascontiguousarray(np.eye(3).ravel() * scale * 1.25)
    f = np.zeros(3)
    taken = 0
    for D in edges():
        if abs(D) >= 2 ** 62:
            continue
        for m in (1, 8):
            d = np.array([D * m, 2 ** 60, -(2 ** 61)], dtype=object)
            if abs(d[0]) >= 2 ** 62:
                continue
            d = d.astype(np.int64)
            if not lib.force(ptr(Q), N, ptr(d), fb, ptr(f)):
                continue
            taken += 1
            for i in range(3):
                ref = Fraction(N) * Fraction(float(Q[4 * i])) * int(d[i]) / Fraction(2) ** fb
                tol = abs(ref) / 2 ** 53 + Fraction(float(Q[4 * i])) * Fraction(N) * Fraction(2 ** 62, 2 ** fb) / 2 ** 56
                assert abs(Fraction(float(f[i])) - ref) <= tol, (int(d[i]), float(f[i]), float(ref))
    assert taken > 0 or N < 2.0 ** -420
