"""The fixed-point arithmetic of the FP64 path's LME evaluation (csrc/otm_fix.cuh), compiled for the host
and checked against 60-digit decimal arithmetic: exponent, weights, the sums Z, r, A and N d."""
import ctypes as C
import os
import shutil
import subprocess
from decimal import Decimal, getcontext
from fractions import Fraction

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2206_08772_gb300", "csrc")

SRC = r'''
#include <cmath>
#include <cstdlib>
#include <vector>
#include "otm_fix.cuh"
using namespace otm;
// the sums of one evaluation (32 lanes) as the kernel forms them; out: Z, r, A in physical units, then the
// weights; prod: N d; returns 0, 1 centre out of range, 2 weights out of the window
extern "C" int eval(int n, const double *x, const double *xp, const double *lam, double beta, double shift, int fb,
                    const u64 *table, u64 bq, double *out, double *w, double *prod)
{
    std::vector<i64> X(3 * n);
    for (int k = 0; k < 3 * n; k++) X[k] = fix_from_double(x[k], fb);
    i64 P[3], v[3];
    double l2 = 0;
    for (int i = 0; i < 3; i++) {
        P[i] = fix_from_double(xp[i], fb);
        const double c = lam[i] * std::ldexp(1.0, fb) / (2 * beta);
        if (!(std::fabs(c) < kFixT)) return 1;
        v[i] = std::llrint(c);
        l2 += lam[i] * lam[i];
    }
    const i64 cst = std::llrint((l2 * 64.0 / (beta * std::log(2.0)) - shift * kFixYScale) * kFixYOne);
    i64 t[10] = {0};
    for (int lane = 0; lane < 32; lane++) {
        FixSums s;
        fix_sums_zero(s);
        for (int k = lane; k < n; k += 32)
            w[k] = fix_pair<true>(X[3 * k], X[3 * k + 1], X[3 * k + 2], P[0] - v[0], P[1] - v[1], P[2] - v[2], cst, bq, table, s);
        if (s.top >= 0) return 2;
        i64 c[10];
        fix_combine(s, c);
        for (int i = 0; i < 10; i++) t[i] += c[i];
    }
    const int I[6] = {0, 1, 2, 0, 1, 0}, J[6] = {0, 1, 2, 1, 2, 2};
    out[0] = std::ldexp((double)t[0], -63);
    for (int i = 0; i < 3; i++) out[1 + i] = std::ldexp((double)fix_r_about(t[0], t[1 + i], v[i]), -fb);
    for (int q = 0; q < 6; q++) {
        const i64 rd = fix_r_about(t[0], t[1 + J[q]], v[J[q]]);
        out[4 + q] = std::ldexp((double)fix_a_about(t[4 + q], t[1 + I[q]], rd, v[I[q]], v[J[q]]), 60 - 2 * fb);
    }
    for (int k = 0; k < n; k++)
        for (int i = 0; i < 3; i++) {
            const i64 D = P[i] - X[3 * k + i];
            const u64 nb = fx_d_bits(w[k]);
            prod[3 * k + i] = llabs(D) >= (2LL << 32)
                                  ? fix_mul_double(((nb & 0xfffffffffffffULL) | 0x10000000000000ULL) << 11, (int)(nb >> 52), D, fb)
                                  : w[k] * std::ldexp((double)D, -fb);
        }
    return 0;
}
'''


KIN = r'''
// one warp's kinematics sums: out[12] = sum N du (3), G = sum du (x) e (9)
extern "C" void gather(int n, const double *row, const double *du, int fu, int fe, double *out)
{
    i64 t[12] = {0};
    for (int lane = 0; lane < 32; lane++) {
        KinFixSums s;
        for (int i = 0; i < 12; i++) s.hh[i] = s.hl[i] = 0, s.ll[i] = 0.f;
        for (int k = lane; k < n; k += 32)
        {
            int uh[3], ul[3];
            for (int i = 0; i < 3; i++) kin_fix_split(fix_from_double(du[3 * k + i], fu), uh[i], ul[i]);
            kin_fix_pair(fix_floor(row[4 * k], 62), fix_floor(row[4 * k + 1], fe), fix_floor(row[4 * k + 2], fe),
                         fix_floor(row[4 * k + 3], fe), uh, ul, s);
        }
        for (int i = 0; i < 12; i++) t[i] += kin_fix_combine(s, i);
    }
    for (int i = 0; i < 12; i++) out[i] = std::ldexp((double)t[i], kin_fix_exponent(fu, i < 3 ? 62 : fe));
}
'''


FORCE = r'''
// f = N Q D 2^-fb; returns whether the rows are in range
extern "C" int force(const double *Q, double N, const i64 *D, int fb, double *f)
{
    double q[9];
    for (int i = 0; i < 9; i++) q[i] = Q[i];
    FixRows R;
    fix_rows(q, fb, R);
    const int dh[3] = {(int)((D[0] + 0x80000000LL) >> 32), (int)((D[1] + 0x80000000LL) >> 32), (int)((D[2] + 0x80000000LL) >> 32)};
    const int dl[3] = {(int)D[0], (int)D[1], (int)D[2]};
    const u64 nb = fx_d_bits(N), nm = ((nb & 0xfffffffffffffULL) | 0x10000000000000ULL) << 11;
    if (R.ok) for (int i = 0; i < 3; i++) f[i] = fix_mul_double(nm, (int)(nb >> 52), fix_row_dot(R, i, dh, dl), R.fb[i]);
    return R.ok;
}
'''

SUMS = r'''
// node sums of n terms: the two's complement 128-bit total
extern "C" void sum128(int n, const double *v, int emax, u64 *out)
{
    Sum128 a = {0, 0};
    for (int i = 0; i < n; i++) add_fixed(a, v[i], emax);
    const u128 t = a.v + (u128)(u64)a.neg;
    out[0] = (u64)t;
    out[1] = (u64)(t >> 64);
}
extern "C" void sum64(int n, const float *v, int emax, u64 *out)
{
    Sum64 a = {0, 0};
    for (int i = 0; i < n; i++) add_fixed(a, v[i], emax);
    out[0] = a.v + (u64)a.neg;
    out[1] = (u64)((i64)out[0] >> 63);
}
'''


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("fix")
    (d / "fix.cpp").write_text(SRC + KIN + FORCE + SUMS)
    so = str(d / "fix.so")
    subprocess.run([gxx, "-O2", "-std=gnu++17", "-shared", "-fPIC", "-I", CSRC, str(d / "fix.cpp"), "-o", so], check=True)
    L = C.CDLL(so)
    L.eval.argtypes = [C.c_int] + [C.c_void_p] * 3 + [C.c_double, C.c_double, C.c_int, C.c_void_p, C.c_uint64] + [C.c_void_p] * 3
    L.gather.argtypes = [C.c_int, C.c_void_p, C.c_void_p, C.c_int, C.c_int, C.c_void_p]
    L.gather.restype = L.sum128.restype = L.sum64.restype = None
    L.force.argtypes = [C.c_void_p, C.c_double, C.c_void_p, C.c_int, C.c_void_p]
    L.sum128.argtypes = L.sum64.argtypes = [C.c_int, C.c_void_p, C.c_int, C.c_void_p]
    return L


# spacing, origin in spacings, whole ball or a corner of the body, centre offset lambda h, support tolerance
@pytest.mark.parametrize("h,origin,corner,lam_h,tol", [
    (0.12e-3, 100.0, False, 0.0, 1e-6), (0.17e-3, 0.0, False, 0.3, 1e-6), (1.0, -3000.0, False, 0.1, 1e-6),
    (0.23e-3, 40.0, True, 0.8, 1e-6), (3.0e-3, 7.0, False, 0.05, 1e-9), (5.0e-3, 1.0, False, 0.0, 1e-2)])
def test_fixed_point_evaluation(lib, h, origin, corner, lam_h, tol):
    getcontext().prec = 60
    rng = np.random.default_rng(int(1e6 * h) + int(corner))
    beta = 0.8 / (h * h)
    rs = np.sqrt(np.log(1 / tol) / beta)
    m = int(rs / h) + 2
    g = np.arange(0 if corner else -m, m + 1)
    x = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3) * h + origin * h
    x = x + rng.uniform(-0.02, 0.02, x.shape) * h
    xp = (origin + (0.3 if corner else 0.0)) * h + rng.uniform(-0.2, 0.2, 3) * h
    x = np.ascontiguousarray(x[((xp - x) ** 2).sum(1) <= rs * rs][:384])
    lam = rng.uniform(-1, 1, 3) * lam_h / h
    n = len(x)
    # constants as the library derives them: 2^63 units = 2^ex >= 2.2 support radii
    fb = 63 - int(np.frexp(2.2 * rs)[1])
    D = Decimal
    ln2 = D(2).ln()
    a = D(2) ** (32 - fb)
    bq = int(D(beta) * 256 / ln2 * a * a * D(2) ** 109)
    assert bq < 2 ** 64
    table = np.array([int((D(2) ** (D(j) / 1024)) * D(2) ** 63 + D("0.5")) for j in range(1024)], np.uint64)
    d = [[D(float(xp[i])) - D(float(x[k, i])) for i in range(3)] for k in range(n)]
    # the kernel's centre is lambda / (2 beta) in whole units: the reference takes that lambda
    v = [int(np.rint(lam[i] * 2.0 ** fb / (2 * beta))) for i in range(3)]
    ld = [D(v[i]) * D(2) ** -fb * 2 * D(beta) for i in range(3)]
    f = [-D(beta) * sum(c * c for c in dk) + sum(l * c for l, c in zip(ld, dk)) for dk in d]
    shift = float(sum(t.exp() for t in f).ln()) + 1.0
    wr = [(t - D(shift)).exp() for t in f]
    out, w, prod = np.zeros(10), np.zeros(n), np.zeros((n, 3))
    ptr = lambda t: t.ctypes.data_as(C.c_void_p)
    st = lib.eval(n, ptr(x), ptr(xp), ptr(lam), beta, shift, fb, ptr(table), bq, ptr(out), ptr(w), ptr(prod))
    assert st == 0
    Z = sum(wr)
    # weights relative to Z: half an ulp of the FP64 weight and Z each, 2e-17 per exponent unit, truncation
    for k in range(n):
        assert abs(D(float(w[k])) / D(float(out[0])) * Z / wr[k] - 1) <= D("8e-16")
    ij = [(0, 0), (1, 1), (2, 2), (0, 1), (1, 2), (0, 2)]
    tr = sum(wk * sum(c * c for c in dk) for wk, dk in zip(wr, d)) / Z
    for i in range(3):
        ref = sum(wk * dk[i] for wk, dk in zip(wr, d)) / Z
        assert abs(D(float(out[1 + i])) / D(float(out[0])) - ref) <= D("4e-16") * tr.sqrt()
    for q, (i, j) in enumerate(ij):
        ref = sum(wk * dk[i] * dk[j] for wk, dk in zip(wr, d)) / Z
        assert abs(D(float(out[4 + q])) / D(float(out[0])) - ref) <= D("2e-15") * tr
    for k in range(n):
        for i in range(3):
            ref = D(float(w[k])) * d[k][i]
            # half an ulp, and half a unit of each coordinate
            assert abs(D(float(prod[k, i])) - ref) <= D(2) ** -53 * abs(ref) + D(float(w[k])) * D(2) ** (1 - fb)


@pytest.mark.parametrize("n,speed", [(1, 0.02), (33, 0.499), (286, 0.02), (384, 0.499), (286, 1e-9)])
def test_fixed_point_kinematics_gather(lib, n, speed):
    """sum N du and sum du (x) e of one support with increments up to half a spacing, all of one sign
    (the largest sums). Units: du 2^-57 h at most, N 2^-61, e 2^-61 of at most twice r_s; dropped low products and
    truncations are a few units each: 2^-57 h and 2^-57 h r_s hold for 384 pairs with sum N = 1."""
    h, rs = 1.3e-4, 5.4e-4
    rng = np.random.default_rng(n)
    N = rng.uniform(0.1, 1.0, n) ** 6
    N /= N.sum()
    row = np.ascontiguousarray(np.concatenate([N[:, None], N[:, None] * rng.uniform(-rs, rs, (n, 3))], 1))
    du = np.ascontiguousarray(rng.uniform(0.9, 1.0, (n, 3)) * speed * h)
    fu, fe = 57 - int(np.floor(np.log2(h))), 61 - int(np.floor(np.log2(rs)))
    out = np.zeros(12)
    ptr = lambda t: t.ctypes.data_as(C.c_void_p)
    lib.gather(n, ptr(row), ptr(du), fu, fe, ptr(out))
    D = Decimal
    for i in range(3):
        ref = sum(D(float(row[k, 0])) * D(float(du[k, i])) for k in range(n))
        assert abs(D(float(out[i])) - ref) <= D(2) ** -53 * abs(ref) + D(2) ** -57 * D(h)
        for j in range(3):
            ref = sum(D(float(du[k, i])) * D(float(row[k, 1 + j])) for k in range(n))
            assert abs(D(float(out[3 + 3 * i + j])) - ref) <= D(2) ** -53 * abs(ref) + D(2) ** -57 * D(h) * D(rs)


@pytest.mark.parametrize("emax", [1023, 3, -40, -900])
def test_node_sum_terms(lib, emax):
    """Node sums: each term is exactly trunc(v 2^(110 - emax)) (FP64) or trunc(v 2^(46 - emax)) (FP32) for exponents
    from emax down past the last unit; zero, subnormal and non-finite terms count nothing."""
    rng = np.random.default_rng(emax + 1000)
    for bits, lsb, lo, fn in ((52, 110, -1022, lib.sum128), (23, 46, -126, lib.sum64)):
        e = emax if bits == 52 else max(min(emax, 127), -60)
        ex = np.concatenate([np.arange(e - 150, e + 1), [e, e, e - 63, e - 64, e - 47, e - 46]])
        ex = np.repeat(ex[ex >= lo], 3)
        m = rng.integers(0, 1 << bits, ex.size)
        m[::7] = 0
        m[1::7] = (1 << bits) - 1
        sg = np.where(rng.uniform(size=ex.size) < 0.5, -1.0, 1.0)
        v = np.ldexp(1.0 + m * 2.0 ** -bits, ex) * sg
        tiny = np.ldexp(1.0, lo - 3)
        v = np.concatenate([v, [0.0, -0.0, tiny, -tiny, np.inf, -np.inf, np.nan]])
        v = np.ascontiguousarray(v, np.float64 if bits == 52 else np.float32)
        out = np.zeros(2, np.uint64)
        fn(v.size, v.ctypes.data_as(C.c_void_p), e, out.ctypes.data_as(C.c_void_p))
        got = int(out[0]) | int(out[1]) << 64
        got -= (1 << 128) if got >> 127 else 0
        # whole numbers by shifting the significand, so that nothing is rounded
        ref = 0
        for mk, ek, sk in zip(m, ex, sg):
            s = int(ek) - bits + lsb - e
            t = (1 << bits) | int(mk)
            ref += int(sk) * (t << s if s >= 0 else t >> -s)
        assert got == ref


@pytest.mark.parametrize("scale,spread", [(1.0, 0), (1e-90, 3), (1e60, 12), (3e7, 40)])
def test_force_rows(lib, scale, spread):
    """f = N Q d with rows of Q of any scale and entries up to 2^spread apart: half an ulp of f and 2^-56 of the
    row's largest entry times N and 2^62 units (5 units of F and one of the product); zero and infinite rows are out
    of range."""
    rng = np.random.default_rng(spread)
    fb = 70
    ptr = lambda t: t.ctypes.data_as(C.c_void_p)
    f = np.zeros(3)
    for _ in range(200):
        Q = np.ascontiguousarray(rng.uniform(-1, 1, 9) * scale * 2.0 ** rng.integers(-spread, 1, 9))
        d = rng.integers(-(1 << 62) + 1, 1 << 62, 3)
        N = float(rng.uniform(0.5, 1.0) * 2.0 ** rng.integers(-30, 1))
        assert lib.force(ptr(Q), N, ptr(d), fb, ptr(f))
        for i in range(3):
            q = [Fraction(float(v)) for v in Q[3 * i:3 * i + 3]]
            ref = sum(a * int(b) for a, b in zip(q, d)) * Fraction(N) / 2 ** fb
            tol = abs(ref) / 2 ** 53 + max(abs(a) for a in q) * Fraction(N) * Fraction(2 ** 62, 2 ** fb) / 2 ** 56
            assert abs(Fraction(float(f[i])) - ref) <= tol
    for bad in (0.0, np.inf, np.nan):
        Q = np.ones(9)
        Q[3:6] = bad
        assert not lib.force(ptr(Q), 0.5, ptr(d), fb, ptr(f))
