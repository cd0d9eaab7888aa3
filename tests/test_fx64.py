"""The fixed-point functions of the FP64 paths (csrc/fx64.cuh) against
arbitrary-precision values: the header compiled as plain C++ (its integer code
is what the GPU runs; only the FP32 seeds of the Newton steps differ, so they
are tried with the error that the GPU's approximate instructions may have).
Inputs sit at the edges of the tables' cells, quadrants and exponent ranges
and at random points; tolerances are the bounds stated at each function."""
import ctypes
import os
import subprocess
from decimal import Decimal as D, getcontext

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r'''
#define FX_HOST
#include "fx64.cuh"
using namespace fx64;
extern "C" {
void t_log(int n, const uint32_t* w, uint64_t* o, int* sc) { for (int i = 0; i < n; i++) o[i] = neg_log(w[i], sc[i]); }
void t_sqrt(int n, const uint64_t* a, uint64_t* o, int* e) { for (int i = 0; i < n; i++) o[i] = sqrt58(a[i], e[i]); }
void t_trig(int n, const uint32_t* w, uint64_t* s, uint64_t* c) { for (int i = 0; i < n; i++) trig_quadrant(w[i], s[i], c[i]); }
int t_bm(int n, const uint32_t* a, const uint32_t* b, double k, double* x, double* y) {
  Scale s;
  if (!to_scale(k, s)) return 0;
  for (int i = 0; i < n; i++) box_muller(a[i], b[i], s, x[i], y[i]);
  return 1;
}
int t_bmf(int n, const uint32_t* a, const uint32_t* b, double k, int64_t* x, int64_t* y, double* d) {
  Scale s;
  if (!to_scale(k, s)) return 0;
  for (int i = 0; i < n; i++) {
    box_muller_fixed(a[i], b[i], s.sm, x[i], y[i]);
    d[i] = from_fixed58((x[i] >> 2) + smulhi(y[i], (int64_t)3 << 60), s.se);  // x + 0.75 y
  }
  return 1;
}
void t_logf(int n, const double* y, double k, int ab, double* o) {
  int64_t kf, yf;
  to_fixed57(k, kf);
  for (int i = 0; i < n; i++) o[i] = to_fixed57(y[i], yf) ? logistic_p1_fixed(yf - kf, ab) : -1.0;
}
void t_logistic(int n, const double* y, int ab, double* o) { for (int i = 0; i < n; i++) o[i] = logistic_p1(y[i], ab); }
void t_lnabs(int n, const double* x, double* o) { for (int i = 0; i < n; i++) o[i] = log_abs(x[i]); }
void t_exp(int n, const double* x, double* o) { for (int i = 0; i < n; i++) o[i] = fx64::exp(x[i]); }
}
'''
getcontext().prec = 60
PI = D("3.14159265358979323846264338327950288419716939937510582097494459")


@pytest.fixture(scope="module", params=["0.0f", "2e-7f", "-2e-7f"])
def lib(request, tmp_path_factory):
    d = tmp_path_factory.mktemp("fx64")
    (d / "t.cpp").write_text(SRC)
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-DFX_SEED_ERR=" + request.param,
                           "-I" + os.path.join(ROOT, "paper_1102_4666_gb300", "csrc"), "-o", str(d / "t.so"),
                           str(d / "t.cpp")])
    return ctypes.CDLL(str(d / "t.so"))


def _p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def _sincos(x):
    s, c, t, n = D(0), D(0), D(1), 0
    while abs(t) > D(10) ** -50 or n < 4:
        c, s = (c + t * (-1) ** (n // 2), s) if n % 2 == 0 else (c, s + t * (-1) ** (n // 2))
        n += 1
        t = t * x / n
    return s, c


def _words():
    rng = np.random.default_rng(11)
    edges = [0, 1, 2, 2**32 - 1, 2**32 - 2]
    edges += [min(2**32 - 1, max(0, (1 << b) + o)) for b in range(32) for o in (-1, 0, 1)]
    edges += [2**32 - 1 - (1 << b) for b in range(32)]
    edges += [((128 + j) << 24) + o for j in (0, 1, 126, 127) for o in (-1, 0, 1)]      # cells of the logarithm
    edges += [(j << 24) + o for j in (1, 31, 32, 63, 64, 192, 255) for o in (-1, 0, 1)]  # cells of the angle
    return np.concatenate([rng.integers(0, 2**32, 300), edges]).astype(np.uint32)


def test_logarithm_and_root(lib):
    w = _words()
    n = len(w)
    L, sc, S, e = np.zeros(n, np.uint64), np.zeros(n, np.int32), np.zeros(n, np.uint64), np.zeros(n, np.int32)
    lib.t_log(n, _p(w), _p(L), _p(sc))
    lib.t_sqrt(n, _p(L), _p(S), _p(e))
    for i in range(n):
        got = D(int(L[i])) / D(2) ** int(sc[i])
        assert sc[i] in (59, 69)
        assert abs(got + ((2 * int(w[i]) + 1) * D(2) ** -33).ln()) < D(2) ** (2 - int(sc[i])), int(w[i])
        root = (D(int(L[i])) / D(2) ** 58).sqrt()
        assert abs(D(int(S[i])) * D(2) ** (int(e[i]) - 63) / root - 1) < D(2) ** -60, int(w[i])


def test_sine_and_cosine(lib):
    w = _words()
    n = len(w)
    s, c = np.zeros(n, np.uint64), np.zeros(n, np.uint64)
    lib.t_trig(n, _p(w), _p(s), _p(c))
    for i in range(n):
        es, ec = _sincos(((2 * int(w[i]) + 1) % 2**31) * PI / 2**32)
        assert abs(D(int(s[i])) / 2**63 - es) < D(2) ** -60, int(w[i])
        assert abs(D(int(c[i])) / 2**63 - ec) < D(2) ** -60, int(w[i])


@pytest.mark.parametrize("k", [1.0, 0.0123456789, 2.0**-400, 3.0e100])
def test_box_muller(lib, k):
    """Rounded once: half an ulp of the result, plus the radius's error (at
    most 2^-52 next to u0 = 1) and the trigonometric one times a radius < 8."""
    a = _words()
    b = np.roll(a, 17).copy()
    n = len(a)
    x, y = np.zeros(n), np.zeros(n)
    assert lib.t_bm(n, _p(a), _p(b), ctypes.c_double(k), _p(x), _p(y)) == 1
    for i in range(n):
        r = (-2 * ((2 * int(a[i]) + 1) * D(2) ** -33).ln()).sqrt() * D(k)
        es, ec = _sincos((2 * int(b[i]) + 1) * PI / 2**32)
        for got, want in ((x[i], r * ec), (y[i], r * es)):
            assert abs(D(float(got)) - want) <= abs(want) * D(2) ** -53 + D(k) * D(2) ** -52, (int(a[i]), int(b[i]))


@pytest.mark.parametrize("bad", [0.0, -1.0, float("nan"), float("inf"), 5e-324, 1e300])
def test_scales_outside_the_range_are_refused(lib, bad):
    w = np.zeros(1, np.uint32)
    z = np.zeros(1)
    assert lib.t_bm(1, _p(w), _p(w), ctypes.c_double(bad), _p(z), _p(z)) == 0


@pytest.mark.parametrize("absolute", [0, 1])
def test_logistic(lib, absolute):
    y = np.concatenate([np.random.default_rng(3).standard_normal(200) * 4,
                        [0.0, -0.0, 5e-324, -5e-324, 1e-20, -1e-20, 1e-9, 0.25, 2.0**-60, 18.0, -18.0, 31.9999, -31.9999,
                         32.0, -32.0, 1e3, -1e3, 1e300, -1e300, np.inf, -np.inf]])
    o = np.zeros(len(y))
    lib.t_logistic(len(y), _p(y), absolute, _p(o))
    for i, v in enumerate(y):
        v = abs(v) if absolute else v
        want = 1 + (D(0) if v > 500 else D(1) if v < -500 else 1 / ((2 * D(float(v))).exp() + 1))
        assert abs(D(float(o[i])) - want) < D(2) ** -D("52.9"), v


def test_exp(lib):
    x = np.concatenate([np.random.default_rng(4).standard_normal(200) * 5, np.random.default_rng(5).uniform(-700, 700, 100),
                        [0.0, -0.0, 5e-324, 1e-300, -1e-18, 255.9999, -255.9999, 256.0, -256.0, 4.605170185988092]])
    o = np.zeros(len(x))
    lib.t_exp(len(x), _p(x), _p(o))
    for i, v in enumerate(x):
        bound = D(2) ** -D("52.5") if abs(v) < 256 else D(2) ** -52
        assert abs(D(float(o[i])) / D(float(v)).exp() - 1) < bound, v
    s = np.array([np.inf, -np.inf, 1e5, -1e5, np.nan])
    o = np.zeros(5)
    lib.t_exp(5, _p(s), _p(o))
    assert o[0] == np.inf and o[1] == 0 and o[2] == np.inf and o[3] == 0 and np.isnan(o[4])


def test_log_absolute(lib):
    rng = np.random.default_rng(6)
    x = np.concatenate([100 * np.exp(rng.standard_normal(200)), np.exp(rng.uniform(-700, 700, 100)),
                        [1.0, np.nextafter(1, 2), np.nextafter(1, 0), 2.0, 0.5, 2.2250738585072014e-308, 1.7e308, 100.0],
                        (128 + np.arange(128)) / 256.0, np.nextafter((129 + np.arange(128)) / 256.0, 0)])
    o = np.zeros(len(x))
    lib.t_lnabs(len(x), _p(x), _p(o))
    for i, v in enumerate(x):
        want = D(float(v)).ln()
        assert abs(D(float(o[i])) - want) <= max(abs(want) * D(2) ** -53, D(2) ** -53) + D(2) ** -53, v
    s = np.array([0.0, np.inf, 5e-324, -1.0])
    o = np.zeros(4)
    lib.t_lnabs(4, _p(s), _p(o))
    assert o[0] == -np.inf and o[1] == np.inf and abs(o[2] - np.log(5e-324)) < 1e-12 and np.isnan(o[3])


@pytest.mark.parametrize("k", [1.0, 0.0123456789, 3.0e100])
def test_fixed_normals_and_their_sums(lib, k):
    """x + 3/4 y of a pair: within the truncations of the two products (a few
    2^-58) and the normals' own error, times the scale, and the last rounding."""
    a = _words()
    b = np.roll(a, 17).copy()
    n = len(a)
    x, y, d = np.zeros(n, np.int64), np.zeros(n, np.int64), np.zeros(n)
    assert lib.t_bmf(n, _p(a), _p(b), ctypes.c_double(k), _p(x), _p(y), _p(d)) == 1
    for i in range(n):
        r = (-2 * ((2 * int(a[i]) + 1) * D(2) ** -33).ln()).sqrt() * D(k)
        es, ec = _sincos((2 * int(b[i]) + 1) * PI / 2**32)
        want = r * ec + r * es * D("0.75")
        assert abs(D(float(d[i])) - want) <= abs(want) * D(2) ** -53 + D(k) * D(2) ** -52, (int(a[i]), int(b[i]))


@pytest.mark.parametrize("absolute", [0, 1])
def test_fixed_logistic(lib, absolute):
    k = 4.605170185988092
    y = np.concatenate([k + np.random.default_rng(3).standard_normal(200) * 4,
                        [k, 0.0, -0.0, 5e-324, 1e-9, k + 1e-9, 31.9999, -31.9999, 32.0, -32.0, np.inf, np.nan]])
    o = np.zeros(len(y))
    lib.t_logf(len(y), _p(y), ctypes.c_double(k), absolute, _p(o))
    for i, v in enumerate(y):
        if not abs(v) < 32:
            assert o[i] == -1.0
            continue
        z = D(float(v)) - D(k)
        want = 1 + 1 / ((2 * (abs(z) if absolute else z)).exp() + 1)
        assert abs(D(float(o[i])) - want) < D(2) ** -D("52.9"), v
