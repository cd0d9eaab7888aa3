"""The fixed-point root and normals of the FP64 paths (csrc/fx64.cuh) where the
root's normalised argument comes next to 1, from below and from above: -2 ln u
next to a power of 4, and radicands there.  The bound 2^-60 is the root's own; the check is
in integers, so the same source runs on the host, with seeds off by up to the
2^-22 that the root admits, and on the GPU with the instruction's seeds, over
all 2^32 words."""
import ctypes
import math
import os
import subprocess
from decimal import Decimal, getcontext

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1102_4666_gb300", "csrc")

# S 2^(e - 63) is the root of A 2^-58: S^2 2^(2e - 68) = A, with S in [2^62, 2^63] (to 2^-60).  (2 S)^2 2^-64
# against A 2^(6 - 2e), both at least 2^62: a relative error of 2^-60 of S, with the truncations,
# is less than 32 of the 2^64 units.
COMMON = r'''
#include "fx64.cuh"
FX_FN bool root_ok(uint64_t A, uint64_t S, int e, uint64_t hi) {
  if (S < (1ull << 62) - 4 || S > (1ull << 63) || e > 3 || e < -29) return false;
  const uint64_t want = A << (6 - 2 * e);
  if (want >> (6 - 2 * e) != A) return false;
  const uint64_t got = S >> 63 ? ~0ull : hi;  // hi: high half of (2 S)^2
  return (got > want ? got - want : want - got) < 32;
}
'''
HOST = "#define FX_HOST\n" + COMMON + r'''
using namespace fx64;
extern "C" int roots(long n, const uint64_t* a, uint8_t* ok) {
  int bad = 0;
  for (long i = 0; i < n; i++) {
    int e;
    const uint64_t S = sqrt58(a[i], e);
    ok[i] = root_ok(a[i], S, e, (uint64_t)(((unsigned __int128)(S << 1) * (S << 1)) >> 64));
    bad += !ok[i];
  }
  return bad;
}
extern "C" void radicands(long n, const uint32_t* w, uint64_t* a) {
  int sc;
  for (long i = 0; i < n; i++) a[i] = neg_log(w[i], sc);
}
extern "C" void logs(long n, const double* x, double* o) {
  for (long i = 0; i < n; i++) o[i] = log_abs(x[i]);
}
extern "C" void normals(long n, const uint32_t* w0, const uint32_t* w1, double* z0, double* z1) {
  Scale s;
  to_scale(1.0, s);
  for (long i = 0; i < n; i++) box_muller(w0[i], w1[i], s, z0[i], z1[i]);
}
'''
DEVICE = COMMON + r'''
__global__ void k_all(unsigned long long* out) {  // wrong words, one of them
  for (uint64_t w = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; w < (1ull << 32); w += (uint64_t)gridDim.x * blockDim.x) {
    int sc, e;
    const uint64_t A = fx64::neg_log((uint32_t)w, sc), S = fx64::sqrt58(A, e);
    if (!root_ok(A, S, e, __umul64hi(S << 1, S << 1))) {
      atomicAdd(out, 1ull);
      out[1] = w;
    }
  }
}
__global__ void k_pairs(int n, const uint32_t* w0, const uint32_t* w1, double* z0, double* z1) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  fx64::Scale s;
  fx64::to_scale(1.0, s);
  if (i < n) fx64::box_muller(w0[i], w1[i], s, z0[i], z1[i]);
}
extern "C" int all_words(unsigned long long* out) {
  k_all<<<1216, 256>>>(out);
  return (int)cudaDeviceSynchronize();
}
extern "C" int pairs(int n, const uint32_t* w0, const uint32_t* w1, double* z0, double* z1) {
  k_pairs<<<(n + 255) / 256, 256>>>(n, w0, w1, z0, z1);
  return (int)cudaDeviceSynchronize();
}
'''


def _p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def _words():
    """w with u = (2 w + 1) 2^-33 next to exp(-4^k / 2), that is -2 ln u next to 4^k."""
    out = []
    for k in range(-16, 3):
        c = int(math.exp(-(4.0 ** k) / 2) * 2.0 ** 32 - 0.5)
        out.append(np.arange(max(0, c - 1500), min(2**32, c + 1500)))
    return np.unique(np.concatenate(out)).astype(np.uint32)


@pytest.mark.parametrize("seed_error", ["0.0f", "6e-8f", "-6e-8f", "1.2e-7f", "-1.2e-7f", "2.38e-7f", "-2.38e-7f"])
def test_root_next_to_powers_of_four(seed_error, tmp_path):
    (tmp_path / "t.cpp").write_text(HOST)
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-DFX_SEED_ERR=" + seed_error, "-I" + CSRC,
                           "-o", str(tmp_path / "t.so"), str(tmp_path / "t.cpp")])
    lib = ctypes.CDLL(str(tmp_path / "t.so"))
    w = _words()
    a = np.zeros(len(w), np.uint64)
    lib.radicands(ctypes.c_long(len(w)), _p(w), _p(a))
    step = [0, 1, 2, 3, 5, 1 << 10, (1 << 20) - 1]
    direct = [4**k + s * (4**k >> sh) + o for k in range(14, 32) for sh in range(18, 28) for s in (-1, 1) for o in step + [-v for v in step]]
    a = np.concatenate([a, np.array([v for v in direct if 0 < v < 2**64], dtype=np.uint64)])
    ok = np.zeros(len(a), np.uint8)
    assert lib.roots(ctypes.c_long(len(a)), _p(a), _p(ok)) == 0, a[ok == 0][:8]
    # the pair itself, within 2^-51 of numpy's FP64 formula's
    w1 = (w * np.uint32(2654435761) + np.uint32(12345)).astype(np.uint32)
    z0, z1 = np.zeros(len(w)), np.zeros(len(w))
    lib.normals(ctypes.c_long(len(w)), _p(w), _p(w1), _p(z0), _p(z1))
    _check_pairs(w, w1, z0, z1)


def _check_pairs(w0, w1, z0, z1):
    """Both sides are off by some ulps of a radius below 6.8 (1e-14 bounds a dozen of
    them); a wrong root is off by a factor of two or more."""
    u = 1.0 - (w0 + 0.5) * 2.0 ** -32
    rad = np.sqrt(-2.0 * np.log1p(-u))
    th = np.pi * ((w1 + 0.5) * 2.0 ** -31)
    assert np.max(np.abs(z0 - rad * np.cos(th))) < 1e-14
    assert np.max(np.abs(z1 - rad * np.sin(th))) < 1e-14


def test_logarithm_of_prices(tmp_path):
    """Within 0.63 ulp (an eighth from the fixed point, half from the rounding) of the true value,
    next to 1, where the sum cancels, next to the changes of form, and far out."""
    (tmp_path / "t.cpp").write_text(HOST)
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I" + CSRC, "-o", str(tmp_path / "t.so"),
                           str(tmp_path / "t.cpp")])
    lib = ctypes.CDLL(str(tmp_path / "t.so"))
    rng = np.random.default_rng(9)
    near = [1.0 + s * 2.0 ** -k for k in range(1, 53) for s in (-1.0, 1.0)]
    forms = [f * b for b in (math.exp(0.25), math.exp(-0.25), 2.0 ** 21, 2.0 ** 22, 2.0 ** -21, 2.0 ** -22, 2.0 ** -23)
             for f in (1.0, 1.0 - 1e-15, 1.0 + 1e-15, 0.999, 1.001)]
    x = np.concatenate([near, forms, np.exp(rng.uniform(-1, 1, 1500)), 100.0 * np.exp(rng.uniform(-1.5, 1.5, 1500)),
                        np.exp(rng.uniform(-700, 700, 1500))])
    x = x[x != 1.0]
    o = np.zeros(len(x))
    lib.logs(ctypes.c_long(len(x)), _p(x), _p(o))
    getcontext().prec = 50
    for v, got in zip(x, o):
        want = Decimal(float(v)).ln()
        ulp = Decimal(float(np.spacing(abs(float(want)))))
        assert abs(Decimal(float(got)) - want) <= ulp * Decimal("0.63"), v


@pytest.mark.gpu
def test_every_word_on_the_gpu(tmp_path):
    import torch
    from paper_1102_4666_gb300 import _build
    (tmp_path / "t.cu").write_text(DEVICE)
    subprocess.check_call([_build.nvcc(), "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17", "-shared",
                           "-Xcompiler", "-fPIC", "-I" + CSRC, "-o", str(tmp_path / "t.so"), str(tmp_path / "t.cu")])
    lib = ctypes.CDLL(str(tmp_path / "t.so"))
    out = torch.zeros(2, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    assert lib.all_words(ctypes.c_void_p(out.data_ptr())) == 0
    assert out[0].item() == 0, out.tolist()
    w = _words()
    w1 = (w * np.uint32(2654435761) + np.uint32(12345)).astype(np.uint32)
    d0, d1 = (torch.from_numpy(v.view(np.int32).copy()).cuda() for v in (w, w1))
    z = torch.zeros(2, len(w), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    ptr = [ctypes.c_void_p(v.data_ptr()) for v in (d0, d1, z[0], z[1])]
    assert lib.pairs(len(w), *ptr) == 0
    _check_pairs(w, w1, z[0].cpu().numpy(), z[1].cpu().numpy())
