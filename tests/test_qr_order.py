"""The pivoted-QR kernel (csrc/k_qr.cu) with one CTA behind all others in every
step: whatever the timing of the CTAs, every one has to choose the same pivot
and leave the same bits.  The kernel's own source is compiled for the host: a
CTA is an OS thread, its 256 threads are coroutines of it that change over at
the block's and the warps' synchronisations, and the CTA that is to be late
reads other CTAs' results only when these wait at the step's grid barrier."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHIM = r'''
#include <math.h>
#include <stdint.h>
#include <string.h>
#include <thread>
#include <ucontext.h>
#include <vector>
using std::isnan;
#define __global__
#define __device__
#define __forceinline__ inline
#define __launch_bounds__(...)
#define __shared__ static thread_local
#define ST_TIMEOUT 2
struct V3 { int x; };
struct Emu {  // one CTA
  ucontext_t main, ctx[256];
  std::vector<char> stack[256];
  bool done[256];
  int cur, arrived, gen, warp_arrived[8], warp_gen[8];
  uint64_t lane[8][2][32];
  V3 block, grid;
  double* smem;
  uint32_t* sync;
  int steps, late;
  void (*body)(void*);
  void* arg;
};
static thread_local Emu* E;
struct Tid { operator int() const { return E->cur; } };
struct { Tid x; } threadIdx;
#define blockIdx (E->block)
#define gridDim (E->grid)
static struct { int x = 256; } blockDim;
static void yield() { swapcontext(&E->ctx[E->cur], &E->main); }
static void __syncthreads() {
  const int g = E->gen;
  if (++E->arrived == 256) { E->arrived = 0; ++E->gen; }
  while (E->gen == g) yield();
}
template <typename T> static T __shfl_xor_sync(unsigned, T v, int o) {
  const int w = E->cur >> 5, l = E->cur & 31, g = E->warp_gen[w];
  memcpy(&E->lane[w][g & 1][l], &v, sizeof(T));
  if (++E->warp_arrived[w] == 32) { E->warp_arrived[w] = 0; ++E->warp_gen[w]; }
  while (E->warp_gen[w] == g) yield();
  memcpy(&v, &E->lane[w][g & 1][l ^ o], sizeof(T));
  return v;
}
// the late CTA reads what others may write when all of them wait for it
static double __ldcg(const double* p) {
  if (E->late)
    while (__atomic_load_n(E->sync, __ATOMIC_ACQUIRE) < (uint32_t)(E->steps * E->grid.x + E->grid.x - 1)) std::this_thread::yield();
  double v;
  __atomic_load((double*)p, &v, __ATOMIC_ACQUIRE);
  return v;
}
static void atomicAdd(uint32_t* p, uint32_t v) { ++E->steps; __atomic_fetch_add(p, v, __ATOMIC_SEQ_CST); }
static void atomicExch(uint32_t* p, uint32_t v) { __atomic_store_n(p, v, __ATOMIC_SEQ_CST); }
static void atomicOr(int* p, int v) { __atomic_fetch_or(p, v, __ATOMIC_SEQ_CST); }
static void __threadfence() { __atomic_thread_fence(__ATOMIC_SEQ_CST); }
static long long __double_as_longlong(double a) { long long b; memcpy(&b, &a, 8); return b; }
static double __longlong_as_double(long long a) { double b; memcpy(&b, &a, 8); return b; }
static void fiber() {
  E->body(E->arg);
  E->done[E->cur] = true;
  swapcontext(&E->ctx[E->cur], &E->main);
}
static void run_cta(Emu* e) {
  E = e;
  for (int t = 0; t < 256; t++) {
    e->stack[t].resize(32768);
    getcontext(&e->ctx[t]);
    e->ctx[t].uc_stack.ss_sp = e->stack[t].data();
    e->ctx[t].uc_stack.ss_size = e->stack[t].size();
    e->ctx[t].uc_link = nullptr;
    makecontext(&e->ctx[t], fiber, 0);
    e->done[t] = false;
  }
  for (bool left = true; left;) {
    left = false;
    for (int t = 0; t < 256; t++)
      if (!e->done[t]) {
        e->cur = t;
        swapcontext(&e->main, &e->ctx[t]);
        left = left || !e->done[t];
      }
  }
}
'''
DRIVER = r'''
struct Call {
  int n, n_pad, p, steps, stage, keep;
  double *W, *y, *nrm;
  int* perm;
  uint32_t* sync;
  int* status;
};
static void body(void* q) {
  Call& c = *(Call*)q;
  auto f = c.keep ? k_qr_factor<true, true> : c.stage ? k_qr_factor<true, false> : k_qr_factor<false, false>;
  f(c.n, c.n_pad, c.p, c.steps, c.W, c.y, c.nrm, c.perm, c.sync, c.status);
}
// the norms' array and what follows it are the caller's
extern "C" int factor(int n, int p, int grid, int late, int stage, int keep, double* W, double* y, double* nrm, int* perm) {
  uint32_t sync[2] = {0, 0};
  int status = 0;
  Call c{n, n, p, p < n ? p : n, stage, keep, W, y, nrm, perm, sync, &status};
  std::vector<std::thread> t;
  for (int b = 0; b < grid; b++)
    t.emplace_back([&, b] {
      Emu* e = new Emu();
      std::vector<double> smem((size_t)n * (p / grid + 3) + p * 2 + 64);
      e->block.x = b;
      e->grid.x = grid;
      e->smem = smem.data();
      e->sync = sync;
      e->late = b == late;
      e->body = body;
      e->arg = &c;
      run_cta(e);
      delete e;
    });
  for (auto& q : t) q.join();
  return status;
}
'''


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("qr")
    src = open(os.path.join(ROOT, "paper_1102_4666_gb300", "csrc", "k_qr.cu")).read()
    i, j = src.index("constexpr int QR_THREADS"), src.index("// basic solution: rank r")
    body = src[i:j].replace("extern __shared__ double qr_smem[];", "double* qr_smem = E->smem;")
    # a late CTA makes the others poll for long
    assert "QR_WAIT_LIMIT = 1u << 24" in body
    (d / "t.cpp").write_text(SHIM + body.replace("QR_WAIT_LIMIT = 1u << 24", "QR_WAIT_LIMIT = ~0u") + DRIVER)
    subprocess.check_call(["g++", "-O1", "-w", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-pthread",
                           "-o", str(d / "t.so"), str(d / "t.cpp")])
    return ctypes.CDLL(str(d / "t.so"))


def _p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def _factor(lib, X, c, grid, late, stage, keep):
    """X: p columns of n rows, one per row of the array."""
    p, n = X.shape
    W, y = X.copy(), c.copy()
    nrm = np.concatenate([np.sum(X * X, axis=1), np.full(p, np.nan)])  # twice p doubles, as the workspace
    perm = np.full(p, -1, np.int32)
    assert lib.factor(n, p, grid, late, stage, keep, _p(W), _p(y), _p(nrm), _p(perm)) == 0
    return W, y, perm


@pytest.mark.parametrize("stage,keep", [(1, 1), (1, 0), (0, 0)])
@pytest.mark.parametrize("orthogonal", [False, True])
@pytest.mark.parametrize("n,p,grid", [(40, 7, 3), (23, 9, 10), (6, 9, 4), (64, 24, 5)])
def test_a_late_cta_changes_nothing(lib, n, p, grid, orthogonal, stage, keep):
    """Columns of like norms that share much of their span, and orthonormal ones: there the norms
    of a step and of the next are equal but for their rounding, either way round."""
    rng = np.random.default_rng(n + p)
    X = rng.standard_normal((p, 3)) @ rng.standard_normal((3, n)) + 0.3 * rng.standard_normal((p, n))
    if orthogonal:
        X = np.linalg.qr(rng.standard_normal((max(n, p), min(n, p))))[0].T
        X = np.ascontiguousarray(X if p <= n else X.T)
    X /= np.linalg.norm(X, axis=1)[:, None]
    if not orthogonal:
        X *= 1.0 + 0.01 * rng.random((p, 1))
    c = rng.standard_normal(n)
    want = _factor(lib, X, c, grid, -1, stage, keep)
    r = min(n, p)
    order = want[2]
    assert sorted(order) == list(range(p))
    R = np.triu(np.array([want[0][l] for l in order]).T[:r])
    d = np.linalg.solve(R[:, :r], want[1][:r])
    best = np.linalg.lstsq(X[order[:r]].T, c, rcond=None)[0]
    assert np.max(np.abs(d - best)) < 1e-9 * np.max(np.abs(best))
    for late in range(grid):
        for a, b in zip(_factor(lib, X, c, grid, late, stage, keep), want):
            assert np.array_equal(a, b), late
