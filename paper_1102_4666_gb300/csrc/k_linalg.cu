// k_linalg.cu -- the least-squares refit of Algorithm 2 (eq. alpha) through
// the normal equations A alpha = sum_i y_i B(t_i, x_i) (eq. alphasys,
// Section 3.2.2), in the correction form alpha^{k+1} = alpha^k + delta with
// A delta = B^T c^k (the fit of u^k + c^k equals alpha^k plus the fit of c^k
// because u^k lies in the span of the basis).  The paper solves with LAPACK
// dgelsy; here the Gram matrix is factored by an FP64 Cholesky on the GPU,
// with an optional FP64 iterative refinement of the normal equations.
// Also: the per-point reduction of eq. chat, the coefficient update and the
// price / delta read-out of Section 5.3.
#include <atomic>

#include <cooperative_groups.h>

#include "common.cuh"

namespace cg = cooperative_groups;

namespace {

// eq. chat: c_i = (1/M) sum of the per-chunk sums, in chunk order
__global__ void k_reduce_c(int i0, int count, int chunks, int M, const double* partial,
                           double* c) {
  pdl_begin();
  const int i = i0 + blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= i0 + count) return;
  double s = 0.0;
  for (int q = 0; q < chunks; ++q) s += partial[(size_t)i * chunks + q];
  c[i] = s / (double)M;
}

// CTA of 256 threads per basis function: out[l] = sum_i B[l][i] y[i], each
// thread over i = tid mod 256, then a fixed shuffle tree and the eight warp
// sums in order; with sub != nullptr, out[l] = sub[l] - that sum.  Bound by the
// latency of its loads at small p (35 CTAs of 128 threads with few loads in
// flight: 5.5 us at n = 2000, this 3.5 us).
__global__ void __launch_bounds__(256) k_bt_times(int n, int n_pad, int p,
                                                  const double* B,
                                                  const double* y,
                                                  const double* sub,
                                                  double* out) {
  pdl_begin();
  __shared__ double ws[8];
  const int l = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const double* row = B + (size_t)l * n_pad;
  double s = 0.0;
#pragma unroll 4
  for (int i = tid; i < n; i += 256) s += row[i] * y[i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) ws[warp] = s;
  __syncthreads();
  if (tid == 0) {
    const double tot = ((ws[0] + ws[1]) + (ws[2] + ws[3])) + ((ws[4] + ws[5]) + (ws[6] + ws[7]));
    out[l] = sub ? (sub[l] - tot) : tot;
  }
}

// v[i] = sum_l B[l][i] x[l]: CTA of 32 points x 8 slices of the basis
// functions (coalesced rows of B per warp), the slice sums added in order
__global__ void __launch_bounds__(256) k_b_times(int n, int n_pad, int p,
                                                 const double* B,
                                                 const double* x,
                                                 double* v) {
  pdl_begin();
  __shared__ double part[8][33];
  const int lane = threadIdx.x & 31, slice = threadIdx.x >> 5;
  const int i = blockIdx.x * 32 + lane;
  const int per = (p + 7) / 8;
  const int l0 = slice * per, l1 = min(p, l0 + per);
  double s = 0.0;
  if (i < n)
    for (int l = l0; l < l1; ++l) s += B[(size_t)l * n_pad + i] * x[l];
  part[slice][lane] = s;
  __syncthreads();
  if (slice == 0 && i < n) {
    double tot = 0.0;
#pragma unroll
    for (int q = 0; q < 8; ++q) tot += part[q][lane];
    v[i] = tot;
  }
}

// Tiles of 16 x 16 outputs, one per thread, for every FP64 contraction here: on
// the two-lane FP64 pipe a tile's 32-deep slice is 2 us of an SM, so that a
// 32 x 32 tile per CTA left most SMs idle behind the last ones (FP64 Gram at
// n = 1000, p = 364: 78 tiles, 310 us; 276 tiles, 135 us).
constexpr int T16 = 16;

// decode lower tile (tj <= ti) number t, row-major
__device__ __forceinline__ void lower_tile(int t, int& ti, int& tj) {
  ti = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
  while (ti * (ti + 1) / 2 > t) --ti;
  while ((ti + 1) * (ti + 2) / 2 <= t) ++ti;
  tj = t - ti * (ti + 1) / 2;
}

// FP64 Gram A = B B^T on CUDA cores: one lower tile per CTA, written to both
// triangles.
__global__ void __launch_bounds__(256) k_gram_f64(int n, int n_pad, int p,
                                                  const double* B,
                                                  double* A) {
  pdl_begin();
  __shared__ double Rs[T16][33], Cs[T16][33];
  int ti, tj;
  lower_tile(blockIdx.x, ti, tj);
  const int r0 = ti * T16, c0 = tj * T16;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int lk = threadIdx.x & 31, lr = threadIdx.x >> 5;  // loads: rows lr and lr + 8
  double acc = 0.0;
  for (int k0 = 0; k0 < n; k0 += 32) {
    const int kg = k0 + lk;
#pragma unroll
    for (int h = 0; h < T16; h += 8) {
      const int rr = lr + h;
      Rs[rr][lk] = (r0 + rr < p && kg < n) ? B[(size_t)(r0 + rr) * n_pad + kg] : 0.0;
      Cs[rr][lk] = (c0 + rr < p && kg < n) ? B[(size_t)(c0 + rr) * n_pad + kg] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < 32; ++kk) acc += Rs[ty][kk] * Cs[tx][kk];
    __syncthreads();
  }
  const int r = r0 + ty, c = c0 + tx;
  if (r < p && c < p) {
    A[(size_t)r * p + c] = acc;
    A[(size_t)c * p + r] = acc;
  }
}

// The factorisation kernels work on a batch of Gram matrices, one per
// blockIdx.y: matrix z is A + z p^2, with its original diagonal at
// diag0 + z p, its reciprocal factor diagonal at dinv + z p and its inverse
// at Ainv + z p^2.

// original diagonal of A, for the relative pivot test of the factorisation
__global__ void k_save_diag(const double* A, int p, double* diag0) {
  pdl_begin();
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  const size_t z = blockIdx.y;
  if (j < p) diag0[z * p + j] = A[z * p * p + (size_t)j * p + j];
}

// Right-looking blocked Cholesky, panel width 32, lower factor in place; the
// upper triangle of A, no longer needed, takes the transposed inverse of the
// factor (its diagonal is dinv).
// Panel step 1: the 32x32 diagonal block, factored and inverted together.  Four
// warps, one per scheduler and FP64 pipe, own every fourth column in registers,
// lanes are rows.  The elimination of column c takes l_c l_q from the columns
// q > c still to be factored; a column q <= c has become column q of the inverse
// (rows unscaled), E_r -= l_rc / l_cc E_c: eight columns per warp either way.
// Every warp computes the pivot's reciprocal root for itself, so that a column
// costs one barrier.  Bound by the chain pivot - root - column - next pivot and
// the eight FMAs between (64 cycles of the pipe each): about 1800 cycles a
// column.  Per block: one warp on shared memory 65 us, this 28 us.
// A pivot below 1e-13 of its original diagonal entry (or not finite) marks the
// matrix as numerically singular: ST_NOT_PD, and the pivot becomes NaN.
__global__ void __launch_bounds__(128) k_chol_diag(double* A, int p, int j0,
                                                   int* status,
                                                   const double* diag0,
                                                   double* dinv) {
  pdl_begin();
  __shared__ double col[2][32], Ls[32][33], Ei[32][33], di[32];
  const size_t z = blockIdx.y;
  A += z * p * p;
  diag0 += z * p;
  dinv += z * p;
  const int nb = min(32, p - j0);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // rows and columns past nb: the identity, which the elimination leaves alone
  for (int q = threadIdx.x; q < 32 * 32; q += 128) {
    const int r = q >> 5, c = q & 31;
    Ls[r][c] = (r < nb && c <= r) ? A[(size_t)(j0 + r) * p + (j0 + c)] : r == c ? 1.0 : 0.0;
  }
  const long long thr = lane < nb ? __double_as_longlong(1e-13 * diag0[j0 + lane]) : 0;
  __syncthreads();
  double R[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) R[k] = Ls[lane][warp + 4 * k];
  if (warp == 0) col[0][lane] = R[0];
  __syncthreads();
#pragma unroll
  for (int c = 0; c < 32; ++c) {
    if (c >= nb) break;  // a short last block
    const double colv = col[c & 1][lane], piv = col[c & 1][c];
    // piv > thr and finite, on the bits (no FP64 comparison); thr >= 0
    const long long pb = __double_as_longlong(piv), tb = __shfl_sync(0xffffffffu, thr, c);
    const bool ok = pb > tb && pb < 0x7ff0000000000000ll;
    const double inv = ok ? rsqrt(piv) : nan("");
    const double l = lane > c ? colv * inv : 0.0;
    // the next column first: its owner hands it on
    if (c < 31) {
      const int k = (c + 1) / 4, w = (c + 1) % 4;
      const double ls = __shfl_sync(0xffffffffu, l, c + 1);
      if (warp == w) {
        R[k] -= l * ls;
        col[(c + 1) & 1][lane] = R[k];
      }
    }
    if (warp == c % 4) {
      Ls[lane][c] = lane == c ? piv * inv : l;
      R[c / 4] = lane == c ? 1.0 : 0.0;
      if (lane == c) di[c] = inv;
      if (lane == 0 && !ok) atomicOr(status, ST_NOT_PD);
    }
    __syncthreads();
    const double l2 = l * inv;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int q = warp + 4 * k;
      if (4 * k > c + 1 || (4 * k + 3 > c + 1 && q > c + 1)) {  // still to be factored
        R[k] -= l * __shfl_sync(0xffffffffu, l, q);
      } else if (q <= c) {
        R[k] -= l2 * __shfl_sync(0xffffffffu, R[k], c);  // zero on the rows up to c, as l2 is
      }
    }
  }
#pragma unroll
  for (int k = 0; k < 8; ++k) Ei[lane][warp + 4 * k] = R[k];
  __syncthreads();
  for (int q = threadIdx.x; q < 32 * 32; q += 128) {
    const int r = q >> 5, c = q & 31;
    if (r < nb && c <= r) A[(size_t)(j0 + r) * p + (j0 + c)] = Ls[r][c];
    if (c < nb && r < c) A[(size_t)(j0 + r) * p + (j0 + c)] = Ei[c][r] * di[c];  // inverse, transposed
  }
  if (threadIdx.x < nb) dinv[j0 + threadIdx.x] = di[threadIdx.x];
}

// the inverse of diagonal block j0 (rows c, columns k <= c) from the upper triangle
__device__ __forceinline__ double diag_inv(const double* __restrict__ A, const double* __restrict__ dinv,
                                           int p, int j0, int c, int k) {
  if (j0 + c >= p || k > c) return 0.0;
  return k == c ? dinv[j0 + c] : A[(size_t)(j0 + k) * p + j0 + c];
}

// Panel step 2: the rows below, L21 = A21 L11^-T: eight rows per CTA, an
// output per thread (a substitution per row left a warp to 496 dependent steps
// on its own: 24 us a panel, this 5 us)
__global__ void __launch_bounds__(256) k_chol_trsm(double* A, int p, int j0,
                                                   const double* dinv) {
  pdl_begin();
  __shared__ double Li[32][33], a[8][33];
  const size_t z = blockIdx.y;
  A += z * p * p;
  dinv += z * p;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int q = warp; q < 32; q += 8) Li[lane][q] = diag_inv(A, dinv, p, j0, lane, q);
  const int row = j0 + 32 + 8 * blockIdx.x + warp;  // a full panel: rows below exist only then
  a[warp][lane] = row < p ? A[(size_t)row * p + j0 + lane] : 0.0;
  __syncthreads();
  double acc = 0.0;
#pragma unroll
  for (int k = 0; k < 32; ++k) acc += a[warp][k] * Li[lane][k];
  if (row < p) A[(size_t)row * p + j0 + lane] = acc;
}

// trailing update A22 -= L21 L21^T on the lower triangle
__global__ void __launch_bounds__(256) k_chol_update(double* A, int p, int j0) {
  pdl_begin();
  __shared__ double Lr[T16][33], Lc[T16][33];
  A += (size_t)blockIdx.y * p * p;
  int ti, tj;
  lower_tile(blockIdx.x, ti, tj);
  const int r0 = j0 + 32 + T16 * ti, c0 = j0 + 32 + T16 * tj;
  const int lk = threadIdx.x & 31, lr = threadIdx.x >> 5;
#pragma unroll
  for (int h = 0; h < T16; h += 8) {
    const int rr = lr + h;
    Lr[rr][lk] = r0 + rr < p ? A[(size_t)(r0 + rr) * p + j0 + lk] : 0.0;
    Lc[rr][lk] = c0 + rr < p ? A[(size_t)(c0 + rr) * p + j0 + lk] : 0.0;
  }
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int r = r0 + ty, c = c0 + tx;
  const bool in = r < p && c <= r;
  const double old = in ? A[(size_t)r * p + c] : 0.0;
  __syncthreads();
  double s = 0.0;
#pragma unroll
  for (int kk = 0; kk < 32; ++kk) s += Lr[ty][kk] * Lc[tx][kk];
  if (in) A[(size_t)r * p + c] = old - s;
}

// M = L^-1 by block columns, transposed into the upper triangle of A: CTA
// (z, strip) computes C columns of M from their diagonal block down,
//   M_I = -L_II^-1 sum_{K < I} L_IK M_K,
// keeping the strip in shared memory; warp = column, lane = row.  The strips of
// the first columns are the longest and start first, those of every matrix
// before the next shorter ones (matrix by matrix the long strips of the last one
// ended the launch: ten of p = 924 3.3 -> 2.5 ms; p^3 / 6 is 2.1).  p^3 / 6 multiply-adds, with k_inv_syrk
// p^3 / 3 instead of the 2 p^3 / 3 of p substitutions.
template <int C>
__global__ void __launch_bounds__(32 * C) k_tri_inv(double* A, int p,
                                                    const double* dinv) {
  pdl_begin();
  extern __shared__ double Ms[];  // [row][C], rows padded to blocks of 32
  __shared__ double Lt[32][33], Ac[32][C + 1];
  constexpr int PER = 32 / C;  // tile elements per thread
  const size_t z = blockIdx.x;
  A += z * p * p;
  dinv += z * p;
  const int c0 = blockIdx.y * C, J = c0 >> 5, T = (p + 31) >> 5;
  const int lane = threadIdx.x & 31, col = threadIdx.x >> 5;
  const int cg = c0 + col;
  // element e of the tile (I, K): row (threadIdx.x >> 5) + e C, column lane
  auto fetch = [&](int I, int K, double (&t)[PER]) {
#pragma unroll
    for (int e = 0; e < PER; ++e) {
      const int r = I * 32 + col + e * C;
      t[e] = r < p ? A[(size_t)r * p + K * 32 + lane] : 0.0;
    }
  };
  Ms[(J * 32 + lane) * C + col] =
      cg < p ? diag_inv(A, dinv, p, J * 32, lane, cg - J * 32) : 0.0;
  double nx[PER];
  if (J + 1 < T) fetch(J + 1, J, nx);
  for (int I = J + 1; I < T; ++I) {
    double acc = 0.0;
    for (int K = J; K < I; ++K) {
      __syncthreads();
#pragma unroll
      for (int e = 0; e < PER; ++e) Lt[col + e * C][lane] = nx[e];
      __syncthreads();
      if (K + 1 < I)
        fetch(I, K + 1, nx);
      else
#pragma unroll
        for (int e = 0; e < PER; ++e) nx[e] = diag_inv(A, dinv, p, I * 32, col + e * C, lane);
      const double* m = Ms + (size_t)K * 32 * C + col;
#pragma unroll
      for (int k = 0; k < 32; ++k) acc += Lt[lane][k] * m[k * C];
    }
    __syncthreads();
#pragma unroll
    for (int e = 0; e < PER; ++e) Lt[col + e * C][lane] = nx[e];
    Ac[lane][col] = acc;
    __syncthreads();
    if (I + 1 < T) fetch(I + 1, J, nx);
    double v = 0.0;
#pragma unroll
    for (int k = 0; k < 32; ++k) v -= Lt[lane][k] * Ac[k][col];
    Ms[(I * 32 + lane) * C + col] = v;
    if (cg < p && I * 32 + lane < p) A[(size_t)cg * p + I * 32 + lane] = v;
  }
}

// A^-1 = M^T M: Ainv[a][b] = sum_{i >= max(a, b)} M_ia M_ib, the columns of M
// being the rows of the upper triangle; lower tiles, written to both triangles
__global__ void __launch_bounds__(256) k_inv_syrk(const double* A, int p,
                                                  const double* dinv,
                                                  double* Ainv) {
  pdl_begin();
  __shared__ double Rs[T16][33], Cs[T16][33];
  const size_t z = blockIdx.y;
  A += z * p * p;
  dinv += z * p;
  Ainv += z * p * p;
  int ti, tj;
  lower_tile(blockIdx.x, ti, tj);  // the longest sums first
  const int r0 = ti * T16, c0 = tj * T16;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int lk = threadIdx.x & 31, lr = threadIdx.x >> 5;
  auto m = [&](int a, int i) {
    if (a >= p || i >= p || i < a) return 0.0;
    return i == a ? dinv[a] : A[(size_t)a * p + i];
  };
  double acc = 0.0;
  for (int i0 = r0 & ~31; i0 < p; i0 += 32) {
#pragma unroll
    for (int h = 0; h < T16; h += 8) {
      Rs[lr + h][lk] = m(r0 + lr + h, i0 + lk);
      Cs[lr + h][lk] = m(c0 + lr + h, i0 + lk);
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < 32; ++kk) acc += Rs[ty][kk] * Cs[tx][kk];
    __syncthreads();
  }
  const int r = r0 + ty, c = c0 + tx;
  if (r < p && c < p) {
    Ainv[(size_t)r * p + c] = acc;
    Ainv[(size_t)c * p + r] = acc;
  }
}

struct EvalArgs {
  int d, p, eta;
  double ctr[BSDE_DMAX + 1], sc[BSDE_DMAX + 1];
};

// T_e and T_e' (e = 1 .. eta) at z, into t[(e - 1) stride] and dt[(e - 1) stride]
__device__ __forceinline__ void cheb_column(double z, int eta, double* t, double* dt, int stride) {
  double t0 = 1.0, t1 = z, d0 = 0.0, d1 = 1.0;
  for (int e = 1; e <= eta; ++e) {
    if (e >= 2) {
      const double t2 = 2.0 * z * t1 - t0, d2 = 2.0 * t1 + 2.0 * z * d1 - d0;
      t0 = t1; t1 = t2; d0 = d1; d1 = d2;
    }
    t[(e - 1) * stride] = t1;
    dt[(e - 1) * stride] = d1;
  }
}

__device__ __forceinline__ void unpack_pair(uint2 pr, int a, int& v, int& e) {
  const uint32_t byte = ((a < 4 ? pr.x >> (8 * a) : pr.y >> (8 * (a - 4)))) & 0xffu;
  v = (int)(byte >> 4);
  e = (int)(byte & 15u);
}

// u and du/dx_v of one basis function from tables T, T' laid out [v][e - 1]
// with the given stride: val = prod T, and grad(v, dval) for every active
// space variate (dval not yet scaled by d xi / dx)
template <typename G>
__device__ __forceinline__ double basis_value(uint2 pr, int nz, int eta, const double* t,
                                              const double* dt, int stride, G&& grad) {
  double tv[BSDE_NNZ_MAX];
  double val = 1.0;
#pragma unroll
  for (int a = 0; a < BSDE_NNZ_MAX; ++a) {
    if (a >= nz) break;
    int v, e;
    unpack_pair(pr, a, v, e);
    tv[a] = t[(v * eta + e - 1) * stride];
    val *= tv[a];
  }
#pragma unroll
  for (int a = 0; a < BSDE_NNZ_MAX; ++a) {
    if (a >= nz) break;
    int v, e;
    unpack_pair(pr, a, v, e);
    if (v == 0) continue;
    double gd = dt[(v * eta + e - 1) * stride];
#pragma unroll
    for (int c = 0; c < BSDE_NNZ_MAX; ++c)
      if (c < nz && c != a) gd *= tv[c];
    grad(v, gd);
  }
  return val;
}

// u and its space derivatives at one point by a CTA of 256 threads, lanes =
// basis functions: the Chebyshev values of the point once in shared memory (the
// last warp; coord(v): its coordinate v), coef(l) gives the coefficients, the
// sums over the threads are taken by one warp per row.  row(0, u) and row(j,
// du/dx_j) are called by one lane each.
constexpr int EVAL_ROWS = BSDE_DMAX + 1;
struct EvalShared {
  double T[EVAL_ROWS * 15], dT[EVAL_ROWS * 15];
  double red[EVAL_ROWS][256];
};
__device__ __forceinline__ double row_sum(const double* q) {  // 256 values, one warp
  q += threadIdx.x & 31;
  double s = ((q[0] + q[32]) + (q[64] + q[96])) + ((q[128] + q[160]) + (q[192] + q[224]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}
template <typename Coord, typename Coef, typename Row>
__device__ __forceinline__ void eval_point(const EvalArgs& ea, const uint2* pairs, const uint8_t* nnz,
                                           EvalShared& sh, Coord&& coord, Coef&& coef, Row&& row) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, d = ea.d;
  if (warp == 7 && lane <= d)
    cheb_column((coord(lane) - ea.ctr[lane]) * ea.sc[lane], ea.eta, sh.T + lane * ea.eta,
                sh.dT + lane * ea.eta, 1);
  for (int j = 1; j <= d; ++j) sh.red[j][tid] = 0.0;
  __syncthreads();
  double u = 0.0;
  for (int l = tid; l < ea.p; l += 256) {
    const double al = coef(l);
    u += al * basis_value(pairs[l], nnz[l], ea.eta, sh.T, sh.dT, 1,
                          [&](int v, double gd) { sh.red[v][tid] += al * gd; });
  }
  sh.red[0][tid] = u;
  __syncthreads();
  for (int r = warp; r <= d; r += 8) {
    const double s = row_sum(sh.red[r]);
    if (lane == 0) row(r, r == 0 ? s : s * ea.sc[r]);
  }
}

// alpha += delta; ||delta||_2, ||delta||_inf into the report block; FP32 copy;
// then the read-out of Section 5.3 at (0, log S0): price V = u and du/dx.  One
// CTA, one launch.
__global__ void __launch_bounds__(256) k_update(const __grid_constant__ EvalArgs ea, int k, double t0,
                                                double* alpha, float* alpha32, const double* delta,
                                                const uint2* pairs, const uint8_t* nnz,
                                                const double* logS0, double* out) {
  pdl_begin();
  __shared__ EvalShared sh;
  __shared__ double w2[8], wi[8];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool it = k >= 0 && k < 64;
  double a2 = 0.0, ai = 0.0;
  eval_point(
      ea, pairs, nnz, sh, [&](int v) { return v == 0 ? t0 : logS0[v - 1]; },
      [&](int l) {
        const double dl = delta[l];
        const double al = alpha[l] + dl;
        alpha[l] = al;
        if (alpha32) alpha32[l] = (float)al;
        a2 += dl * dl;
        ai = fmax(ai, fabs(dl));
        return al;
      },
      [&](int j, double s) {
        if (j > 0) {
          out[OUT_DUDX + j - 1] = s;
        } else {
          out[OUT_PRICE] = s;
          if (it) out[OUT_PRICE_IT + k] = s;
        }
      });
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a2 += __shfl_xor_sync(0xffffffffu, a2, o);
    ai = fmax(ai, __shfl_xor_sync(0xffffffffu, ai, o));
  }
  if (lane == 0) {
    w2[warp] = a2;
    wi[warp] = ai;
  }
  __syncthreads();
  if (tid == 0 && it) {
    for (int w = 1; w < 8; ++w) {
      a2 += w2[w];
      ai = fmax(ai, wi[w]);
    }
    out[OUT_RES2 + k] = sqrt(a2);
    out[OUT_RESI + k] = ai;
  }
}

// The whole refit of one iteration for a small basis by one cluster: the mean
// corrections, B^T c, A^-1, the refinement steps, alpha + delta (CTA 0, with its
// norms), the read-out (the last CTA) and the monomial coefficients for the next
// iteration's paths (the others).  CTA r keeps the points [r nl, r nl + nl) of B in
// shared memory and A^-1 beside them; of a sum over the points every CTA forms its
// part, which all of them read through distributed shared memory and add in rank
// order; the p x p products every CTA takes for itself.  The last CTA has no points:
// it tabulates the basis and its derivatives at the read-out point meanwhile.
// Bound by latency and the two-lane FP64 pipe: of 21 us at n = 2000, p = 35 the loads
// take 3, a product with B 1.4 to 2 (five of them), one with A^-1 1.1 and an exchange
// 1.5 (three of each).
// Once B is in shared memory the next kernel on the stream may start, so that the
// next iteration's points and basis are written meanwhile (launch_basis, early).
constexpr int REFIT_P = 64;
struct RefitArgs {
  int n, n_pad, p, nl, ldb, chunks, M, refine, k, pm;
  const double *B, *Ainv, *partial;
  double *c, *alpha;
  float* alpha32;
  const uint2* pairs;
  const uint8_t* nnz;
  const double* logS0;
  double* out;
  const int *conv_row, *conv_l;
  const double* conv_c;
  double* beta;
  float* beta32;
};

__device__ __forceinline__ void copy8_async(double* dst, const double* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

__global__ void __launch_bounds__(256) k_refit(const __grid_constant__ EvalArgs ea,
                                               const __grid_constant__ RefitArgs a) {
  pdl_wait();
  extern __shared__ double rf[];
  __shared__ double part[2][REFIT_P], vec[REFIT_P], prod[REFIT_P], delta[REFIT_P], al[REFIT_P];
  __shared__ double T[EVAL_ROWS * 15], dT[EVAL_ROWS * 15], at[EVAL_ROWS][REFIT_P + 1];
  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, p = a.p;
  const int rank = (int)cluster.block_rank(), ranks = (int)cluster.num_blocks();
  const int i0 = rank * a.nl, cnt = max(0, min(a.nl, a.n - i0));
  double* As = rf;                      // [c][l], symmetric
  double* Bs = As + p * p;              // [l][i], rows of odd length
  double* ys = Bs + (size_t)p * a.ldb;  // at this CTA's points: c, then B delta
  double* red = ys + a.nl;              // 256
  double first[4];  // the loads that the sums wait for go first
#pragma unroll
  for (int q = 0; q < 4; ++q)
    first[q] = tid < cnt && q < a.chunks ? a.partial[(size_t)(i0 + tid) * a.chunks + q] : 0.0;
  for (int i = tid; i < p * p; i += 256) copy8_async(As + i, a.Ainv + i);
  for (int l = warp; l < p; l += 8)
    for (int i = lane; i < cnt; i += 32)
      copy8_async(Bs + (size_t)l * a.ldb + i, a.B + (size_t)l * a.n_pad + i0 + i);
  if (tid < p) al[tid] = a.alpha[tid];
  for (int i = tid; i < cnt; i += 256) {
    double c;
    if (a.chunks > 0) {
      double s = 0.0;
      for (int q = 0; q < a.chunks; ++q)
        s += i == tid && q < 4 ? (q == 0 ? first[0] : q == 1 ? first[1] : q == 2 ? first[2] : first[3])
                               : a.partial[(size_t)(i0 + i) * a.chunks + q];
      c = s / (double)a.M;
      a.c[i0 + i] = c;
    } else {
      c = a.c[i0 + i];
    }
    ys[i] = c;
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  pdl_trigger();
  if (rank == ranks - 1) {
    // at[0][l] = B_l and at[j][l] = dB_l / dx_j at (0, log S0)
    if (warp == 7 && lane <= ea.d)
      cheb_column(((lane == 0 ? 0.0 : a.logS0[lane - 1]) - ea.ctr[lane]) * ea.sc[lane], ea.eta,
                  T + lane * ea.eta, dT + lane * ea.eta, 1);
    for (int i = tid; i < (ea.d + 1) * (REFIT_P + 1); i += 256) at[0][i] = 0.0;
    __syncthreads();
    if (tid < p)
      at[0][tid] = basis_value(a.pairs[tid], a.nnz[tid], ea.eta, T, dT, 1,
                               [&](int v, double gd) { at[v][tid] = gd * ea.sc[v]; });
  }
  // dst[l] = sum_{i < len} m[l sl + i si] x[i], thread = (l, i mod parts): rows of
  // odd length or columns, so without bank conflicts
  const int parts = min(8, 256 / p), q = tid / p, l = tid - q * p;
  auto product = [&](const double* m, int sl, int si, const double* x, int len, double* dst) {
    if (q < parts) {
      double s0 = 0.0, s1 = 0.0;
      int i = q;
      m += l * sl;
      for (; i + parts < len; i += 2 * parts) {
        s0 += m[i * si] * x[i];
        s1 += m[(i + parts) * si] * x[i + parts];
      }
      if (i < len) s0 += m[i * si] * x[i];
      red[q * p + l] = s0 + s1;
    }
    __syncthreads();
    if (tid < p) {
      double v[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = e < parts ? red[e * p + tid] : 0.0;
      dst[tid] = ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
    }
  };
  double rhs = 0.0;
  for (int r = 0;; ++r) {
    // B^T y over the cluster.  The parts' buffer alternates: a CTA may write its
    // next part while others still read this one
    product(Bs, a.ldb, 1, ys, cnt, part[r & 1]);
    cluster.sync();
    if (tid < p) {
      double v[16];
#pragma unroll
      for (int e = 0; e < 16; ++e) v[e] = e < ranks ? cluster.map_shared_rank(part[r & 1], e)[tid] : 0.0;
#pragma unroll
      for (int w = 1; w < 16; w *= 2)
#pragma unroll
        for (int e = 0; e < 16; e += 2 * w) v[e] += v[e + w];
      if (r == 0) rhs = v[0];
      vec[tid] = r == 0 ? rhs : rhs - v[0];
    }
    __syncthreads();
    if (r == a.refine) break;
    product(As, 1, p, vec, p, prod);
    if (tid < p) delta[tid] = r == 0 ? prod[tid] : delta[tid] + prod[tid];
    __syncthreads();
    // two threads a point
    for (int j0 = 0; j0 < cnt; j0 += 128) {
      const int i = j0 + (tid & 127), h = tid >> 7, half = (p + 1) / 2, l1 = h ? p : half;
      double s0 = 0.0, s1 = 0.0;
      if (i < cnt) {
        int m = h * half;
        for (; m + 1 < l1; m += 2) {
          s0 += Bs[m * a.ldb + i] * delta[m];
          s1 += Bs[(m + 1) * a.ldb + i] * delta[m + 1];
        }
        if (m < l1) s0 += Bs[m * a.ldb + i] * delta[m];
      }
      red[tid] = s0 + s1;
      __syncthreads();
      if (h == 0 && i < cnt) ys[i] = red[tid] + red[tid + 128];
      __syncthreads();
    }
  }
  auto left = cluster.barrier_arrive();  // no CTA's parts are read after this
  product(As, 1, p, vec, p, prod);
  if (tid < p) {
    const double dl = a.refine == 0 ? prod[tid] : delta[tid] + prod[tid];
    delta[tid] = dl;
    al[tid] += dl;
  }
  __syncthreads();
  if (rank == 0) {
    if (tid < p) {
      a.alpha[tid] = al[tid];
      if (a.alpha32) a.alpha32[tid] = (float)al[tid];
    }
    if (warp == 7 && a.k >= 0 && a.k < 64) {
      const double d0 = lane < p ? delta[lane] : 0.0, d1 = lane + 32 < p ? delta[lane + 32] : 0.0;
      double a2 = d0 * d0 + d1 * d1, ai = fmax(fabs(d0), fabs(d1));
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        a2 += __shfl_xor_sync(0xffffffffu, a2, o);
        ai = fmax(ai, __shfl_xor_sync(0xffffffffu, ai, o));
      }
      if (lane == 0) {
        a.out[OUT_RES2 + a.k] = sqrt(a2);
        a.out[OUT_RESI + a.k] = ai;
      }
    }
  } else if (rank == ranks - 1) {
    for (int r = warp; r <= ea.d; r += 8) {
      double s = (lane < p ? al[lane] * at[r][lane] : 0.0) + (lane + 32 < p ? al[lane + 32] * at[r][lane + 32] : 0.0);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) {
        if (r > 0) {
          a.out[OUT_DUDX + r - 1] = s;
        } else {
          a.out[OUT_PRICE] = s;
          if (a.k >= 0 && a.k < 64) a.out[OUT_PRICE_IT + a.k] = s;
        }
      }
    }
  } else {
    for (int m = (rank - 1) * 256 + tid; m < a.pm; m += (ranks - 2) * 256) {
      double s = 0.0;
      for (int e = a.conv_row[m]; e < a.conv_row[m + 1]; ++e) s += a.conv_c[e] * al[a.conv_l[e]];
      a.beta[m] = s;
      a.beta32[m] = (float)s;
    }
  }
  cluster.barrier_wait(std::move(left));
}

// u and dV/dS (delta may be null) at a few query points, one CTA each
__global__ void __launch_bounds__(256) k_eval_few(const __grid_constant__ EvalArgs ea,
                                                  const double* alpha, const uint2* pairs,
                                                  const uint8_t* nnz, const double* qt, const double* S,
                                                  double* price, double* delta) {
  __shared__ EvalShared sh;
  const size_t q = blockIdx.x;
  const double* Sq = S + q * ea.d;
  eval_point(
      ea, pairs, nnz, sh, [&](int v) { return v == 0 ? qt[q] : fx64::log_abs(Sq[v - 1]); },
      [&](int l) { return alpha[l]; },
      [&](int j, double s) {
        if (j == 0)
          price[q] = s;
        else if (delta)
          delta[q * ea.d + j - 1] = s / Sq[j - 1];
      });
}

// u and du/dx at query points, threads = queries: CTA of 32 points x slices of
// the basis functions (one warp each); every warp tabulates its share of the
// points' Chebyshev values in shared memory ([slot][point]), then takes its
// slice, the function's variates being the same for the whole warp.  S: prices;
// x = log S here, and the derivative is returned as dV/dS.  Bound by the FP64
// pipe (84 % busy in the form that treated every function on its own), so the
// functions that differ in their last variate only, neighbours in the basis
// order, share the product P of the others and one sum S of the last factors:
// three FP64 instructions per function and a few per group instead of twelve.
// The functions are taken from the last, of the highest degree, to the first: the
// constant and the linear terms, mostly the largest, come last, so that few
// additions round at their size.
// 20000 points, d = 10, p = 364: one CTA per point 840 us, function by function
// 352 us, this 112 us.
__global__ void __launch_bounds__(256) k_eval_many(const __grid_constant__ EvalArgs ea, int nq,
                                                   const double* __restrict__ alpha,
                                                   const uint2* __restrict__ pairs,
                                                   const uint8_t* __restrict__ nnz,
                                                   const double* __restrict__ qt,
                                                   const double* __restrict__ S,
                                                   double* __restrict__ price,
                                                   double* __restrict__ delta) {
  extern __shared__ double ev[];  // T, dT: (d + 1) eta x 32 each; sums: slices x (d + 1) x 32
  const int lane = threadIdx.x & 31, slice = threadIdx.x >> 5, slices = blockDim.x >> 5;
  const int d = ea.d, rows = (d + 1) * ea.eta;
  double* T = ev + lane;
  double* dT = T + (size_t)rows * 32;
  double* acc = ev + (size_t)2 * rows * 32 + (size_t)slice * (d + 1) * 32 + lane;
  const int q = blockIdx.x * 32 + lane;
  const int qc = q < nq ? q : nq - 1;
  for (int v = slice; v <= d; v += slices) {
    const double y = v == 0 ? qt[qc] : fx64::log_abs(S[(size_t)qc * d + v - 1]);
    cheb_column((y - ea.ctr[v]) * ea.sc[v], ea.eta, T + (size_t)v * ea.eta * 32,
                dT + (size_t)v * ea.eta * 32, 32);
  }
  for (int j = 0; j <= d; ++j) acc[j * 32] = 0.0;
  __syncthreads();
  const int per = (ea.p + slices - 1) / slices;
  const int l1 = min(ea.p, (slice + 1) * per);
  double u = 0.0;
  // the open group: its m shared factors, their product and the sum of the rest
  uint64_t group = ~0ull;
  int m = 0;
  double P = 1.0, sum = 0.0;
  auto close = [&]() {
    u += P * sum;
    for (int a = 0; a < m; ++a) {
      const int va = (int)(group >> (8 * a + 4)) & 15;
      if (va == 0) continue;
      double gd = sum * dT[(va * ea.eta + ((int)(group >> (8 * a)) & 15) - 1) * 32];
      for (int c = 0; c < m; ++c)
        if (c != a)
          gd *= T[(((int)(group >> (8 * c + 4)) & 15) * ea.eta + ((int)(group >> (8 * c)) & 15) - 1) * 32];
      acc[va * 32] += gd;
    }
  };
  for (int l = l1 - 1; l >= slice * per; --l) {
    const double al = alpha[l];
    const int nz = nnz[l];
    if (nz == 0) {
      u += al;
      continue;
    }
    const uint2 pr = pairs[l];
    const uint64_t w = ((uint64_t)pr.y << 32) | pr.x;
    const uint64_t head = w & ((1ull << (8 * (nz - 1))) - 1);
    if (head != group || nz - 1 != m) {
      close();
      group = head;
      m = nz - 1;
      P = 1.0;
      sum = 0.0;
      for (int a = 0; a < m; ++a) {
        const double t = T[(((int)(head >> (8 * a + 4)) & 15) * ea.eta + ((int)(head >> (8 * a)) & 15) - 1) * 32];
        P = a == 0 ? t : P * t;
      }
    }
    const int last = (int)(w >> (8 * (nz - 1))), v = (last >> 4) & 15;
    const int slot = (v * ea.eta + (last & 15) - 1) * 32;
    sum += al * T[slot];
    if (v > 0) acc[v * 32] += (al * P) * dT[slot];
  }
  close();
  acc[0] = u;
  __syncthreads();
  // sums over the slices, in pairs, the last first; row j = 0: u, else the derivative in x_j
  const double* a0 = ev + (size_t)2 * rows * 32 + lane;
  for (int j = slice; j <= d; j += slices) {
    double s = 0.0;
    for (int w = slices - 2; w >= 0; w -= 2)
      s += a0[((size_t)(w + 1) * (d + 1) + j) * 32] + a0[((size_t)w * (d + 1) + j) * 32];
    if (slices == 1) s = a0[j * 32];
    if (q >= nq) continue;
    if (j == 0)
      price[q] = s;
    else if (delta)
      delta[(size_t)q * d + j - 1] = s * ea.sc[j] / S[(size_t)q * d + j - 1];
  }
}

// monomial coefficients of u^k (basis of total degree <= 3): beta_m =
// sum over the CSR row m of coef * alpha_l, in FP64, with an FP32 copy
__global__ void k_cheb2mono(int pm, const int* row, const int* lidx,
                            const double* coef, const double* alpha,
                            double* beta, float* beta32) {
  pdl_begin();
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= pm) return;
  double s = 0.0;
  for (int e = row[m]; e < row[m + 1]; ++e) s += coef[e] * alpha[lidx[e]];
  beta[m] = s;
  beta32[m] = (float)s;
}

// x (+)= Ainv b: warp per row, fixed shuffle order
__global__ void k_inv_gemv(int p, const double* Ainv, const double* b,
                           double* x, int accumulate) {
  pdl_begin();
  const int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (row >= p) return;
  const double* a = Ainv + (size_t)row * p;
  double s = 0.0;
  for (int c = lane; c < p; c += 32) s += a[c] * b[c];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) x[row] = accumulate ? x[row] + s : s;
}

// The two halves of A^-1 b = M^T (M b), M in the upper triangle of A.  y = M b:
// CTA of 256 threads for eight entries, thread = (term mod 32, entry), so that a
// row of A is read in whole sectors and every SM has a part of the p^2 / 2
// multiply-adds (32 entries per CTA would leave one SM 7 us of them at p = 924).
__global__ void __launch_bounds__(256) k_m_times(int p, const double* A, const double* dinv,
                                                 const double* b, double* y) {
  pdl_begin();
  __shared__ double ws[8][8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int i = blockIdx.x * 8 + (threadIdx.x & 7);
  double s = 0.0;
  if (i < p) {
    const int a0 = threadIdx.x >> 3;
#pragma unroll 8
    for (int a = a0; a < i; a += 32) s += A[(size_t)a * p + i] * b[a];
    if ((i & 31) == a0) s += dinv[i] * b[i];
  }
  s += __shfl_xor_sync(0xffffffffu, s, 8);
  s += __shfl_xor_sync(0xffffffffu, s, 16);
  if (lane < 8) ws[warp][lane] = s;
  __syncthreads();
  if (threadIdx.x < 8 && i < p) {
    const int c = threadIdx.x;
    y[i] = ((ws[0][c] + ws[1][c]) + (ws[2][c] + ws[3][c])) + ((ws[4][c] + ws[5][c]) + (ws[6][c] + ws[7][c]));
  }
}

// x (+)= M^T y: warp per row, fixed shuffle order
__global__ void __launch_bounds__(256) k_mt_times(int p, const double* A, const double* dinv,
                                                  const double* y, double* x, int accumulate) {
  pdl_begin();
  const int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (row >= p) return;
  const double* a = A + (size_t)row * p;
  double s = lane == 0 ? dinv[row] * y[row] : 0.0;
#pragma unroll 8
  for (int c = row + 1 + lane; c < p; c += 32) s += a[c] * y[c];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) x[row] = accumulate ? x[row] + s : s;
}

}  // namespace

// one small matrix is a chain of latencies, and early launches help it (a whole FP64
// iteration at p = 364 2.78 -> 2.70 ms); a batch fills the SMs (see launch_kernel)
static bool factor_early(const ProblemDev& P, int nb) { return nb == 1 && P.p <= 512; }

template <int C>
static void launch_tri_inv(const ProblemDev& P, int nb, cudaStream_t st) {
  const size_t smem = (size_t)((P.p + 31) / 32 * 32) * C * sizeof(double);
  constexpr int fixed = (32 * 33 + 32 * (C + 1)) * (int)sizeof(double);  // its static part
  if (smem > 32 * 1024) smem_limit<SMEM_PER_CTA - fixed>(k_tri_inv<C>);
  launch_kernel(factor_early(P, nb), k_tri_inv<C>, dim3(nb, (P.p + C - 1) / C), 32 * C, smem, st, P.A, P.p, P.dinv);
}

// strips of 8 columns when there are enough of them for two CTAs per SM (they
// read the factor half as often as strips of 4) and their p x 8 values fit the
// shared memory, else of 4, or 1 for the largest bases
void launch_inverse(const ProblemDev& P, int nb, bool full, cudaStream_t st) {
  const size_t col = (size_t)((P.p + 31) / 32 * 32) * sizeof(double), room = 208 * 1024;
  if ((long long)((P.p + 7) / 8) * nb >= 2LL * device_sm_count() && 8 * col <= room)
    launch_tri_inv<8>(P, nb, st);
  else if (4 * col <= room)
    launch_tri_inv<4>(P, nb, st);
  else
    launch_tri_inv<1>(P, nb, st);
  if (!full) return;
  const int T = (P.p + T16 - 1) / T16;
  launch_kernel(factor_early(P, nb), k_inv_syrk, dim3(T * (T + 1) / 2, nb), 256, 0, st, P.A, P.p, P.dinv, P.Ainv);
}

void launch_inv_gemv(const ProblemDev& P, const double* b, double* x, int accumulate,
                     cudaStream_t st) {
  launch_pdl(k_inv_gemv, (P.p * 32 + 255) / 256, 256, 0, st, P.p, P.Ainv, b, x, accumulate);
}

void launch_factor_solve(const ProblemDev& P, const double* b, double* x, int accumulate,
                         cudaStream_t st) {
  launch_pdl(k_m_times, (P.p + 7) / 8, 256, 0, st, P.p, P.A, P.dinv, b, P.v);
  launch_pdl(k_mt_times, (P.p + 7) / 8, 256, 0, st, P.p, P.A, P.dinv, P.v, x, accumulate);
}

void launch_cheb2mono(const ProblemDev& P, cudaStream_t st) {
  launch_pdl(k_cheb2mono, (P.pm + 127) / 128, 128, 0, st, P.pm, P.conv_row, P.conv_l, P.conv_c, P.alpha,
                                                   P.beta, P.beta32);
}

void launch_reduce_c(const ProblemDev& P, int M, cudaStream_t st) {
  const int count = P.shard_n > 0 ? P.shard_n : P.n;
  if (count <= 0) return;
  launch_pdl(k_reduce_c, (count + 255) / 256, 256, 0, st, P.shard_i0, count, P.chunks, M, P.partial, P.c);
}

void launch_gram_f64(const ProblemDev& P, cudaStream_t st) {
  const int T = (P.p + T16 - 1) / T16;
  launch_kernel(false, k_gram_f64, T * (T + 1) / 2, 256, 0, st, P.n, P.n_pad, P.p, P.B, P.A);
}

void launch_rhs(const ProblemDev& P, cudaStream_t st) {
  launch_pdl(k_bt_times, P.p, 256, 0, st, P.n, P.n_pad, P.p, P.B, P.c, nullptr, P.rhs);
}

void launch_cholesky(const ProblemDev& P, int nb, cudaStream_t st) {
  launch_kernel(factor_early(P, nb), k_save_diag, dim3((P.p + 255) / 256, nb), 256, 0, st, P.A, P.p, P.diag0);
  for (int j0 = 0; j0 < P.p; j0 += 32) {
    launch_kernel(factor_early(P, nb), k_chol_diag, dim3(1, nb), 128, 0, st, P.A, P.p, j0, P.status, P.diag0, P.dinv);
    const int m = P.p - j0 - 32;
    if (m > 0) {
      launch_kernel(factor_early(P, nb), k_chol_trsm, dim3((m + 7) / 8, nb), 256, 0, st, P.A, P.p, j0, P.dinv);
      const int T = (m + T16 - 1) / T16;
      launch_kernel(factor_early(P, nb), k_chol_update, dim3(T * (T + 1) / 2, nb), 256, 0, st, P.A, P.p, j0);
    }
  }
}

void launch_refine_residual(const ProblemDev& P, cudaStream_t st) {
  launch_pdl(k_b_times, (P.n + 31) / 32, 256, 0, st, P.n, P.n_pad, P.p, P.B, P.delta, P.v);
  launch_pdl(k_bt_times, P.p, 256, 0, st, P.n, P.n_pad, P.p, P.B, P.v, P.rhs, P.res);
}

static EvalArgs eval_args(const ModelHost& m, const GridHost& g, const ProblemDev& P) {
  EvalArgs ea;
  memset(&ea, 0, sizeof(ea));
  ea.d = m.d;
  ea.p = P.p;
  ea.eta = P.eta < 1 ? 1 : P.eta;
  for (int v = 0; v <= m.d; ++v) {
    ea.ctr[v] = 0.5 * (g.lo[v] + g.hi[v]);
    ea.sc[v] = 2.0 / (g.hi[v] - g.lo[v]);
  }
  return ea;
}

// alpha^{k+1} and the price and du/dx at (0, log S0) after iteration k; log S0
// lives in the tail of the report block
void launch_update(const ModelHost& m, const GridHost& g, const ProblemDev& P, int k, cudaStream_t st) {
  launch_pdl(k_update, 1, 256, 0, st, eval_args(m, g, P), k, 0.0, P.alpha, P.alpha32, P.delta, P.pairs, P.nnz,
                              P.out + OUT_SIZE + 1 + BSDE_DMAX, P.out);
}

// Whether the refit is k_refit's: a small basis whose B fits the cluster's shared
// memory and is not more than its 16 SMs are worth.  An iteration with hardly any
// paths as eleven launches and so: n = 200, p = 15 32.7 and 21.1 us, n = 2000, p = 35
// 49.4 and 39.5, n = 2600, p = 56 (the line) 60.5 and 55.0, n = 20000, p = 6 92.7 and
// 89.1, n = 37000, p = 3 141 and 145 (the means of that many points).  Beside other
// work the cluster waits a little for its SMs: small requests one at a time next to a
// d = 10 solve in the server, median and 90th percentile: 7.4 and 10.4 ms so, 7.2 and
// 9.5 as a chain, 6.9 and 11.5 with eight CTAs; alone on the device 1.7, 2.0 and 1.7 ms.
constexpr long long REFIT_NP = 150000;
constexpr int REFIT_SMEM = 203 * 1024;  // of p^2 + (p + 1) nl + ... at eight CTAs
bool refit_small(int n, int p) { return p <= REFIT_P && n <= 16384 && (long long)n * (p + 1) <= REFIT_NP; }

static cudaLaunchConfig_t refit_config(int n, int p, int ranks, cudaLaunchAttribute* at, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = ranks;
  at->val.clusterDim.y = at->val.clusterDim.z = 1;
  const int nl = (n + ranks - 2) / (ranks - 1);  // the last CTA has no points
  cfg.gridDim = ranks;
  cfg.blockDim = 256;
  cfg.dynamicSmemBytes = ((size_t)p * p + (size_t)p * (nl | 1) + nl + 256) * sizeof(double);
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cfg;
}

// CTAs of the cluster: sixteen where the device can hold one of the largest
// admitted size, else the portable eight (asked for once per device)
static int refit_ranks() {
  static std::atomic<int> known[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 8;
  int r = known[dev].load(std::memory_order_relaxed);
  if (r == 0) {
    cudaLaunchAttribute at;
    const cudaLaunchConfig_t cfg = refit_config((int)(REFIT_NP / (REFIT_P + 1)), REFIT_P, 16, &at, nullptr);
    int held = 0;
    r = 8;
    if (cudaFuncSetAttribute(k_refit, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
        smem_limit<REFIT_SMEM>(k_refit) == cudaSuccess &&
        cudaOccupancyMaxActiveClusters(&held, k_refit, &cfg) == cudaSuccess && held > 0)
      r = 16;
    else
      cudaGetLastError();
    known[dev].store(r, std::memory_order_relaxed);
  }
  return r;
}

// c: reduced here from P.partial when reduce is set, else given
cudaError_t launch_refit(const ModelHost& m, const GridHost& g, const ProblemDev& P, int M, bool reduce,
                         int refine, int k, cudaStream_t st) {
  RefitArgs a;
  memset(&a, 0, sizeof(a));
  a.n = P.n; a.n_pad = P.n_pad; a.p = P.p;
  a.chunks = reduce ? P.chunks : 0;
  a.M = M; a.refine = refine; a.k = k;
  a.pm = P.dense ? P.pm : 0;
  a.B = P.B; a.Ainv = P.Ainv; a.partial = P.partial; a.c = P.c;
  a.alpha = P.alpha; a.alpha32 = P.alpha32; a.pairs = P.pairs; a.nnz = P.nnz;
  a.logS0 = P.out + OUT_SIZE + 1 + BSDE_DMAX;
  a.out = P.out;
  a.conv_row = P.conv_row; a.conv_l = P.conv_l; a.conv_c = P.conv_c;
  a.beta = P.beta; a.beta32 = P.beta32;
  const int ranks = refit_ranks();
  cudaLaunchAttribute at;
  const cudaLaunchConfig_t cfg = refit_config(P.n, P.p, ranks, &at, st);
  a.nl = (P.n + ranks - 2) / (ranks - 1);
  a.ldb = a.nl | 1;
  cudaError_t e = smem_limit<REFIT_SMEM>(k_refit);
  return e == cudaSuccess ? cudaLaunchKernelEx(&cfg, k_refit, eval_args(m, g, P), a) : e;
}

// price and dV/dS (delta may be null) at q points (t, S).  Up to eight points per
// SM: a CTA per point, as a warp of k_eval_many takes as long for one point as for
// 32 (the call with 600 points at d = 10, p = 1001 115 us; 620 points in the
// other form 196 us, 1500 points 212 us); more: as many slices of the basis as
// keep eight warps on every scheduler, at most eight.
cudaError_t launch_eval_points(const ModelHost& m, const GridHost& g, const ProblemDev& P, int q,
                               const double* t, const double* S, double* price, double* delta,
                               cudaStream_t st) {
  const EvalArgs ea = eval_args(m, g, P);
  if (q <= 8 * device_sm_count()) {
    k_eval_few<<<q, 256, 0, st>>>(ea, P.alpha, P.pairs, P.nnz, t, S, price, delta);
    return cudaGetLastError();
  }
  const int groups = (q + 31) / 32;
  int slices = 8;
  while (slices > 1 && (long long)groups * slices > 32LL * device_sm_count()) slices >>= 1;
  const size_t smem = ((size_t)2 * (ea.d + 1) * ea.eta + (size_t)slices * (ea.d + 1)) * 32 * sizeof(double);
  constexpr int most = (2 * EVAL_ROWS * 15 + 8 * EVAL_ROWS) * 32 * (int)sizeof(double);
  cudaError_t e = smem_limit<most>(k_eval_many);
  if (e != cudaSuccess) return e;
  k_eval_many<<<groups, 32 * slices, smem, st>>>(ea, q, P.alpha, P.pairs, P.nnz, t, S, price, delta);
  return cudaGetLastError();
}
