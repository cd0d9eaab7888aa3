// k_qr.cu -- least-squares refit of eq. alpha by Householder QR with column
// pivoting on the design matrix, in FP64: the role the paper gives to
// LAPACK's dgelsy (Section 3.2.2: the Gram matrix is often ill-conditioned,
// so the paper avoids Cholesky).  Selected by bsde_solve_params.ls_mode = 1.
//
// The design matrix X[i][l] = B_l(t_i, x_i) is stored column by column
// (B[l][i], point index fastest), which is the layout Householder needs.
// Step j: pick the remaining column of largest norm as column j, build the reflector H_j = I - tau v v^T (v_0 = 1) that zeroes it below the
// diagonal, apply H_j to the remaining columns and to the right-hand side c,
// and refresh the remaining columns' norms.  Columns whose diagonal |R_jj|
// falls below 1e-13 |R_00| are treated as dependent (rank truncation); the
// solution is the basic solution R_11 delta_1 = (Q^T c)_1, delta_2 = 0,
// scattered back through the column permutation.
#include "common.cuh"

namespace {

// copy B -> W, c -> y, squared column norms
__global__ void k_qr_init(int n, int n_pad, int p, const double* B,
                          const double* c, double* W,
                          double* y, double* nrm, int* perm,
                          uint32_t* sync) {
  pdl_begin();
  if (blockIdx.x == 0 && threadIdx.x < 2) sync[threadIdx.x] = 0u;
  const int l = blockIdx.x;  // column (p of them) or the right-hand side (l == p)
  const double* src = (l < p) ? B + (size_t)l * n_pad : c;
  double* dst = (l < p) ? W + (size_t)l * n_pad : y;
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const double v = src[i];
    dst[i] = v;
    s += v * v;
  }
  __shared__ double red[32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0 && l < p) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    nrm[l] = t;
    perm[l] = l;
  }
}

constexpr int QR_THREADS = 256;
constexpr int QR_WARPS = QR_THREADS / 32;
// polls of a grid barrier before it gives up (each takes about a microsecond;
// a step of the factorisation takes a few)
constexpr uint32_t QR_WAIT_LIMIT = 1u << 24;

// Sums of two values over the CTA, times k, in every thread.  A warp's FP64
// instruction (a comparison too) holds the two-lane FP64 pipe for 64 cycles,
// however few of its lanes matter: the threads' values are added by two warps
// on different schedulers instead of by shuffles in every warp.  k is used by
// warps 0 and 1 only.  buf: 2 x QR_THREADS values and 2 results; safe to call
// again after another __syncthreads.
__device__ __forceinline__ void qr_sum2(double& a, double& b, double k, double* buf) {
  const int tid = threadIdx.x;
  buf[tid] = a;
  buf[QR_THREADS + tid] = b;
  __syncthreads();
  if (tid < 64) {  // warp 0: the first value, warp 1: the second
    const double* q = buf + (tid >> 5) * QR_THREADS + (tid & 31);
    double t = ((q[0] + q[32]) + (q[64] + q[96])) + ((q[128] + q[160]) + (q[192] + q[224]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((tid & 31) == 0) buf[2 * QR_THREADS + (tid >> 5)] = k * t;
  }
  __syncthreads();
  a = buf[2 * QR_THREADS];
  b = buf[2 * QR_THREADS + 1];
}

// order of non-negative doubles as integers (no FP64 comparison), NaN last
__device__ __forceinline__ long long qr_key(double a) {
  const long long b = __double_as_longlong(a);
  return b > 0x7ff0000000000000ll ? -1ll : b;
}

// The whole factorisation in one cooperative launch, one CTA per SM at most.
// CTA b owns the columns b, b + CTAs, ... of W (the right-hand side is column
// p) and keeps them up to date.  Columns stay where they are; pos[] holds the
// logical order.  Step j:
//   1. every CTA finds the pivot from the norms in memory (of two sets in turn:
//      a CTA ahead of the others writes those of step j + 1 while they still
//      choose from those of step j); its norm is that of
//      the rows from j on, so beta = -sign(x_0) sqrt(norm) needs no further
//      pass, and with the reflector left unscaled, v = (x_0 - beta, x_1, ...),
//      H = I - v v^T / (beta (beta - x_0)), none but the pivot column's load;
//   2. each CTA applies H to its own columns and refreshes their norms;
//   3. one grid barrier (the next step reads norms and the pivot column).
// Bound by the FP64 pipe (three multiply-adds per element of a column, two
// lanes per SM and clock: 1 us per column of 2000 rows) and by the latencies of
// a step (barrier, pivot column from L2, two block sums).  Measured at n = 2000,
// p = 210 (two columns per CTA), the whole refit in a graph: 3.69 ms with two
// launches per column, 2.12 ms now.
// sync[0]: arrivals (zero before the launch), sync[1]: set when a wait gave up.
// STAGE: the pivot column is copied to shared memory (n doubles); KEEP: the
// CTA's own columns are kept there too (and written through to W, where the
// other CTAs read a pivot column).
template <bool STAGE, bool KEEP>
__global__ void __launch_bounds__(QR_THREADS, 1)
    k_qr_factor(int n, int n_pad, int p, int steps, double* W, double* y, double* nrm, int* perm,
                uint32_t* sync, int* status) {
  extern __shared__ double qr_smem[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int G = gridDim.x, me = blockIdx.x;
  const int mine = (p - me) / G + 1;  // columns of this CTA (p + 1 in all, me <= p)
  double* v = qr_smem;                // n (STAGE)
  double* kept = qr_smem + n;         // mine x n (KEEP)
  int* pos = reinterpret_cast<int*>(qr_smem + (STAGE ? (size_t)n : 0) +
                                    (KEEP ? (size_t)n * (p / G + 1) : 0));  // p
  uint8_t* done = reinterpret_cast<uint8_t*>(pos + p);                      // p + 1
  __shared__ double buf[2 * QR_THREADS + 2];
  __shared__ long long bv[QR_WARPS];
  __shared__ int bw[QR_WARPS], s_abort;
  for (int l = tid; l <= p; l += QR_THREADS) {
    if (l < p) pos[l] = l;
    done[l] = 0;
  }
  if (KEEP) {
    for (int q = 0; q < mine; ++q) {
      const int l = me + q * G;
      const double* col = l < p ? W + (size_t)l * n_pad : y;
      for (int i = tid; i < n; i += QR_THREADS) kept[(size_t)q * n + i] = col[i];
    }
  }
  if (tid == 0) s_abort = 0;
  __syncthreads();
  for (int j = 0; j < steps; ++j) {
    // pivot: the largest remaining norm, the first logical column on ties
    const double* norms = nrm + (j & 1) * p;
    double* next_norms = nrm + ((j & 1) ^ 1) * p;
    long long best = -1;
    int bi = p;
    for (int l = j + tid; l < p; l += QR_THREADS) {
      const long long t = qr_key(__ldcg(norms + pos[l]));
      if (t > best) {
        best = t;
        bi = l;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const long long t = __shfl_xor_sync(0xffffffffu, best, o);
      const int it = __shfl_xor_sync(0xffffffffu, bi, o);
      if (t > best || (t == best && it < bi)) {
        best = t;
        bi = it;
      }
    }
    if (lane == 0) {
      bv[warp] = best;
      bw[warp] = bi;
    }
    __syncthreads();
    for (int w = 0; w < QR_WARPS; ++w) {
      const long long t = bv[w];
      const int it = bw[w];
      if (t > best || (t == best && it < bi)) {
        best = t;
        bi = it;
      }
    }
    if (bi >= p) bi = j;  // only NaN norms left
    const int c = pos[bi];
    const double* x = W + (size_t)c * n_pad;
    const double x0 = __ldcg(x + j);
    if (STAGE) {
#pragma unroll 8
      for (int i = j + 1 + tid; i < n; i += QR_THREADS) v[i] = __ldcg(x + i);
    }
    // beta, v_0 = x_0 - beta and 1 / (beta (beta - x_0)), in the two warps that
    // use them; a column of squared norm below 2^-963 is zero and left as it is
    double beta = x0, v0 = 0.0, kap = 0.0;
    if (warp < 2 && !(best >= 0 && best < 0x03c0000000000000ll)) {  // norm >= 2^-963 or NaN
      const double nx = sqrt(best < 0 ? nan("") : __longlong_as_double(best));
      beta = x0 <= 0.0 ? nx : -nx;
      v0 = x0 - beta;
      kap = -1.0 / (beta * v0);
    }
    // H on the columns of this CTA, two at a time
    int q = 0;
    while (q < mine) {
      int ql[2], m = 0;
      for (; q < mine && m < 2; ++q) {
        const int l = me + q * G;
        if (!done[l] && l != c) ql[m++] = q;
      }
      if (m == 0) break;
      const int l0 = me + ql[0] * G, l1 = m < 2 ? l0 : me + ql[1] * G;
      double* g0 = l0 < p ? W + (size_t)l0 * n_pad : y;
      double* g1 = l1 < p ? W + (size_t)l1 * n_pad : y;
      double* c0 = KEEP ? kept + (size_t)ql[0] * n : g0;
      double* c1 = KEEP ? kept + (size_t)(m < 2 ? ql[0] : ql[1]) * n : g1;
      double s0 = tid == 0 ? v0 * c0[j] : 0.0, s1 = tid == 0 && m == 2 ? v0 * c1[j] : 0.0;
#pragma unroll 4
      for (int i = j + 1 + tid; i < n; i += QR_THREADS) {
        const double vi = STAGE ? v[i] : __ldcg(x + i);
        s0 += vi * c0[i];
        if (m == 2) s1 += vi * c1[i];
      }
      qr_sum2(s0, s1, kap, buf);
      const double f0 = s0, f1 = s1;
      double q0 = 0.0, q1 = 0.0;
#pragma unroll 4
      for (int i = j + 1 + tid; i < n; i += QR_THREADS) {
        const double vi = STAGE ? v[i] : __ldcg(x + i);
        const double n0 = c0[i] - f0 * vi;
        c0[i] = n0;
        if (KEEP) g0[i] = n0;
        q0 += n0 * n0;
        if (m == 2) {
          const double n1 = c1[i] - f1 * vi;
          c1[i] = n1;
          if (KEEP) g1[i] = n1;
          q1 += n1 * n1;
        }
      }
      if (tid < m) {  // row j
        double* cc = tid ? c1 : c0;
        const double t = cc[j] - (tid ? f1 : f0) * v0;
        cc[j] = t;
        if (KEEP) (tid ? g1 : g0)[j] = t;
      }
      __syncthreads();  // the first sums have been read
      qr_sum2(q0, q1, 1.0, buf);
      if (tid == 0 && l0 < p) next_norms[l0] = q0;
      if (tid == 0 && m == 2 && l1 < p) next_norms[l1] = q1;
      __syncthreads();
    }
    // grid barrier; every wait is bounded
    __syncthreads();
    if (tid == 0) {
      __threadfence();
      atomicAdd(sync, 1u);
      pos[bi] = pos[j];
      pos[j] = c;
      done[c] = 1;
      const uint32_t want = (uint32_t)(j + 1) * (uint32_t)G;
      volatile uint32_t* cnt = sync;
      uint32_t polls = 0;
      while (*cnt < want) {
        if (++polls > QR_WAIT_LIMIT || cnt[1] != 0) {
          atomicExch(sync + 1, 1u);
          atomicOr(status, ST_TIMEOUT);
          s_abort = 1;
          break;
        }
      }
      __threadfence();
      // R_jj, after every CTA has read x0
      if (c % G == me && !s_abort) W[(size_t)c * n_pad + j] = beta;
    }
    __syncthreads();
    if (s_abort) return;
  }
  if (me == 0)
    for (int l = tid; l < p; l += QR_THREADS) perm[l] = pos[l];
}

// basic solution: rank r from |R_jj| > 1e-13 |R_00|, R_11 d = y_1 by back
// substitution, delta[perm[j]] = d_j (0 beyond r).  One CTA; blocks of 32
// columns: warp 0 solves the block's triangle with shuffles, then every thread
// takes the block's columns off its rows, the last column first.
__global__ void __launch_bounds__(256) k_qr_solve(int n, int n_pad, int p, const double* W,
                                                  const double* y,
                                                  const int* perm,
                                                  double* delta,
                                                  double* work, int* rank_out) {
  pdl_begin();
  __shared__ int s_rank;
  __shared__ double xs[32];
  __shared__ const double* cols[32];
  __shared__ double tri[32][33];
  const int tid = threadIdx.x, lane = tid & 31;
  if (tid == 0) s_rank = p;
  __syncthreads();
  const double r00 = fabs(W[(size_t)perm[0] * n_pad]);
  for (int c = tid; c < p; c += 256)
    if (c >= n || !(fabs(W[(size_t)perm[c] * n_pad + c]) > 1e-13 * r00)) atomicMin(&s_rank, c);
  __syncthreads();
  const int r = s_rank;
  if (tid == 0) *rank_out = r;
  for (int q = tid; q < p; q += 256) work[q] = (q < r) ? y[q] : 0.0;
  __syncthreads();
  for (int c1 = r; c1 > 0; c1 -= 32) {
    const int c0 = max(0, c1 - 32), nb = c1 - c0;
    if (tid < 32) {
      const double* col = W + (size_t)perm[lane < nb ? c0 + lane : c0] * n_pad;
      cols[lane] = col;
      __syncwarp();
#pragma unroll 8
      for (int c = 0; c < nb; ++c)
        if (lane < c) tri[c][lane] = cols[c][c0 + lane];
      __syncwarp();
      double w = lane < nb ? work[c0 + lane] : 0.0;
      const double dg = lane < nb ? 1.0 / col[c0 + lane] : 1.0;
      for (int c = nb - 1; c >= 0; --c) {
        if (lane == c) w *= dg;
        const double xc = __shfl_sync(0xffffffffu, w, c);
        if (lane < c) w -= tri[c][lane] * xc;
      }
      xs[lane] = w;
      if (lane < nb) work[c0 + lane] = w;
    }
    __syncthreads();
    for (int q = tid; q < c0; q += 256) {
      double w = work[q];
#pragma unroll 8
      for (int c = nb - 1; c >= 0; --c) w -= cols[c][q] * xs[c];  // R_qc = W[perm[c]][q]
      work[q] = w;
    }
    __syncthreads();
  }
  for (int q = tid; q < p; q += 256) delta[perm[q]] = work[q];
}

}  // namespace

// delta = argmin |c - X delta| by pivoted QR; the workspace (W: p x n_pad,
// y: n, norms, perm, rank, the barrier's words) is P.qr_*
void launch_qr_solve(const ProblemDev& P, cudaStream_t st) {
  launch_pdl(k_qr_init, P.p + 1, 256, 0, st, P.n, P.n_pad, P.p, P.B, P.c, P.qr_W, P.qr_y, P.qr_nrm,
                                     P.qr_perm, P.qr_sync);
  int n = P.n, n_pad = P.n_pad, p = P.p, steps = P.p < P.n ? P.p : P.n;
  double *W = P.qr_W, *y = P.qr_y, *nrm = P.qr_nrm;
  int *perm = P.qr_perm, *status = P.status;
  uint32_t* sync = P.qr_sync;
  const int sms = device_sm_count();
  const int grid = p + 1 < sms ? p + 1 : sms;
  const size_t order = (size_t)p * 5 + 16, col = (size_t)n * 8, room = 200 * 1024;  // order: pos and done
  const bool stage = col + order <= room;
  const bool keep = col * (1 + (size_t)(p / grid + 1)) + order <= room;
  const size_t smem = order + (keep ? col * (1 + (size_t)(p / grid + 1)) : stage ? col : 0);
  const void* kern = keep    ? (const void*)k_qr_factor<true, true>
                     : stage ? (const void*)k_qr_factor<true, false>
                             : (const void*)k_qr_factor<false, false>;
  smem_limit<SMEM_PER_CTA - 5 * 1024>(kern);  // less the static part
  void* args[] = {&n, &n_pad, &p, &steps, &W, &y, &nrm, &perm, &sync, &status};
  cudaLaunchCooperativeKernel(kern, dim3(grid), dim3(QR_THREADS), args, smem, st);
  launch_pdl(k_qr_solve, 1, 256, 0, st, n, n_pad, p, W, y, perm, P.delta, P.res, P.qr_rank);
}
