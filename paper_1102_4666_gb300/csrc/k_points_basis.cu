// k_points_basis.cu -- the random points of Algorithm 2 and the basis matrix
// B_l(t_i, x_i) of the least-squares extrapolation (eq. lspb, Section 3.2.2).
#include "basis.cuh"

namespace {

// B[l][i] = prod over the active variates v of T_{nu_lv}(xi_v(t_i, x_i)),
// xi_v = (2 y_v - (lo_v + hi_v)) / (hi_v - lo_v), Chebyshev T_e by the
// three-term recurrence.  A CTA draws 32 consecutive points and tabulates their
// Chebyshev values (basis_tables; a launch of their own for the points cost 2 us
// and a gap, twice an iteration; the CTAs of the first range store them), then
// each warp forms the basis functions l = warp, warp + warps, ... of the CTA's
// range, one lane per point (a 256-byte row segment of B per store).  With
// split != 0 it writes the 3xTF32 operands of the tensor-core Gram instead:
// hi = tf32(fp32(B)), lo = tf32(fp32(B) - hi).  With early != 0 it writes before the
// kernel launched before it (k_refit, which lets it start once it has read B) has
// ended, 10 us an iteration beside it instead of after it.  The basis functions are split over
// gridDim.y ranges only as far as needed for two CTAs per SM.
__global__ void k_basis(int n, int n_pad, int p, int l_per, int dp, int eta, const uint2* pairs,
                        const uint8_t* nnz, const uint32_t* key, uint32_t k, double* t, double* x,
                        const __grid_constant__ BoxArgs box, double* B, float* Bhi, float* Blo,
                        int split, int early) {
  if (!early) pdl_begin();
  extern __shared__ double cheb[];  // [v][e][point]
  const int i0 = blockIdx.x * BASIS_PTS;
  const bool keep = blockIdx.y == 0 && !split;
  basis_tables(n, i0, dp, eta, key, k, box, cheb, [&](int c, int i, double y) {
    if (keep) (c == 0 ? t : x + (size_t)(c - 1) * n)[i] = y;
  });
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int i = i0 + lane;
  const int l0 = blockIdx.y * l_per;
  const int l1 = i < n ? min(p, l0 + l_per) : 0;
  for (int l = l0 + warp; l < l1; l += nw) {
    const double val = basis_at(pairs[l], nnz[l], eta, cheb);
    if (split) {
      const float b32 = __double2float_rn(val);
      const float hi = to_tf32(b32);
      const float lo = to_tf32(b32 - hi);
      Bhi[(size_t)l * n_pad + i] = hi;
      Blo[(size_t)l * n_pad + i] = lo;
    } else {
      B[(size_t)l * n_pad + i] = val;
    }
  }
  if (early) pdl_wait();  // the launches after this one rely on both
}

}  // namespace

void launch_basis(const ModelHost& m, const GridHost& g, const ProblemDev& P, uint32_t k, bool split,
                  bool early, cudaStream_t st) {
  const int dp = m.d + 1, eta = P.eta < 1 ? 1 : P.eta;
  const int tpb = 128;
  const size_t smem = (size_t)dp * (eta + 1) * BASIS_PTS * sizeof(double);
  if (smem > 48 * 1024) smem_limit<(BSDE_DMAX + 1) * 16 * BASIS_PTS * (int)sizeof(double)>(k_basis);
  const int gx = (P.n + BASIS_PTS - 1) / BASIS_PTS;
  const int want = (2 * device_sm_count() + gx - 1) / gx;
  int gy = (P.p + 31) / 32;
  if (gy > want) gy = want;
  if (gy < 1) gy = 1;
  const int l_per = (P.p + gy - 1) / gy;
  gy = (P.p + l_per - 1) / l_per;
  launch_kernel(early, k_basis, dim3(gx, gy), tpb, smem, st, P.n, P.n_pad, P.p, l_per, dp, eta, P.pairs, P.nnz,
             P.key, k, P.t, P.x, box_args(m, g), P.B, P.Bhi, P.Blo, split ? 1 : 0,
             early ? 1 : 0);
}
