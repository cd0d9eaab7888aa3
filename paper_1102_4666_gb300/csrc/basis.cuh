// basis.cuh -- the random points of Algorithm 2 and the basis values at them,
// shared by the basis-matrix kernel and the fused Gram kernel.
#pragma once
#include "common.cuh"

struct BoxArgs {
  double lo[BSDE_DMAX + 1], hi[BSDE_DMAX + 1];
};
inline BoxArgs box_args(const ModelHost& m, const GridHost& g) {
  BoxArgs box = {};
  for (int v = 0; v <= m.d; ++v) {
    box.lo[v] = g.lo[v];
    box.hi[v] = g.hi[v];
  }
  return box;
}

constexpr int BASIS_PTS = 32;  // points per CTA, one per lane

__device__ __forceinline__ float to_tf32(float v) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(v));
  return __uint_as_float(r);
}

// Algorithm 2, first step of iteration k: point i takes coordinate c from
// lane c%4 of the Philox block (c/4, i, 0, TAG_PTS<<24 | k) and maps the
// uniform u = (w + 1/2) 2^-32 onto [lo_c, hi_c].  Explicit _rn operations
// keep every rounding as written (no FMA contraction).  A CTA draws the points
// i0 .. i0 + 31 (store(c, i, y) is called for every coordinate) and tabulates
// T_0..T_eta of their dp reduced coordinates in shared memory, cheb[v][e][point],
// so that the FP64 division and recurrence run once per (point, variate) and CTA.
template <typename Store>
__device__ __forceinline__ void basis_tables(int n, int i0, int dp, int eta, const uint32_t* key,
                                             uint32_t k, const BoxArgs& box, double* cheb,
                                             Store&& store) {
  const int tid = threadIdx.x, nth = blockDim.x;
  const int vrow = (eta + 1) * BASIS_PTS;  // one variate's table
  const Philox ph{key[0], key[1]};
  for (int idx = tid; idx < (dp + 3) / 4 * BASIS_PTS; idx += nth) {
    const int blk = idx / BASIS_PTS, q = idx - blk * BASIS_PTS, i = i0 + q;
    if (i >= n) continue;
    const uint4 o = ph((uint32_t)blk, (uint32_t)i, 0u, (TAG_PTS << 24) | k);
    const uint32_t w[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
    for (int c4 = 0; c4 < 4; ++c4) {
      const int c = blk * 4 + c4;
      if (c >= dp) break;
      const double u = __dmul_rn((double)w[c4] + 0.5, 2.3283064365386962890625e-10);
      const double y = __dadd_rn(box.lo[c], __dmul_rn(__dsub_rn(box.hi[c], box.lo[c]), u));
      cheb[c * vrow + q] = y;  // the place of T_0 until the tables are built
      store(c, i, y);
    }
  }
  __syncthreads();
  for (int idx = tid; idx < dp * BASIS_PTS; idx += nth) {
    const int v = idx / BASIS_PTS, q = idx - v * BASIS_PTS;
    if (i0 + q >= n) continue;
    double* tv = cheb + (size_t)v * vrow + q;
    const double y = tv[0];
    const double xi = __ddiv_rn(__dsub_rn(__dmul_rn(2.0, y), __dadd_rn(box.lo[v], box.hi[v])),
                                __dsub_rn(box.hi[v], box.lo[v]));
    tv[0] = 1.0;
    if (eta >= 1) tv[BASIS_PTS] = xi;
    double tm1 = 1.0, tc = xi;
    for (int e = 2; e <= eta; ++e) {
      const double tn = __dsub_rn(__dmul_rn(__dmul_rn(2.0, xi), tc), tm1);
      tm1 = tc;
      tc = tn;
      tv[(size_t)e * BASIS_PTS] = tc;
    }
  }
  __syncthreads();
}

// one basis function at the lane's point, the factors in the order of the definition
__device__ __forceinline__ double basis_at(uint2 pr, int nz, int eta, const double* cheb) {
  const int lane = threadIdx.x & 31;
  double val = 1.0;
  for (int a = 0; a < nz; ++a) {
    const uint32_t byte = ((a < 4 ? pr.x >> (8 * a) : pr.y >> (8 * (a - 4)))) & 0xffu;
    const int v = (int)(byte >> 4), e = (int)(byte & 15u);
    val = __dmul_rn(val, cheb[((size_t)v * (eta + 1) + e) * BASIS_PTS + lane]);
  }
  return val;
}
