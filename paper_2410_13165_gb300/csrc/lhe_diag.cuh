// lhe_diag.cuh -- the per-node body and the block reduction of the diagnostics (mass, kinetic
// entropy of Eq. (skfk), max |phi|, non-finite count), shared by the handle's reduction kernels
// (lhe_misc.cu) and the allocation-free entry point (lhe_noalloc.cu), so that both compute the same
// formula in the same order.
#pragma once

#include <cstdint>

#include "lhe_device.cuh"

namespace lhe {

// Constants of the diagnostics of one state, formed on the host: iw_k = 1 / (2 omega_k) and
// inv2 = 1 / (1 - s)^2 (1 for s = 1), so that a node takes no FP64 division: the GB300 retires ~2 FP64
// operations per clock per SM, and two divisions per population made the reduction ~35 times slower than
// reading the state (D3Q19 96^3: 753 us with the final pass, now 136; reading the state takes 20).
struct DiagCoef {
  double omega[kMaxQ];
  double iw[kMaxQ];
  double inv2;
};

inline DiagCoef diag_coef(int Q, const double *omega, double s) {
  DiagCoef c{};
  for (int k = 0; k < Q; ++k) {
    c.omega[k] = omega[k];
    c.iw[k] = 1.0 / (2.0 * omega[k]);
  }
  c.inv2 = s != 1.0 ? 1.0 / ((1.0 - s) * (1.0 - s)) : 1.0;
  return c;
}

__device__ __forceinline__ bool nonfinite_bits(double x) { return (__double2hiint(x) & 0x7FF00000) == 0x7FF00000; }

// One node of an FP64 post-collision state f* (k-major, Q*S): phi = sum_k f*_k - dt R; the
// pre-collision populations recovered from f* = (1 - s) f + omega (s phi + dt R) (for s = 1 the
// post-collision values are used: psi = 0); the entropy sum_k f_k^2 / (2 omega_k) and the
// number of non-finite populations. Accumulates into v = {mass, entropy, max |phi|, non-finite}.
// Each population is read once; the moment sum and the test for non-finite values run on the integer
// pipes, so three FP64 operations per population remain (d = f*_k - omega_k psi, d^2, and the sum).
template <int Q>
__device__ __forceinline__ void diag_site_fp64(const double *__restrict__ pop, int64_t S, int64_t site,
                                               const DiagCoef &c, double s, double dtR, double (&v)[4]) {
  double f[Q];
  int bad = 0;
#pragma unroll
  for (int k = 0; k < Q; ++k) f[k] = __ldg(pop + k * S + site);
#pragma unroll
  for (int k = 0; k < Q; ++k) bad += nonfinite_bits(f[k]) ? 1 : 0;
  double sum = fixed_moment_sum<Q, 0>(f);
  if (bad) {  // the floating sum of infinities and NaN
    sum = 0.0;
#pragma unroll
    for (int k = 0; k < Q; ++k) sum += f[k];
  }
  const double phi = sum - dtR;
  const double psi = s != 1.0 ? s * phi + dtR : 0.0;
  double ent = 0.0;
#pragma unroll
  for (int k = 0; k < Q; ++k) {
    const double d = fma(-c.omega[k], psi, f[k]);
    ent = fma(d * d, c.iw[k], ent);
  }
  v[0] += phi;
  v[1] = fma(ent, c.inv2, v[1]);
  v[2] = fmax(v[2], fabs(phi));
  v[3] += (double)bad;
}

// Sum (max for v[2]) of v over the block: warp shuffles, then warp 0's lane 0 adds the warps'
// results in warp order. The block's total is valid in thread 0 only. sh: 4 doubles per warp.
__device__ __forceinline__ void block_reduce4(double (&v)[4], double *sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    v[0] += __shfl_down_sync(0xffffffffu, v[0], o);
    v[1] += __shfl_down_sync(0xffffffffu, v[1], o);
    v[2] = fmax(v[2], __shfl_down_sync(0xffffffffu, v[2], o));
    v[3] += __shfl_down_sync(0xffffffffu, v[3], o);
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (lane == 0)
    for (int j = 0; j < 4; ++j) sh[wid * 4 + j] = v[j];
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < nw; ++w) {
      v[0] += sh[w * 4 + 0];
      v[1] += sh[w * 4 + 1];
      v[2] = fmax(v[2], sh[w * 4 + 2]);
      v[3] += sh[w * 4 + 3];
    }
  }
}

// Second pass (loads past L1: the partials may come from this launch): one block adds the per-block partials (4 per block) in block order and writes the
// four totals to out.
__device__ __forceinline__ void reduce_partials_final(const double *partials, int nblocks, double *out, double *sh) {
  double v[4] = {0.0, 0.0, 0.0, 0.0};
  for (int b = threadIdx.x; b < nblocks; b += blockDim.x) {
    v[0] += __ldcg(partials + b * 4 + 0);
    v[1] += __ldcg(partials + b * 4 + 1);
    v[2] = fmax(v[2], __ldcg(partials + b * 4 + 2));
    v[3] += __ldcg(partials + b * 4 + 3);
  }
  block_reduce4(v, sh);
  if (threadIdx.x == 0)
    for (int j = 0; j < 4; ++j) out[j] = v[j];
}

}  // namespace lhe
