// lhe_misc.cu -- initialisation, finite-difference gradient, diagnostics reduction and the
// adjoint seed / gradient kernels.
#include <algorithm>
#include <type_traits>

#include "lhe_diag.cuh"
#include "lhe_internal.h"
#include "lhe_sites.cuh"

namespace lhe {

// ------------------------------------------------------------------------------ FD gradient
// Periodic fourth-order central difference: d_i phi ~ (-phi(x+2e_i) + 8 phi(x+e_i) - 8 phi(x-e_i)
// + phi(x-2e_i)) / (12 dx).
__device__ __forceinline__ int32_t wrap_off(int xi, int o, int32_t n, int32_t stride) {
  int y = xi + o;
  if (y < 0) y += n;
  if (y >= n) y -= n;
  return (y - xi) * stride;
}

// phi(x + e_i) - phi(x - e_i) and phi(x + 2e_i) - phi(x - 2e_i); `near`: the largest high word of their magnitudes.
__device__ __forceinline__ void fd_differences(const double *__restrict__ v, int32_t site, int xi, int32_t n,
                                               int32_t stride, double &d1, double &d2, unsigned &near) {
  const double p1 = __ldg(v + site + wrap_off(xi, 1, n, stride)), m1 = __ldg(v + site + wrap_off(xi, -1, n, stride));
  const double p2 = __ldg(v + site + wrap_off(xi, 2, n, stride)), m2 = __ldg(v + site + wrap_off(xi, -2, n, stride));
  d1 = p1 - m1;
  d2 = p2 - m2;
  const unsigned a = max((unsigned)__double2hiint(p1) & 0x7FFFFFFFu, (unsigned)__double2hiint(m1) & 0x7FFFFFFFu);
  const unsigned b = max((unsigned)__double2hiint(p2) & 0x7FFFFFFFu, (unsigned)__double2hiint(m2) & 0x7FFFFFFFu);
  near = max(near, max(a, b));
}

// Adds D_i^T G_i = -D_i G_i to `out` (the transpose of the difference).
template <int D>
__global__ void __launch_bounds__(256) k_fd_transpose(const Geom g, double inv12dx, const double *__restrict__ in,
                                                      double *__restrict__ out) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= g.S) return;
  int x[D];
  const int32_t site = decode_site<D, false>(g, t, x);
  double acc = out[site];
#pragma unroll
  for (int i = 0; i < D; ++i) {
    const double *v = in + (int64_t)i * g.S;
    const double p2 = v[site + wrap_off(x[i], 2, g.n[i], g.stride[i])];
    const double p1 = v[site + wrap_off(x[i], 1, g.n[i], g.stride[i])];
    const double m1 = v[site + wrap_off(x[i], -1, g.n[i], g.stride[i])];
    const double m2 = v[site + wrap_off(x[i], -2, g.n[i], g.stride[i])];
    acc -= (-p2 + 8.0 * p1 - 8.0 * m1 + m2) * inv12dx;
  }
  out[site] = acc;
}

cudaError_t launch_fd_grad_transpose_add(int d, const Geom &g, double dx, const double *G, double *out,
                                         cudaStream_t st) {
  const unsigned blocks = (unsigned)((g.S + 255) / 256);
  const double w = 1.0 / (12.0 * dx);
  switch (d) {
    case 1: k_fd_transpose<1><<<blocks, 256, 0, st>>>(g, w, G, out); break;
    case 2: k_fd_transpose<2><<<blocks, 256, 0, st>>>(g, w, G, out); break;
    case 3: k_fd_transpose<3><<<blocks, 256, 0, st>>>(g, w, G, out); break;
    case 4: k_fd_transpose<4><<<blocks, 256, 0, st>>>(g, w, G, out); break;
    case 5: k_fd_transpose<5><<<blocks, 256, 0, st>>>(g, w, G, out); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------ initialisation
// Eq. (ini-simp): f_k(x,0) = omega_k [phi0 + (dt/2)(u - c e_k) . grad phi0] (order 3) or
// omega_k phi0 (order 1); the stored state is post-collision. The first moment of the correction
// vanishes (sum_k omega_k (u - c e_k) = 0), so the collision f*_k = (1 - s) f_k + omega_k (s phi0 + dt R) is
//   f*_k = omega_k (B - sum_i e_ki h_i),  h_i = (1 - s)(dt/2) c d_i phi0,
//   B = phi0 + dt R + (1 - s)(dt/2) u . grad phi0                                    (FP64)
//   g*_k = f*_k - omega_k phi0: the same with B = dt R + (1 - s)(dt/2) u . grad phi0,  phi = phi0   (FP32_DEV)
// The gradient is read (kGradGiven) or formed here from phi0 (kGradFD), which saves its trip through memory.
// Bound by the FP64 pipe (~2 operations per clock per SM), not by memory, unless operations are spared:
// two per population here (the four values B -+ (h_i +- h_j) of a pair share their sums), against five
// before (D3Q19 256^3, gradient formed: 3.03 -> 1.89 ms; the memory floor is 0.42).
// FP32_DEV results are rounded to float, so the sums and products run on float pairs (48 bits) on the FP32
// pipe and only the differences of phi0 in FP64. A result whose rounding the pairs' error could change
// (Ziv's rounding test, "Fast evaluation of elementary mathematical functions with correctly rounded last
// bit", TOMS 1991), and every one outside the pairs' range (largest term outside 2^-60 .. 2^100, infinities, NaN),
// is formed in FP64 instead, so the stored floats are those of the FP64 form at every node. (The test's bound counts
// what ff_split drops of a term below 2^-70, at most 2^-94, with the largest weight it can meet: relative to the largest
// term alone, a source of 2^-71 beside a gradient of 2^-58 was rounded wrongly at 2 to 3 of 100 populations.) D3Q19 128^3
// 451 -> 77 us (memory floor 36), D5Q51 24^5 4.24 -> 0.66 ms (floor 0.26).
constexpr int kGradNone = 0, kGradGiven = 1, kGradFD = 2;

// v_k = omega_k (B - sum_i e_ki h_i) for every k, with the arithmetic of T (double or float pairs).
template <int D, class T, class Add, class Sub, class Out>
__device__ __forceinline__ void init_populations(T B, const T (&h)[D], Add add, Sub sub, Out out) {
  out(0, B);
#pragma unroll
  for (int i = 0; i < D; ++i) {
    out(1 + i, sub(B, h[i]));
    out(1 + D + i, add(B, h[i]));
  }
  int k = 2 * D + 1;
#pragma unroll
  for (int i = 0; i < D; ++i)
#pragma unroll
    for (int j = i + 1; j < D; ++j) {  // components (1, 1), (-1, 1), (-1, -1), (1, -1)
      const T p = add(h[i], h[j]), q = sub(h[i], h[j]);
      out(k, sub(B, p));
      out(k + 1, add(B, q));
      out(k + 2, add(B, p));
      out(k + 3, sub(B, q));
      k += 4;
    }
}

// g*_k of one node in FP64, rounded to float, for the populations of `mask` at least. The gradient is formed once; a
// few populations are formed one by one, and all of them together (the others' stored floats stay the same) once a
// lane of the warp has half of them to do, as on plateaus of phi0, where the pairs decide no rounding. (A gradient per population:
// constant field, D3Q19 128^3 1,977 us, now 452; D5Q51 16^5 4,020, now 559; fields whose roundings are decided 76 and 78.)
template <int D, int GRAD>
__device__ __noinline__ void deviations_fp64(const InitArgs &a, int32_t site, uint64_t mask) {
  constexpr Lattice<D> L{};
  constexpr int Q = Lattice<D>::Q;
  const double dtR = a.Rfield ? a.dt * __ldg(a.Rfield + site) : a.dtR;
  int x[D];
  decode_site<D, false>(a.g, site, x);
  double gr[D], ug = 0.0;
#pragma unroll
  for (int i = 0; i < D; ++i) {
    gr[i] = 0.0;
    if (GRAD == kGradGiven) gr[i] = __ldg(a.grad + i * a.g.S + site);
    if (GRAD == kGradFD) {
      const double p2 = __ldg(a.phi0 + site + wrap_off(x[i], 2, a.g.n[i], a.g.stride[i]));
      const double p1 = __ldg(a.phi0 + site + wrap_off(x[i], 1, a.g.n[i], a.g.stride[i]));
      const double m1 = __ldg(a.phi0 + site + wrap_off(x[i], -1, a.g.n[i], a.g.stride[i]));
      const double m2 = __ldg(a.phi0 + site + wrap_off(x[i], -2, a.g.n[i], a.g.stride[i]));
      gr[i] = (fma(-8.0, m1, fma(8.0, p1, -p2)) + m2) * a.inv12dx;
    }
    ug = fma(a.u[i], gr[i], ug);
  }
  float *__restrict__ dst = static_cast<float *>(a.dst) + site;
  const auto value = [&](int k, double eg) { return (float)fma(a.omega[k], dtR, fma(-a.c2[k], eg, a.c1[k] * ug)); };
  if (__any_sync(__activemask(), __popcll(mask) > Q / 2)) {
#pragma unroll
    for (int k = 0; k < Q; ++k) {
      double eg = 0.0;
#pragma unroll
      for (int i = 0; i < D; ++i) {
        if (L.e[k][i] == 1) eg += gr[i];
        if (L.e[k][i] == -1) eg -= gr[i];
      }
      dst[k * a.g.S] = value(k, eg);
    }
    return;
  }
  for (; mask; mask &= mask - 1) {
    const int k = __ffsll((long long)mask) - 1;
    double g0 = 0.0, g1 = 0.0;  // e_ki d_i phi0 of the link's first and last direction (a sum over all i is D FP64 operations)
#pragma unroll
    for (int i = 0; i < D; ++i) {
      const int e = a.e[k][i];
      const double v = __hiloint2double(__double2hiint(gr[i]) ^ (e & (int)0x80000000), __double2loint(gr[i]));
      if (e != 0) {
        g0 = g1;
        g1 = v;
      }
    }
    dst[k * a.g.S] = value(k, g0 + g1);
  }
}

template <int D, bool DEV, int GRAD>
__global__ void __launch_bounds__(256) k_init(const __grid_constant__ InitArgs a) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t S = a.g.S;
  if (t >= S) return;
  const int32_t site = (int32_t)t;
  const double phi0 = __ldg(a.phi0 + site);
  const double dtR = a.Rfield ? a.dt * __ldg(a.Rfield + site) : a.dtR;
  // g1: the gradient, or phi(x+e_i) - phi(x-e_i), and g2 = phi(x+2e_i) - phi(x-2e_i)
  double g1[D], g2[D];
  unsigned near = 0u;  // high word of the largest |phi0| that the differences were formed from
  if (GRAD == kGradFD) {
    int x[D];
    decode_site<D, false>(a.g, t, x);
#pragma unroll
    for (int i = 0; i < D; ++i) fd_differences(a.phi0, site, x[i], a.g.n[i], a.g.stride[i], g1[i], g2[i], near);
  } else {
#pragma unroll
    for (int i = 0; i < D; ++i) {
      g1[i] = GRAD == kGradGiven ? __ldg(a.grad + i * S + site) : 0.0;
      g2[i] = 0.0;
    }
  }
  if (DEV) {
    float *__restrict__ dst = static_cast<float *>(a.dst);
    int top = double_exponent(dtR);
#pragma unroll
    for (int i = 0; i < D; ++i) {
      top = max(top, double_exponent(g1[i]));
      if (GRAD == kGradFD) top = max(top, double_exponent(g2[i]));
    }
    const int ep = double_exponent(phi0), en = (int)(near >> 20) - 1023;
    a.phi_dst[site] = (ep >= -60 && ep <= 100) ? ff_split(phi0) : df_split(phi0);
    uint64_t doubt = ~0ull;  // populations whose rounding the pairs do not decide
    if (a.pairs && en <= 100 && ((top >= -60 && top <= 100) || top == -1023)) {
      float2 h[D], B = ff_split(dtR);
      float err = fabsf(B.x);  // sum of the magnitudes of the terms
#pragma unroll
      for (int i = 0; i < D; ++i) {
        float2 g = ff_split(g1[i]);
        float m = fabsf(g.x);
        if (GRAD == kGradFD) {
          const float2 w = ff_split(g2[i]);
          g = ff_sub(make_float2(8.0f * g.x, 8.0f * g.y), w);
          m = fmaf(8.0f, m, fabsf(w.x));
        }
        if (GRAD != kGradNone) B = ff_add(B, ff_mul(a.wu_f[i], g));
        h[i] = ff_mul(a.wc_f, g);
        err = fmaf(a.werr, m, err);
      }
      // bound of the difference to the FP64 form: 2^-43 of the terms (an operation on pairs is within ~2^-45
      // of its operands), what the split drops, and the rounding of the FP64 differences, 2^-48 of the values that enter them
      const float terms = err;
      err *= 0x1p-43f;
      if (top != -1023) err += a.edrop;
      if (GRAD == kGradFD) err = fmaf(a.werr * 0x1p-48f, ff_split(__hiloint2double((int)near, 0)).x, err);
      if (err <= terms * 0x1p-28f) {  // (else few roundings are decided: plateaus of phi0, or a small signal on a large mean)
        doubt = 0;
        init_populations<D>(
            B, h, [](float2 p, float2 q) { return ff_add(p, q); }, [](float2 p, float2 q) { return ff_sub(p, q); },
            [&](int k, float2 v) {
              const float2 w = a.omega_f[k];
              const float p = __fmul_rn(w.x, v.x);
              const float e = __fmaf_rn(w.x, v.y, __fmaf_rn(w.y, v.x, __fmaf_rn(w.x, v.x, -p)));
              const float r = __fadd_rn(p, __fmaf_rn(w.x, err, e));
              doubt |= (uint64_t)(r != __fadd_rn(p, __fmaf_rn(-w.x, err, e))) << k;
              dst[k * S + site] = r;
            });
      }
    }
    if (doubt) deviations_fp64<D, GRAD>(a, site, doubt);
    return;
  }
  double h[D], B = phi0 + dtR;
#pragma unroll
  for (int i = 0; i < D; ++i) {
    const double g = GRAD == kGradFD ? fma(8.0, g1[i], -g2[i]) : g1[i];
    if (GRAD != kGradNone) B = fma(a.wu[i], g, B);
    h[i] = a.wc * g;
  }
  double *__restrict__ dst = static_cast<double *>(a.dst);
  init_populations<D>(B, h, [](double p, double q) { return p + q; }, [](double p, double q) { return p - q; },
                      [&](int k, double v) { dst[k * S + site] = a.omega[k] * v; });
}

template <int D, int GRAD>
static cudaError_t init_dg(bool dev, const InitArgs &a, cudaStream_t st) {
  const unsigned blocks = (unsigned)((a.g.S + 255) / 256);
  if (dev) k_init<D, true, GRAD><<<blocks, 256, 0, st>>>(a);
  else k_init<D, false, GRAD><<<blocks, 256, 0, st>>>(a);
  return cudaGetLastError();
}

template <int D>
static cudaError_t init_d(bool dev, const InitArgs &a, cudaStream_t st) {
  if (a.order != 3) return init_dg<D, kGradNone>(dev, a, st);
  return a.grad ? init_dg<D, kGradGiven>(dev, a, st) : init_dg<D, kGradFD>(dev, a, st);
}

cudaError_t launch_init(int d, bool dev, const InitArgs &a, cudaStream_t st) {
  switch (d) {
    case 1: return init_d<1>(dev, a, st);
    case 2: return init_d<2>(dev, a, st);
    case 3: return init_d<3>(dev, a, st);
    case 4: return init_d<4>(dev, a, st);
    case 5: return init_d<5>(dev, a, st);
    default: return cudaErrorInvalidValue;
  }
}

// ------------------------------------------------------------------------------ diagnostics
// Per site: phi (from the post-collision state: sum_k f*_k - dt R), the pre-collision populations
// recovered from f* = (1-s) f + omega (s phi + dt R) (s != 1; for s = 1 the post-collision values
// are used), the kinetic entropy sum_k f_k^2 / (2 omega_k) (Eq. (skfk)), |phi| and non-finite
// values. Block partials go to a scratch array; the block that finishes last adds them in block
// order, so the result does not depend on scheduling.
template <int D, bool DEV>
__global__ void __launch_bounds__(256) k_reduce(const ReduceArgs a) {
  constexpr int Q = Lattice<D>::Q;
  __shared__ double sh[8 * 4];
  __shared__ bool last;
  const int64_t S = a.g.S;
  double v[4] = {0.0, 0.0, 0.0, 0.0};
  for (int64_t site = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; site < S;
       site += (int64_t)gridDim.x * blockDim.x) {
    const double dtR = a.Rfield ? a.dt * a.Rfield[site] : a.dtR;
    if (DEV) {
      // sum_k f_k^2/(2 w_k) = phi^2/2 + sum_k g_k^2/(2 w_k) since sum_k g_k = 0
      const float *__restrict__ g = static_cast<const float *>(a.pop);
      const double phi = df_value(a.phi[site]);
      const double rdtR = a.s != 1.0 ? dtR : 0.0;
      int bad = nonfinite_bits(phi) ? 1 : 0;
      double ent = 0.0;
#pragma unroll
      for (int k = 0; k < Q; ++k) {
        const double gs = (double)__ldg(g + k * S + site);
        bad += nonfinite_bits(gs) ? 1 : 0;
        const double d = fma(-a.c.omega[k], rdtR, gs);
        ent = fma(d * d, a.c.iw[k], ent);
      }
      v[0] += phi;
      v[1] += fma(ent, a.c.inv2, 0.5 * phi * phi);
      v[2] = fmax(v[2], fabs(phi));
      v[3] += (double)bad;
    } else {
      diag_site_fp64<Q>(static_cast<const double *>(a.pop), S, site, a.c, a.s, dtR, v);
    }
  }
  block_reduce4(v, sh);
  if (threadIdx.x == 0) {
    for (int j = 0; j < 4; ++j) a.partials[blockIdx.x * 4 + j] = v[j];
    __threadfence();
    last = atomicInc(a.done, gridDim.x - 1) == gridDim.x - 1;  // wraps to 0 for the next launch
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  reduce_partials_final(a.partials, (int)gridDim.x, a.out, sh);
}

template <int D>
static cudaError_t reduce_d(bool dev, const ReduceArgs &a, int nblocks, cudaStream_t st) {
  if (dev) k_reduce<D, true><<<nblocks, 256, 0, st>>>(a);
  else k_reduce<D, false><<<nblocks, 256, 0, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_reduce(int d, bool dev, const ReduceArgs &a, int nblocks, cudaStream_t st) {
  nblocks = (int)std::min<int64_t>(nblocks, (a.g.S + 255) / 256);
  switch (d) {
    case 1: return reduce_d<1>(dev, a, nblocks, st);
    case 2: return reduce_d<2>(dev, a, nblocks, st);
    case 3: return reduce_d<3>(dev, a, nblocks, st);
    case 4: return reduce_d<4>(dev, a, nblocks, st);
    case 5: return reduce_d<5>(dev, a, nblocks, st);
    default: return cudaErrorInvalidValue;
  }
}

// ------------------------------------------------------------------------------ adjoint
// Seed: nu_k(x, T) = dL/dphi_T(x) for every k (phi_T = sum_k f*_k - dt R), stored as
// zeta_k = omega_k nu_k (FP64) or as W = dL/dphi_T, eps_k = 0 (FP32_DEV); dL/dR := 0.
template <int D, bool DEV>
__global__ void __launch_bounds__(256) k_adj_seed(const Geom g, const StepArgs w, const double *__restrict__ seed,
                                                  void *adj, float2 *adjW, double *gR) {
  constexpr int Q = Lattice<D>::Q;
  const int64_t site = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (site >= g.S) return;
  const double s0 = seed[site];
#pragma unroll
  for (int k = 0; k < Q; ++k) {
    if (DEV) static_cast<float *>(adj)[k * g.S + site] = 0.0f;
    else static_cast<double *>(adj)[k * g.S + site] = w.omega[k] * s0;
  }
  if (DEV) adjW[site] = df_split(s0);
  gR[site] = 0.0;
}

template <int D>
static cudaError_t seed_d(bool dev, const Geom &g, const StepArgs &w, const double *seed, void *adj, float2 *adjW,
                          double *gR, cudaStream_t st) {
  const unsigned blocks = (unsigned)((g.S + 255) / 256);
  if (dev) k_adj_seed<D, true><<<blocks, 256, 0, st>>>(g, w, seed, adj, adjW, gR);
  else k_adj_seed<D, false><<<blocks, 256, 0, st>>>(g, w, seed, adj, adjW, gR);
  return cudaGetLastError();
}

cudaError_t launch_adjoint_seed(int d, bool dev, const Geom &g, const double *omega, const double *seed, void *adj,
                                float2 *adjW, double *gR, cudaStream_t st) {
  StepArgs w{};
  for (int k = 0; k < kMaxQ; ++k) w.omega[k] = omega[k];
  switch (d) {
    case 1: return seed_d<1>(dev, g, w, seed, adj, adjW, gR, st);
    case 2: return seed_d<2>(dev, g, w, seed, adj, adjW, gR, st);
    case 3: return seed_d<3>(dev, g, w, seed, adj, adjW, gR, st);
    case 4: return seed_d<4>(dev, g, w, seed, adj, adjW, gR, st);
    case 5: return seed_d<5>(dev, g, w, seed, adj, adjW, gR, st);
    default: return cudaErrorInvalidValue;
  }
}

// Transpose of the initialisation (with its collision) applied to zeta^0 = omega nu^0,
// nu^0 = dL/df(0):  dL/dphi0 = Z = sum_k zeta_k;  G_i = (dt/2) sum_k (u_i - c e_ki) zeta_k
// = (dt/2)(u_i Z - c E_i), E_i = sum_k e_ki zeta_k (= dL/d(grad phi0)_i for order 3). FP32_DEV: zeta_k =
// omega_k W + eps_k, where the W part cancels in G because sum_k omega_k (u - c e_k) = 0.
// The D + 1 sums run in 64-bit fixed point (as the moment sum: error below one unit in the last place of the
// largest term) and share each term's alignment, so that ~4 (D + 1) FP64 operations per node remain instead
// of (D + 1) Q + Q conversions: D3Q19 128^3 FP32 deviations 428 -> 71 us (memory floor 34).
template <int D, bool DEV>
__global__ void __launch_bounds__(256) k_adj_grads(const AdjGradArgs a) {
  constexpr Lattice<D> L{};
  constexpr int Q = Lattice<D>::Q;
  const int64_t site = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t S = a.g.S;
  if (site >= S) return;
  const bool want_g = a.order == 3 && a.G;
  using Z_t = typename std::conditional<DEV, float, double>::type;
  Z_t z[Q];
  unsigned top = 0u;  // largest exponent field: of the floats, or in place in the doubles' high words
#pragma unroll
  for (int k = 0; k < Q; ++k) {
    z[k] = __ldg(static_cast<const Z_t *>(a.adj) + k * S + site);
    top = max(top, DEV ? ((unsigned)__float_as_int((float)z[k]) >> 23) & 0xFFu : (unsigned)__double2hiint((double)z[k]) & kExpField);
  }
  double Z = 0.0, E[D];
  if (top == (DEV ? 0xFFu : kExpField) || (!DEV && top < kFixedLeast)) {  // plain sums (infinities, NaN, and values below 2^-954)
#pragma unroll
    for (int i = 0; i < D; ++i) E[i] = 0.0;
#pragma unroll
    for (int k = 0; k < Q; ++k) {
      Z += z[k];
#pragma unroll
      for (int i = 0; i < D; ++i) {
        if (L.e[k][i] == 1) E[i] += z[k];
        if (L.e[k][i] == -1) E[i] -= z[k];
      }
    }
  } else {
    constexpr int G = 10 - ceil_log2(Q);
    const unsigned emf = DEV ? (max(top, 1u) + 896u) << 20 : top;
    long long accz = 0, acce[D];
#pragma unroll
    for (int i = 0; i < D; ++i) acce[i] = 0;
#pragma unroll
    for (int k = 0; k < Q; ++k) {
      const long long v = fixed_align<G>(z[k], DEV ? top : emf);
      accz += v;
#pragma unroll
      for (int i = 0; i < D; ++i) {
        if (L.e[k][i] == 1) acce[i] += v;
        if (L.e[k][i] == -1) acce[i] -= v;
      }
    }
    Z = fixed_value<G, 0>(accz, emf);
#pragma unroll
    for (int i = 0; i < D; ++i) E[i] = want_g ? fixed_value<G, 0>(acce[i], emf) : 0.0;
  }
  a.gphi0[site] = DEV ? df_value(a.adjW[site]) + Z : Z;
  if (want_g)
#pragma unroll
    for (int i = 0; i < D; ++i) a.G[i * S + site] = 0.5 * a.dt * fma(a.u[i], Z, -(a.c * E[i]));
}

template <int D>
static cudaError_t grads_d(bool dev, const AdjGradArgs &a, cudaStream_t st) {
  const unsigned blocks = (unsigned)((a.g.S + 255) / 256);
  if (dev) k_adj_grads<D, true><<<blocks, 256, 0, st>>>(a);
  else k_adj_grads<D, false><<<blocks, 256, 0, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_adjoint_grads(int d, bool dev, const AdjGradArgs &a, cudaStream_t st) {
  switch (d) {
    case 1: return grads_d<1>(dev, a, st);
    case 2: return grads_d<2>(dev, a, st);
    case 3: return grads_d<3>(dev, a, st);
    case 4: return grads_d<4>(dev, a, st);
    case 5: return grads_d<5>(dev, a, st);
    default: return cudaErrorInvalidValue;
  }
}

// phi of the FP32-deviation form: double-float pair -> double, two nodes per thread; one FP64 operation per node (the
// conversions by their bits). D5Q51 24^5: 46 -> 19 us (memory floor 19).
__global__ void __launch_bounds__(256) k_df_to_double(const float2 *__restrict__ src, double *__restrict__ dst, int64_t n,
                                                      bool pairs) {
  const int64_t i = 2 * (blockIdx.x * (int64_t)blockDim.x + threadIdx.x);
  if (i >= n) return;
  if (pairs && i + 1 < n) {  // 16-byte accesses (dst is 16-byte aligned)
    const float4 p = *reinterpret_cast<const float4 *>(src + i);
    *reinterpret_cast<double2 *>(dst + i) =
        make_double2(float_to_double(p.x) + float_to_double(p.y), float_to_double(p.z) + float_to_double(p.w));
    return;
  }
  for (int64_t j = i; j < n && j < i + 2; ++j) dst[j] = float_to_double(src[j].x) + float_to_double(src[j].y);
}

cudaError_t launch_df_to_double(const float2 *src, double *dst, int64_t n, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const bool pairs = (reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst)) % 16 == 0;
  k_df_to_double<<<(unsigned)((n + 511) / 512), 256, 0, st>>>(src, dst, n, pairs);
  return cudaGetLastError();
}

// In-place multiplication of an FP64 population array by a constant (undoes the scaled
// representation of the state; see lhe_api.cu).
__global__ void __launch_bounds__(256) k_scale_fp64(double *__restrict__ p, int64_t n, double factor) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) p[i] *= factor;
}

cudaError_t launch_scale_fp64(double *p, int64_t n, double factor, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  k_scale_fp64<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(p, n, factor);
  return cudaGetLastError();
}

}  // namespace lhe
