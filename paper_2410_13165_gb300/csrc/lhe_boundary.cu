// lhe_boundary.cu -- boundary-node kernels of a Dirichlet box (Sec. 3.2).
//
// One thread per boundary node x (some coordinate at 0 or n_i - 1). For every population k:
//   source x - e_k inside the box : f_k(x, t+dt) = f*_k(x - e_k, t)      (streamed)
//   source outside (unknown)      : full-way, Eq. (bun1), data at (x, t+dt):
//       order 1: omega_k phi
//       order 3: omega_k [phi - (dt/2)(c_k.grad phi + d_t phi)] + (dt/2) omega_k R
//       order 4: order 3 + omega_k (dt^3/24) (c_k.grad + d_t)^3 phi
//     (the four dt^3 terms of Eq. (bun1) are the binomial expansion of (c_k.grad + d_t)^3 / 24)
//                                   half-way, Eq. (bun2) at x_b = x - c_k dt/2, time t:
//       f_k(x, t+dt) = -f*_kbar(x, t) + (w_k + w_kbar)[phi + (dt/2)(phi_t + R) - (dt^2/8) c c:grad^2 phi
//                       - (dt^3/16) c c:grad^2 phi_t - (dt^3/24) phi_ttt]
//                       - (w_k - w_kbar)[(dt^2/4) c.grad phi_t + (dt^3/8) c.grad phi_tt]   (terms by order)
// then the node collides like the bulk. The Dirichlet data phi = h come from the exact-solution
// family h = b + R t + g.(x - u t) + sum_m a_m sin(xi_m), xi_m = kappa_m.(x - u t) + theta_m. Along
// c_k every derivative d_t^q (c_k.grad)^p of a mode is a_m A^p B^q sin^(p+q)(xi_m), A = kappa_m.c_k,
// B = -kappa_m.u, so each scheme is, per unknown k, a node value plus sum_m (U_mk sin xi_m + V_mk
// cos xi_m) with coefficients that depend only on (m, k), the order and the lattice; the host
// tabulates them (the half-way shift to x_b is the rotation of (sin, cos) by (dx/2) kappa_m.e_k,
// folded into U and V). Full-way: f_k = omega_k [h(x) - C_k - sum_m T_mk cos xi_m]; half-way:
// f_k = wp_k lin(x) + K_k + sum_m (U_mk sin xi_m + V_mk cos xi_m) - f*_kbar(x), lin = linear part of h.
// The phase xi_m at a node is assembled from tabulated per-axis factors; boundary nodes come
// grouped by face signature so that a warp shares one set of unknown populations. The per-node
// evaluation (lhe_bnode.cuh) is shared with the FP64 interior kernel of Dirichlet boxes, which treats
// the nodes of the two x_1 faces (whose other coordinates are interior) in the lanes of their rows.
#include <algorithm>
#include <type_traits>

#include "lhe_bnode.cuh"

namespace lhe {

template <int D, int KIND, bool DEV, bool EARLY>
__global__ void __launch_bounds__(128) k_boundary(const BoundaryArgs a) {
  constexpr Lattice<D> L{};
  constexpr int Q = Lattice<D>::Q;
  // FP32 deviations: the family's coefficients in shared memory, since an unknown link's loads are behind a branch and
  // follow one another. FP64 boxes (LHE_FLAG_NODE_BOUNDARY) read them through L1 in CTAs of 128 threads: 33^3 full-way
  // 50 us a step with the copy and smaller CTAs, now 33 (37 before them), 1200^2 97, now 85 (88)
  extern __shared__ double table[];
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  pdl_wait();
  if (DEV && a.rec == nullptr) {
    for (int i = threadIdx.x; i < 2 * (a.nmodes + 1) * Q; i += blockDim.x) table[i] = __ldg(a.table + i);
    __syncthreads();
  }
  if (t >= a.nsites) return;
  const int32_t site = a.sites[t];
  const int64_t S = a.g.S;
  int x[D];
  {
    uint32_t r = (uint32_t)site;
#pragma unroll
    for (int i = 0; i < D; ++i) {
      if (i == D - 1) {
        x[i] = (int)r;
      } else {
        const uint32_t q = a.g.dv[i].div(r);
        x[i] = (int)(r - q * (uint32_t)a.g.n[i]);
        r = q;
      }
    }
  }
  const auto coef = [&](int i) { return DEV ? table[i] : __ldg(a.table + i); };
  BNode<D> nd;
  const bool jets = a.rec != nullptr;  // data from jet records (else from the exact-solution family)
  const double *__restrict__ rec = jets ? a.rec + a.roff[t] : nullptr;
  // EARLY: every load first, so that they are in flight together: a population is read at its pull source, or for an
  // unknown link where the half-way scheme's f*_kbar lies, at the node itself. Else the loads are behind the branch on `inside` and
  // follow one another, Q trips to L2 a node, which is what few nodes wait for; many nodes hide them, and are held back by the
  // registers and the unknown links' extra loads instead (node_launch). FP32 deviations, us per step, late / early, full-way and half-way:
  // D3Q19 16^3 18.9 / 16.4 and 24.6 / 16.0, 48^3 (13,000 nodes) 20.9 / 18.4 and 27.0 / 18.1, D4Q33 16^4 (27,000) 36 / 32 and 47 / 32,
  // 24^4 (97,500) 99 / 107 and 117 / 101, 32^4 (239,000) 241 / 326 and 275 / 312.
  using T = typename std::conditional<DEV, float, double>::type;
  const T *__restrict__ src = static_cast<const T *>(a.src);
  T raw[EARLY ? Q : 1];
  float2 ph[EARLY && DEV ? Q : 1];
  double v[Q];
  uint64_t in = 0;  // links whose pull source lies in the box
  int ju = 0;
  auto value = [&](int k, int32_t o) {  // f*_k at o
    return DEV ? fma(a.omega[k], df_value(a.phi_src[o]), (double)src[k * S + o]) : (double)src[k * S + o];
  };
  if (!EARLY && !jets) bnode_prepare<D, KIND>(a, x, nd);
#pragma unroll
  for (int k = 0; k < Q; ++k) {
    bool inside = true;
    int32_t o = site;
#pragma unroll
    for (int i = 0; i < D; ++i) {
      if (L.e[k][i] != 0) {
        const int xs = x[i] - L.e[k][i];
        if (xs < 0 || xs >= a.g.n[i]) inside = false;
        o -= L.e[k][i] * a.g.stride[i];
      }
    }
    if constexpr (EARLY) {
      in |= (uint64_t)inside << k;
      raw[k] = __ldg(src + (inside ? k * S + o : (KIND == 2 ? L.opp[k] * S + site : site)));
      if (DEV) ph[k] = __ldg(a.phi_src + (inside ? o : site));
      v[k] = jets && !inside ? __ldg(rec + ju) : 0.0;
      ju += inside ? 0 : 1;
    } else if (inside) {
      v[k] = value(k, o);
    } else {
      // (one rounding for a record's scale and the half-way difference, as in k_bdata_step)
      const double less = KIND == 1 ? 0.0 : value(L.opp[k], site);
      if (jets) v[k] = KIND == 1 ? a.rec_scale * __ldg(rec + ju++) : fma(a.rec_scale, __ldg(rec + ju++), -less);
      else v[k] = KIND == 1 ? bnode_data<D, KIND>(a, coef, nd, k) : bnode_data<D, KIND>(a, coef, nd, k) - less;
    }
  }
  if constexpr (EARLY) {
    if (!jets) bnode_prepare<D, KIND>(a, x, nd);
#pragma unroll
    for (int k = 0; k < Q; ++k) {
      const bool inside = (in >> k) & 1ull;
      const double there = DEV ? fma(inside ? a.omega[k] : a.omega[L.opp[k]], float_to_double(ph[k].x) + float_to_double(ph[k].y),
                                     float_to_double((float)raw[k]))
                               : (double)raw[k];
      if (inside) {
        v[k] = there;
        continue;
      }
      if (jets) v[k] = KIND == 1 ? a.rec_scale * v[k] : fma(a.rec_scale, v[k], -there);
      else v[k] = KIND == 1 ? bnode_data<D, KIND>(a, coef, nd, k) : bnode_data<D, KIND>(a, coef, nd, k) - there;
    }
  }
  // collision, as in the bulk: phi = sum_k f_k, f*_k = (1 - s) f_k + omega_k (s phi + dt R)
  const double phi = DEV ? split_moment_sum<Q, kNodeFixedTerms<Q>>(v) : fixed_moment_sum<Q, 0>(v);
  const double psi = fma(a.s, phi, a.dt * (a.Rfield ? __ldg(a.Rfield + site) : a.R));
  const bool s2 = a.s == 2.0;
  if (DEV) {
    float *gdst = static_cast<float *>(a.dst);
#pragma unroll
    for (int k = 0; k < Q; ++k) {
      const double fs = s2 ? fma(a.omega[k], psi, -v[k]) : fma(a.omega[k], psi, a.oms * v[k]);
      gdst[k * S + site] = (float)fma(-a.omega[k], phi, fs);
    }
    a.phi_dst[site] = df_split(phi);
  } else {
    double *fdst = static_cast<double *>(a.dst);
#pragma unroll
    for (int k = 0; k < Q; ++k)
      fdst[k * S + site] = s2 ? fma(a.omega[k], psi, -v[k]) : fma(a.omega[k], psi, a.oms * v[k]);
  }
}

// Records of the boundary data from jets of phi (lhe_lbm_set_boundary_jet): for every boundary node
// and unknown link k (in the order of k), with c = c e_k,
//   full-way, jet at the node and t + dt (Eq. (bun1)):
//     order 1: omega_k phi;  order 3: omega_k [phi - (dt/2)(c.grad + d_t) phi] + (dt/2) omega_k R;
//     order 4: order 3 + omega_k (dt^3/24) (c.grad + d_t)^3 phi
//   half-way, jet at x_b = x - c dt/2 and t (Eq. (bun2) without -f*_kbar), w+- = omega_k +- omega_kbar:
//     w+ phi + [P >= 2] w+ (dt/2)(phi_t + R) - [P >= 3] (w+ (dt^2/8) cc:grad^2 phi + w- (dt^2/4) c.grad phi_t)
//     - [P >= 4] (w+ (dt^3/16) cc:grad^2 phi_t + w+ (dt^3/24) phi_ttt + w- (dt^3/8) c.grad phi_tt).
// R is the source at the node (the per-site field of the step, when there is one).
// A jet holds every derivative of order <= 3 in (t, x_1..x_d); J.i3[a*36 + b*6 + e] and
// J.i2[a*6 + b] give the position of the derivative in the variables a, b(, e) (0: t, i: x_i), in
// any order. One thread per record (links[r]: the record's boundary node and link), so that a node's links, up to 40
// dependent chains of up to 27 terms, run side by side: with a thread per node these chains were the whole
// time of small boxes (D2Q9 48 x 40, 172 nodes, 516 records: 27.5 -> 8 us). The sums keep their order of terms.
struct JetTables {
  int16_t i3[216];
  int16_t i2[36];
  int8_t e[kMaxQ * kMaxD];
};

template <int D, int KIND>
__global__ void __launch_bounds__(64) k_jet_records(const BoundaryArgs a, const int2 *__restrict__ links, int64_t nrec,
                                                    const double *__restrict__ jet, const JetTables T,
                                                    double *__restrict__ rec) {
  constexpr int JL = (D + 4) * (D + 3) * (D + 2) / 6;
  __shared__ JetTables J;  // links differ within a warp: the parameter bank would serialise
  for (int i = threadIdx.x; i < (int)(sizeof(JetTables) / 2); i += blockDim.x)
    reinterpret_cast<int16_t *>(&J)[i] = reinterpret_cast<const int16_t *>(&T)[i];
  __syncthreads();
  pdl_wait();
  const int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (r >= nrec) return;
  const int2 nk = __ldg(links + r);
  const int k = nk.y, P = a.order;
  const double dt = a.dt;
  const double R = a.Rfield ? a.Rfield[a.sites[nk.x]] : a.R;  // the source at the node
  const double *__restrict__ j = jet + (size_t)(KIND == 1 ? nk.x : r) * JL;
  double w[D + 1];  // weights of the variables in (d_t + c.grad): 1 for t, c_i for x_i
  int var[3] = {0, 0, 0}, nv = 1;  // the variables of non-zero weight, t first
  w[0] = 1.0;
#pragma unroll
  for (int i = 0; i < D; ++i) {
    const int e = J.e[k * D + i];
    w[i + 1] = a.c * e;
    if (e != 0) {
      if (nv == 1) var[1] = i + 1;
      else var[2] = i + 1;
      ++nv;
    }
  }
  double val;
  if (KIND == 1) {
    const double wk = a.omega[k];
    val = wk * j[0];
    if (P >= 3) {
      double d1 = 0.0;
#pragma unroll
      for (int v = 0; v <= D; ++v) d1 += w[v] * j[1 + v];
      val = wk * (j[0] - 0.5 * dt * d1) + 0.5 * dt * wk * R;
    }
    if (P >= 4) {
      double wv[3] = {1.0, 0.0, 0.0};
#pragma unroll
      for (int i = 1; i < 3; ++i) wv[i] = i < nv ? a.c * J.e[k * D + var[i] - 1] : 0.0;
      double d3 = 0.0;
#pragma unroll
      for (int p0 = 0; p0 < 3; ++p0)
#pragma unroll
        for (int p1 = 0; p1 < 3; ++p1)
#pragma unroll
          for (int p2 = 0; p2 < 3; ++p2)
            if (p0 < nv && p1 < nv && p2 < nv) {
              const double ww = wv[p0] * wv[p1] * wv[p2];
              d3 += ww * j[J.i3[var[p0] * 36 + var[p1] * 6 + var[p2]]];
            }
      val += wk * dt * dt * dt / 24.0 * d3;
    }
  } else {
    const int kb = a.kbar[k];
    const double wp = a.omega[k] + a.omega[kb], wm = a.omega[k] - a.omega[kb];
    val = wp * j[0];
    if (P >= 2) val += 0.5 * dt * wp * (j[1] + R);
    if (P >= 3) {
      double cch = 0.0, cgt = 0.0;
#pragma unroll
      for (int p0 = 1; p0 <= D; ++p0) {
        cgt += w[p0] * j[J.i2[p0 * 6]];
#pragma unroll
        for (int p1 = 1; p1 <= D; ++p1) cch += w[p0] * w[p1] * j[J.i2[p0 * 6 + p1]];
      }
      val -= dt * dt / 8.0 * wp * cch + dt * dt / 4.0 * wm * cgt;
    }
    if (P >= 4) {
      double ccht = 0.0, cgtt = 0.0;
#pragma unroll
      for (int p0 = 1; p0 <= D; ++p0) {
        cgtt += w[p0] * j[J.i3[p0 * 36]];
#pragma unroll
        for (int p1 = 1; p1 <= D; ++p1) ccht += w[p0] * w[p1] * j[J.i3[p0 * 36 + p1 * 6]];
      }
      val -= dt * dt * dt / 16.0 * wp * ccht + dt * dt * dt / 24.0 * wp * j[J.i3[0]] + dt * dt * dt / 8.0 * wm * cgtt;
    }
  }
  rec[a.rmap ? a.rmap[r] : r] = val;  // node-major, or in the order of the dense entries
}

template <int D>
static cudaError_t jet_records_d(int kind, const BoundaryArgs &a, const int2 *links, int64_t nrec, const double *jet,
                                 const JetTables &T, double *rec, cudaStream_t st) {
  if (nrec <= 0) return cudaSuccess;
  const unsigned blocks = (unsigned)((nrec + 63) / 64);
  return launch_kernel(kind == 1 ? k_jet_records<D, 1> : k_jet_records<D, 2>, blocks, 64, 0, st, a.pdl != 0, a, links, nrec,
                       jet, T, rec);
}

cudaError_t launch_jet_records(int d, int kind, const BoundaryArgs &a, const int2 *links, int64_t nrec, const int32_t *e,
                               const double *jet, const int16_t *jidx, double *rec, cudaStream_t st) {
  JetTables T{};
  for (int i = 0; i < 216; ++i) T.i3[i] = jidx[i];
  for (int i = 0; i < 36; ++i) T.i2[i] = jidx[216 + i];
  for (int i = 0; i < (2 * d * d + 1) * d; ++i) T.e[i] = (int8_t)e[i];
  switch (d) {
    case 1: return jet_records_d<1>(kind, a, links, nrec, jet, T, rec, st);
    case 2: return jet_records_d<2>(kind, a, links, nrec, jet, T, rec, st);
    case 3: return jet_records_d<3>(kind, a, links, nrec, jet, T, rec, st);
    case 4: return jet_records_d<4>(kind, a, links, nrec, jet, T, rec, st);
    case 5: return jet_records_d<5>(kind, a, links, nrec, jet, T, rec, st);
    default: return cudaErrorInvalidValue;
  }
}

// Cotangent of the jets of one Dirichlet step (lhe_lbm_adjoint_jet_grad): the transpose of
// k_jet_records. a.src holds the adjoint state rho_k(x) = omega_k dL/df_k(x) of the pre-collision
// populations that the step produced, so the cotangent of an unknown population's value is
// rho_k / omega_k (the R terms and the half-way -f*_kbar do not depend on the jets). The records are linear in
// the jets with weights that depend on the link alone: w[k JL + q] is the weight of derivative q in the record of link k, over
// omega_k (formed once per handle). Full-way: one row per boundary node, summed over its unknown links;
// half-way: one row per unknown population. One thread per entry of the result, so that the weights and the
// result are read and written contiguously (a thread per node walked its links and up to 84 derivatives
// in turn: D2Q9 48 x 40 26.3 -> 4.8 us). FP32 deviations (DEV): rho_k = omega_k W + eps_k.
template <int D, int KIND, bool DEV>
__global__ void __launch_bounds__(128) k_jet_grad(const BoundaryArgs a, const int2 *__restrict__ links, int64_t nrec,
                                                  const double *__restrict__ w, double *__restrict__ out) {
  constexpr int JL = (D + 4) * (D + 3) * (D + 2) / 6;
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t row = t / JL;
  const int q = (int)(t - row * JL);
  pdl_wait();
  if (row >= (KIND == 1 ? a.nsites : nrec)) return;
  const int64_t S = a.g.S;
  const int64_t r0 = KIND == 1 ? a.roff[row] : row;
  const int64_t r1 = KIND == 1 ? (row + 1 < a.nsites ? a.roff[row + 1] : nrec) : row + 1;
  double acc = 0.0;
  for (int64_t r = r0; r < r1; ++r) {
    const int2 nk = __ldg(links + r);
    const int32_t site = a.sites[nk.x];
    const double rk = DEV ? fma(a.omega[nk.y], df_value(a.phi_src[site]), (double)static_cast<const float *>(a.src)[nk.y * S + site])
                          : static_cast<const double *>(a.src)[nk.y * S + site];
    acc = fma(__ldg(w + nk.y * JL + q), rk, acc);
  }
  out[t] = acc;
}

template <int D>
static cudaError_t jet_grad_d(int kind, bool dev, const BoundaryArgs &a, const int2 *links, int64_t nrec,
                              const double *w, double *out, cudaStream_t st) {
  if (nrec <= 0) return cudaSuccess;
  constexpr int64_t JL = (D + 4) * (D + 3) * (D + 2) / 6;
  const unsigned blocks = (unsigned)(((kind == 1 ? a.nsites : nrec) * JL + 127) / 128);
  auto kernel = kind == 1 ? (dev ? k_jet_grad<D, 1, true> : k_jet_grad<D, 1, false>)
                          : (dev ? k_jet_grad<D, 2, true> : k_jet_grad<D, 2, false>);
  return launch_kernel(kernel, blocks, 128, 0, st, a.pdl != 0, a, links, nrec, w, out);
}

cudaError_t launch_jet_grad(int d, int kind, bool dev, const BoundaryArgs &a, const int2 *links, int64_t nrec,
                            const double *w, double *out, cudaStream_t st) {
  switch (d) {
    case 1: return jet_grad_d<1>(kind, dev, a, links, nrec, w, out, st);
    case 2: return jet_grad_d<2>(kind, dev, a, links, nrec, w, out, st);
    case 3: return jet_grad_d<3>(kind, dev, a, links, nrec, w, out, st);
    case 4: return jet_grad_d<4>(kind, dev, a, links, nrec, w, out, st);
    case 5: return jet_grad_d<5>(kind, dev, a, links, nrec, w, out, st);
    default: return cudaErrorInvalidValue;
  }
}

// Adjoint of a Dirichlet step at the boundary nodes (FP64), in the weighted variable
// rho_k(x) = omega_k dL/df_k(x) of the pre-collision populations (the interior nodes use the bulk
// adjoint kernel). Transposing the pull: mu_j(x) = omega_j dL/df*_j(x) = rho_j(x + e_j) where
// x + e_j is a node of the box. Where it is not, the post-collision population leaves the box: in
// the full-way scheme it feeds nothing (Eq. (bun1) sets the unknown population at the far side
// from the boundary data alone), in the half-way scheme it is the -f*_j(x) of the unknown
// f_jbar(x) = -f*_j(x) + B (Eq. (bun2)), so mu_j(x) = -(omega_j / omega_jbar) rho_jbar(x). Then
// rho_k <- (1 - s) mu_k + s omega_k sum_j mu_j, as in the bulk. FP32 deviations (DEV): the adjoint state
// is rho_k = omega_k W + eps_k (W a double-float pair, eps in FP32), formed in FP64 here, and the result
// is stored as the forward boundary kernel stores a state: W' = sum_j mu_j, eps'_k = rho'_k - omega_k W'.
template <int D, int KIND, bool DEV, bool EARLY>
__global__ void __launch_bounds__(128) k_adj_boundary(const BoundaryArgs a) {
  constexpr Lattice<D> L{};
  constexpr int Q = Lattice<D>::Q;
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  pdl_wait();
  if (t >= a.nsites) return;
  const int32_t site = a.sites[t];
  const int64_t S = a.g.S;
  int x[D];
  {
    uint32_t r = (uint32_t)site;
#pragma unroll
    for (int i = 0; i < D; ++i) {
      if (i == D - 1) {
        x[i] = (int)r;
      } else {
        const uint32_t q = a.g.dv[i].div(r);
        x[i] = (int)(r - q * (uint32_t)a.g.n[i]);
        r = q;
      }
    }
  }
  using T = typename std::conditional<DEV, float, double>::type;
  const T *__restrict__ src = static_cast<const T *>(a.src);
  // EARLY as in k_boundary: every load first, rho_k at x + e_k, or for a link that leaves the box rho_kbar at the node
  T raw[EARLY ? Q : 1];
  float2 ph[EARLY && DEV ? Q : 1];
  double mu[Q];
  uint64_t in = 0;
  auto rho = [&](int k, int32_t o) {
    return DEV ? fma(a.omega[k], df_value(a.phi_src[o]), (double)src[k * S + o]) : (double)src[k * S + o];
  };
#pragma unroll
  for (int k = 0; k < Q; ++k) {
    bool inside = true;
    int32_t o = site;
#pragma unroll
    for (int i = 0; i < D; ++i) {
      if (L.e[k][i] != 0) {
        const int xs = x[i] + L.e[k][i];
        if (xs < 0 || xs >= a.g.n[i]) inside = false;
        o += L.e[k][i] * a.g.stride[i];
      }
    }
    if constexpr (EARLY) {
      in |= (uint64_t)inside << k;
      raw[k] = __ldg(src + (inside ? k * S + o : L.opp[k] * S + site));
      if (DEV) ph[k] = __ldg(a.phi_src + (inside ? o : site));
    } else {
      if (inside) mu[k] = rho(k, o);
      else mu[k] = KIND == 2 ? -a.wratio[k] * rho(L.opp[k], site) : 0.0;
    }
  }
  if constexpr (EARLY) {
#pragma unroll
    for (int k = 0; k < Q; ++k) {
      const bool inside = (in >> k) & 1ull;
      const double there = DEV ? fma(inside ? a.omega[k] : a.omega[L.opp[k]], float_to_double(ph[k].x) + float_to_double(ph[k].y),
                                     float_to_double((float)raw[k]))
                               : (double)raw[k];
      mu[k] = inside ? there : (KIND == 2 ? -a.wratio[k] * there : 0.0);
    }
  }
  if (DEV) {
    const double M = fixed_moment_sum<Q, 0, false>(mu);
    const double psi = a.s * M;
    float *edst = static_cast<float *>(a.dst);
#pragma unroll
    for (int k = 0; k < Q; ++k) {
      const double r = a.s == 2.0 ? fma(a.omega[k], psi, -mu[k]) : fma(a.omega[k], psi, a.oms * mu[k]);
      edst[k * S + site] = (float)fma(-a.omega[k], M, r);
    }
    a.phi_dst[site] = df_split(M);
    return;
  }
  double *__restrict__ dst = static_cast<double *>(a.dst);
  if (a.s == 2.0) {
    const double psi = fixed_moment_sum<Q, 1, false>(mu);  // 2 sum_j mu_j
#pragma unroll
    for (int k = 0; k < Q; ++k) dst[k * S + site] = fma(a.omega[k], psi, -mu[k]);
  } else {
    const double psi = a.s * fixed_moment_sum<Q, 0, false>(mu);
#pragma unroll
    for (int k = 0; k < Q; ++k) dst[k * S + site] = fma(a.omega[k], psi, a.oms * mu[k]);
  }
}

// FP32 deviations: boundary nodes up to which the kernels issue every load first (EARLY, k_boundary): one wave of CTAs of 64
// threads, as many an SM as the registers allow (k_boundary 80, 168, 254 and 255 for D = 2 .. 5, k_adj_boundary 72, 87, 142 and 216).
template <int D>
static int64_t early_nodes(int sms, bool adjoint) {
  constexpr int ctas[2][6] = {{0, 32, 12, 6, 4, 4}, {0, 32, 14, 11, 7, 4}};
  return (int64_t)sms * ctas[adjoint][D] * 64;
}

// Threads per CTA of the boundary-node kernels: a node is ~150 FP64 operations behind several dependent loads, so few
// nodes are spread over as many SMs as there are (128 threads: D3Q19 32^3, 5768 nodes, on 46 of 152 SMs).
static int boundary_threads(int64_t nodes, int sms) {
  return nodes <= (int64_t)sms * 4 * 32 ? 32 : (nodes <= (int64_t)sms * 8 * 64 ? 64 : 128);
}

// How the kernels of one box are launched. FP32 deviations, us per step before there was an early form / early up to 40,000
// nodes, more than a wave in D4Q33, and beside the rows' last wave / now (lhe_step_dev.cu), full-way and its adjoint:
// D4Q33 18^4 (39,440 nodes) 50 / 63 / 45 and 41 / 33 / 30, 19^4 56 / 62 / 50 and 41 / 47 / 32, 22^4 (74,256) 76 / 78 / 73 and
// 56 / 60 / 52, 24^4 (97,520) 109 / 106 / 106 and 79 / 76 / 76; D3Q19 90^3 (47,528) 55 / 49 / 49 and 45 / 40 / 40.
struct NodeLaunch {
  bool early;
  int threads;
};

template <int D>
static NodeLaunch node_launch(bool dev, bool adjoint, const BoundaryArgs &a) {
  const int threads = boundary_threads(a.nsites, a.sms);
  if (!dev) return {false, adjoint ? threads : 128};  // (k_boundary)
  return a.nsites <= early_nodes<D>(a.sms, adjoint) ? NodeLaunch{true, std::min(threads, 64)} : NodeLaunch{false, threads};
}

template <int D>
static cudaError_t adj_boundary_d(int kind, bool dev, const BoundaryArgs &a, cudaStream_t st) {
  if (a.nsites <= 0) return cudaSuccess;
  const NodeLaunch n = node_launch<D>(dev, true, a);
  const unsigned blocks = (unsigned)((a.nsites + n.threads - 1) / n.threads);
  auto kernel = !dev ? (kind == 1 ? k_adj_boundary<D, 1, false, false> : k_adj_boundary<D, 2, false, false>)
                : n.early              ? (kind == 1 ? k_adj_boundary<D, 1, true, true> : k_adj_boundary<D, 2, true, true>)
                                          : (kind == 1 ? k_adj_boundary<D, 1, true, false> : k_adj_boundary<D, 2, true, false>);
  return launch_kernel(kernel, blocks, n.threads, 0, st, a.pdl != 0, a);
}

cudaError_t launch_adjoint_boundary(int d, int kind, bool dev, const BoundaryArgs &a, cudaStream_t st) {
  switch (d) {
    case 1: return adj_boundary_d<1>(kind, dev, a, st);
    case 2: return adj_boundary_d<2>(kind, dev, a, st);
    case 3: return adj_boundary_d<3>(kind, dev, a, st);
    case 4: return adj_boundary_d<4>(kind, dev, a, st);
    case 5: return adj_boundary_d<5>(kind, dev, a, st);
    default: return cudaErrorInvalidValue;
  }
}

template <int D>
static cudaError_t boundary_d(int kind, bool dev, const BoundaryArgs &a, cudaStream_t st) {
  if (a.nsites <= 0) return cudaSuccess;
  const NodeLaunch n = node_launch<D>(dev, false, a);
  const unsigned blocks = (unsigned)((a.nsites + n.threads - 1) / n.threads);
  auto kernel = !dev ? (kind == 1 ? k_boundary<D, 1, false, false> : k_boundary<D, 2, false, false>)
                : n.early              ? (kind == 1 ? k_boundary<D, 1, true, true> : k_boundary<D, 2, true, true>)
                                          : (kind == 1 ? k_boundary<D, 1, true, false> : k_boundary<D, 2, true, false>);
  const size_t smem = a.rec || !dev ? 0 : sizeof(double) * 2 * (size_t)(a.nmodes + 1) * Lattice<D>::Q;
  return launch_kernel(kernel, blocks, n.threads, smem, st, a.pdl != 0, a);
}

cudaError_t launch_boundary(int d, int kind, bool dev, const BoundaryArgs &a, cudaStream_t st) {
  switch (d) {
    case 1: return boundary_d<1>(kind, dev, a, st);
    case 2: return boundary_d<2>(kind, dev, a, st);
    case 3: return boundary_d<3>(kind, dev, a, st);
    case 4: return boundary_d<4>(kind, dev, a, st);
    case 5: return boundary_d<5>(kind, dev, a, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace lhe
