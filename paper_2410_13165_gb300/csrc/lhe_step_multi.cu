// lhe_step_multi.cu -- several steps of a small or 32-bit periodic box (1D to 3D) in one launch.
//
// A step of such a grid is bound by its launch (~1.8 us from one step kernel to the next) and, in 32 bits, by L2,
// not by arithmetic. A CTA owns a tile of nodes and takes it through H steps in shared memory: the first
// step pulls from global memory and covers the tile plus H - 1 rings of nodes, each further step
// one ring less, pulled from the shared-memory copy of the step before (two copies in turn), and the last
// writes the tile. The rings are computed by every tile that needs them, so that no CTA waits for another. The arithmetic
// per node is that of k_step_fp64 / k_step_dev, in the same order: the same bits. plan_multi (below) picks the tile and
// H from the grid, or none.
#include <algorithm>

#include "lhe_internal.h"
#include "lhe_sites.cuh"

namespace lhe {

namespace {

constexpr int kModeGeneral = 0, kModeS2 = 1;  // collision forms: s = 2, or by the step's constants

__device__ __forceinline__ int wrap_once(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

}  // namespace

// Where a CTA's tile lies and how the nodes of a step are numbered.
template <int D>
struct MultiTile {
  int x0[D], n[D], own[D], stride[D];  // origin of the first region, box, the tile's own nodes, strides within a copy
  __device__ __forceinline__ explicit MultiTile(const StepArgs &a, const MultiPlan &p) {
    int b = blockIdx.x, st = 1;
#pragma unroll
    for (int i = 0; i < D; ++i) {
      const int q = i == D - 1 ? 0 : b / p.tiles[i];
      const int first = (i == D - 1 ? b : b - q * p.tiles[i]) * p.t[i];
      b = q;
      n[i] = a.g.n[i];
      x0[i] = first - (p.H - 1);
      own[i] = min(p.t[i], n[i] - first);  // (a last tile may stick out of the box: the nodes beyond are another tile's)
      stride[i] = st;
      st *= p.w[i];
    }
  }
  // place of a node of the region in a copy, and in the box
  __device__ __forceinline__ int at(const int (&i)[D]) const {
    int c = 0;
#pragma unroll
    for (int q = 0; q < D; ++q) c += i[q] * stride[q];
    return c;
  }
  __device__ __forceinline__ int32_t site(const Geom &g, const int (&i)[D], int (&x)[D]) const {
    int32_t s = 0;
#pragma unroll
    for (int q = 0; q < D; ++q) {
      x[q] = wrap_once(x0[q] + i[q], n[q]);
      s += x[q] * g.stride[q];
    }
    return s;
  }
  __device__ __forceinline__ int32_t site(const Geom &g, const int (&i)[D]) const {
    int x[D];
    return site(g, i, x);
  }
  // place among the tile's own nodes, or -1
  __device__ __forceinline__ int mine(const MultiPlan &p, const int (&i)[D]) const {
    int c = 0, st = 1;
    bool in = true;
#pragma unroll
    for (int q = 0; q < D; ++q) {
      const int l = i[q] - (p.H - 1);
      in = in && l >= 0 && l < own[q];
      c += l * st;
      st *= p.t[q];
    }
    return in ? c : -1;
  }
};

// t = r w + rest for 0 <= t < 2^13, inv ~ 1 / w: the product is within 2^-21 t / w of (t + 1/2) / w, which is at
// least 1 / (2 w) from an integer.
__device__ __forceinline__ int row_of(int t, float inv) { return (int)(((float)t + 0.5f) * inv); }

// Calls node(i) for the nodes i of step j (1 .. H) of the region, one after another per thread.
template <int D, class F>
__device__ __forceinline__ void multi_nodes(const MultiPlan &p, int j, F node) {
  const int o = j - 1;
  int w[D], nodes = 1;
#pragma unroll
  for (int q = 0; q < D; ++q) {
    w[q] = p.w[q] - 2 * o;
    nodes *= w[q];
  }
  const float inv0 = __fdividef(1.0f, (float)w[0]), inv1 = __fdividef(1.0f, (float)w[D > 1 ? 1 : 0]);
  for (int t = threadIdx.x; t < nodes; t += blockDim.x) {
    int i[D];
    if constexpr (D == 1) {
      i[0] = t + o;
    } else {
      const int r = row_of(t, inv0);
      i[0] = t - r * w[0] + o;
      if constexpr (D == 2) {
        i[1] = r + o;
      } else {
        const int z = row_of(r, inv1);
        i[1] = r - z * w[1] + o;
        i[2] = z + o;
      }
    }
    node(i);
  }
}

// The copies hold the nodes' populations together (Q consecutive values a node): a neighbour's address is one
// of 3^(D-1) row addresses plus a constant, and Q is odd, so that the lanes of a warp fall on different banks.
// (With population-major copies each access took its own address arithmetic: 329 instructions a D2Q9 node and
// step in 32 bits, twice the arithmetic's.)
template <int D, bool ADJ>
__device__ __forceinline__ int pull_row(const MultiTile<D> &tile, int k) {
  constexpr Lattice<D> L{};
  int r = 0;
#pragma unroll
  for (int q = 1; q < D; ++q) r += (ADJ ? L.e[k][q] : -L.e[k][q]) * tile.stride[q];
  return r;
}

template <int D, bool ADJ, class T>
__device__ __forceinline__ void pull_shared(const T *__restrict__ from, int c, const MultiTile<D> &tile, T (&f)[Lattice<D>::Q]) {
  constexpr Lattice<D> L{};
  constexpr int Q = Lattice<D>::Q;
#pragma unroll
  for (int k = 0; k < Q; ++k) f[k] = from[(c + pull_row<D, ADJ>(tile, k)) * Q + (ADJ ? L.e[k][0] : -L.e[k][0]) * Q + k];
}

template <int D, bool ADJ, int MODE>
__global__ void __launch_bounds__(multi_threads(D)) k_multi_fp64(const __grid_constant__ MultiArgs m) {
  constexpr Lattice<D> L{};
  constexpr int Q = Lattice<D>::Q;
  extern __shared__ __align__(16) unsigned char smem[];
  const StepArgs &a = m.a;
  const MultiPlan &p = m.p;
  const int H = p.H, N = p.nodes;
  double *buf = reinterpret_cast<double *>(smem);  // p.copies of N x Q
  double *acc = buf + p.copies * N * Q;            // adjoint: dL/dR of the tile
  const MultiTile<D> tile(a, p);
  const int64_t S = a.g.S;
  // the collision of step o + 1 at node i: psi from the pulled populations, dL/dR on the way
  auto collide = [&](const double (&f)[Q], int o, const int (&i)[D]) {
    double psi;
    if (ADJ) {
      const double w2 = MODE == kModeS2 ? fixed_moment_sum<Q, 1>(f) : fixed_moment_sum<Q, 0>(f);
      psi = MODE == kModeS2 ? w2 : m.sig[o] * w2;
      const int c = a.gR ? tile.mine(p, i) : -1;
      if (c >= 0) {
        const int32_t site = tile.site(a.g, i);
        const double g = fma(MODE == kModeS2 ? a.half_dt : m.gsc[o], w2, o == 0 ? a.gR[site] : acc[c]);
        if (o == H - 1) a.gR[site] = g;
        else acc[c] = g;
      }
    } else {
      const double R = a.Rfield ? __ldg(a.Rfield + tile.site(a.g, i)) : 0.0;
      if (MODE == kModeS2) psi = fixed_moment_sum<Q, 1>(f) + (a.Rfield ? a.dt * R : a.dtR);
      else psi = fma(m.sig[o], fixed_moment_sum<Q, 0>(f), a.Rfield ? m.rho_dt[o] * R : m.rho_dtR[o]);
    }
    return psi;
  };
  auto out = [&](double f, double psi, int o, int k) {
    if (MODE == kModeS2) return fma(a.omega[k], psi, -f);
    return m.collide[o] == kCollideScaled ? fma(a.omega[k], psi, f) : fma(a.omega[k], psi, m.mu[o] * f);
  };
  pdl_wait();
  const double *__restrict__ src = static_cast<const double *>(a.src);
  multi_nodes<D>(p, 1, [&](const int (&i)[D]) {
    int x[D];
    const int32_t site = tile.site(a.g, i, x);
    int32_t om[D], op[D];
    axis_offsets<D, false>(a.g, x, om, op);
    double f[Q];
#pragma unroll
    for (int k = 0; k < Q; ++k) f[k] = __ldg(src + k * S + source_site<D, ADJ>(L, k, site, om, op));
    const double psi = collide(f, 0, i);
    double *to = buf + tile.at(i) * Q;
#pragma unroll
    for (int k = 0; k < Q; ++k) to[k] = out(f[k], psi, 0, k);
  });
  __syncthreads();
  int cur = 0;
  for (int j = 2; j < H; ++j) {
    const double *from = buf + cur * N * Q;
    double *dst = buf + (cur ^ 1) * N * Q;
    multi_nodes<D>(p, j, [&](const int (&i)[D]) {
      const int c = tile.at(i);
      double f[Q];
      pull_shared<D, ADJ>(from, c, tile, f);
      const double psi = collide(f, j - 1, i);
      double *to = dst + c * Q;
#pragma unroll
      for (int k = 0; k < Q; ++k) to[k] = out(f[k], psi, j - 1, k);
    });
    __syncthreads();
    cur ^= 1;
  }
  const double *from = buf + cur * N * Q;
  double *__restrict__ dst = static_cast<double *>(a.dst);
  multi_nodes<D>(p, H, [&](const int (&i)[D]) {
    if (tile.mine(p, i) < 0) return;
    const int32_t site = tile.site(a.g, i);
    double f[Q];
    pull_shared<D, ADJ>(from, tile.at(i), tile, f);
    const double psi = collide(f, H - 1, i);
#pragma unroll
    for (int k = 0; k < Q; ++k) dst[k * S + site] = out(f[k], psi, H - 1, k);
  });
}

template <int D, bool ADJ, bool S2>
__global__ void __launch_bounds__(multi_threads(D)) k_multi_dev(const __grid_constant__ MultiArgs m) {
  constexpr Lattice<D> L{};
  constexpr int Q = Lattice<D>::Q;
  extern __shared__ __align__(16) unsigned char smem[];
  const StepArgs &a = m.a;
  const MultiPlan &p = m.p;
  const int H = p.H, N = p.nodes;
  double *acc = reinterpret_cast<double *>(smem);                         // adjoint: dL/dR of the tile
  float2 *bphi = reinterpret_cast<float2 *>(acc + (ADJ ? p.own : 0));      // p.copies of N
  float *buf = reinterpret_cast<float *>(bphi + p.copies * N);            // p.copies of N x Q
  const MultiTile<D> tile(a, p);
  const int64_t S = a.g.S;
  const bool field = !ADJ && a.Rfield != nullptr;
  const float oms = (float)a.oms;
  // step o + 1 at node i from the pulled deviations and the differences of phi: the new pair of phi; gk becomes the new deviations
  auto collide = [&](float (&gk)[Q], const float (&dl)[Q], float2 p0, int o, const int (&i)[D]) {
    float accw = 0.0f, accg = 0.0f;
#pragma unroll
    for (int k = 0; k < Q; ++k) {
      accw = fmaf(a.omega_f[k], dl[k], accw);
      accg += gk[k];
    }
    const float Delta = accw + accg;
    const float2 pn = df_add(p0.x, p0.y + Delta);
    float dtR = 0.0f;
    if (ADJ) {
      const int q = a.gR ? tile.mine(p, i) : -1;
      if (q >= 0) {
        const int32_t site = tile.site(a.g, i);
        const double g = fma(a.dt, df_value(pn), o == 0 ? a.gR[site] : acc[q]);
        if (o == H - 1) a.gR[site] = g;
        else acc[q] = g;
      }
    } else if (field) {
      dtR = (float)(a.dt * __ldg(a.Rfield + tile.site(a.g, i)));
    }
#pragma unroll
    for (int k = 0; k < Q; ++k) {
      const float r = fmaf(a.omega_f[k], dl[k] - Delta, gk[k]);
      const float src_k = ADJ ? 0.0f : (field ? a.omega_f[k] * dtR : a.dtwR_f[k]);
      gk[k] = S2 ? (src_k - r) : fmaf(oms, r, src_k);
    }
    return pn;
  };
  // pulled values of a node from the shared copies
  auto pull = [&](const float *from, const float2 *pf, int c, float (&gk)[Q], float (&dl)[Q]) {
    pull_shared<D, ADJ>(from, c, tile, gk);
    const float2 p0 = pf[c];
    dl[0] = 0.0f;
#pragma unroll
    for (int k = 1; k < Q; ++k) {
      const float2 pk = pf[(c + pull_row<D, ADJ>(tile, k)) + (ADJ ? L.e[k][0] : -L.e[k][0])];
      dl[k] = (pk.x - p0.x) + (pk.y - p0.y);
    }
    return p0;
  };
  pdl_wait();
  const float *__restrict__ src = static_cast<const float *>(a.src);
  const float2 *__restrict__ phis = a.phi_src;
  multi_nodes<D>(p, 1, [&](const int (&i)[D]) {
    int x[D];
    const int32_t site = tile.site(a.g, i, x);
    int32_t om[D], op[D];
    axis_offsets<D, false>(a.g, x, om, op);
    const float2 p0 = __ldg(phis + site);
    float gk[Q], dl[Q];
#pragma unroll
    for (int k = 0; k < Q; ++k) {
      const int32_t q = source_site<D, ADJ>(L, k, site, om, op);
      gk[k] = __ldg(src + k * S + q);
      dl[k] = 0.0f;
      if (k > 0) {
        const float2 pk = __ldg(phis + q);
        dl[k] = (pk.x - p0.x) + (pk.y - p0.y);
      }
    }
    const int c = tile.at(i);
    bphi[c] = collide(gk, dl, p0, 0, i);
#pragma unroll
    for (int k = 0; k < Q; ++k) buf[c * Q + k] = gk[k];
  });
  __syncthreads();
  int cur = 0;
  for (int j = 2; j < H; ++j) {
    const float *from = buf + cur * N * Q;
    float *to = buf + (cur ^ 1) * N * Q;
    const float2 *pf = bphi + cur * N;
    float2 *pt = bphi + (cur ^ 1) * N;
    multi_nodes<D>(p, j, [&](const int (&i)[D]) {
      const int c = tile.at(i);
      float gk[Q], dl[Q];
      const float2 p0 = pull(from, pf, c, gk, dl);
      pt[c] = collide(gk, dl, p0, j - 1, i);
#pragma unroll
      for (int k = 0; k < Q; ++k) to[c * Q + k] = gk[k];
    });
    __syncthreads();
    cur ^= 1;
  }
  const float *from = buf + cur * N * Q;
  const float2 *pf = bphi + cur * N;
  float *__restrict__ dst = static_cast<float *>(a.dst);
  multi_nodes<D>(p, H, [&](const int (&i)[D]) {
    if (tile.mine(p, i) < 0) return;
    const int32_t site = tile.site(a.g, i);
    float gk[Q], dl[Q];
    const float2 p0 = pull(from, pf, tile.at(i), gk, dl);
    a.phi_dst[site] = collide(gk, dl, p0, H - 1, i);
#pragma unroll
    for (int k = 0; k < Q; ++k) dst[k * S + site] = gk[k];
  });
}

namespace {

// H steps over tiles of t nodes, a thread per node of the first region up to `most`.
MultiPlan make_multi(const Geom &g, bool dev, int tx, int ty, int tz, int H, int most) {
  MultiPlan p;
  const int t[3] = {tx, g.d > 1 ? ty : 1, g.d > 2 ? tz : 1};
  p.H = H;
  p.copies = H > 2 ? 2 : 1;
  p.nodes = p.own = p.grid = 1;
  for (int i = 0; i < 3; ++i) {
    p.t[i] = t[i];
    p.w[i] = t[i] + (i < g.d ? 2 * (H - 1) : 0);
    p.tiles[i] = i < g.d ? (g.n[i] + t[i] - 1) / t[i] : 1;
    p.nodes *= p.w[i];
    p.own *= t[i];
    p.grid *= p.tiles[i];
  }
  p.threads = std::min(most, (p.nodes + 31) / 32 * 32);
  const size_t Q = 2 * g.d * g.d + 1;
  p.smem = 8 * (size_t)p.own + p.copies * (size_t)p.nodes * (dev ? 4 * Q + 8 : 8 * Q);
  return p;
}

template <int D>
const void *multi_kernel_dev(bool adjoint, bool s2) {
  return adjoint ? (s2 ? (const void *)k_multi_dev<D, true, true> : (const void *)k_multi_dev<D, true, false>)
                 : (s2 ? (const void *)k_multi_dev<D, false, true> : (const void *)k_multi_dev<D, false, false>);
}

template <int D>
const void *multi_kernel_fp64(bool adjoint, bool s2) {
  return adjoint ? (s2 ? (const void *)k_multi_fp64<D, true, kModeS2> : (const void *)k_multi_fp64<D, true, kModeGeneral>)
                 : (s2 ? (const void *)k_multi_fp64<D, false, kModeS2> : (const void *)k_multi_fp64<D, false, kModeGeneral>);
}

const void *multi_kernel(int d, bool dev, bool adjoint, bool s2) {
  if (!dev) return d == 1 ? multi_kernel_fp64<1>(adjoint, s2) : multi_kernel_fp64<2>(adjoint, s2);
  return d == 1 ? multi_kernel_dev<1>(adjoint, s2) : (d == 2 ? multi_kernel_dev<2>(adjoint, s2) : multi_kernel_dev<3>(adjoint, s2));
}

}  // namespace

// The plan of a periodic box, or none (one step per launch). Small grids: one tile per SM, the one with the
// smallest first region, a thread per node of it, and as many steps as pay for the rings that the tiles share
// with their neighbours: FP64 is held back by the FP64 pipe (~2 operations per clock per SM, 10 a node), so that H
// falls with the tile's size, and none pays from ~260^2 on. 32 bits pay further on, where a launch is short beside a
// step, and again from 1.5 M nodes, where the two states leave L2 and H steps pass memory once.
// us per step, one step per launch / this rule (forward):
//   FP64 D2Q9 16^2 1.90 / 1.31, 64^2 2.14 / 1.39, 128^2 2.22 / 1.66, 200^2 3.08 / 2.46, 256^2 3.66 / 3.21, 270 x 260 3.68 / 3.52 with the
//     adjoint 3.52 / 3.69 (not taken), 500 x 333 5.9 / 7.1 (32 x 8, H = 2; not taken); D1Q3 64 1.92 / 0.74, 30000 2.01 / 1.03,
//     10^6 16.4 / 18.4 (not taken)
//   32 bits D2Q9 16^2 1.90 / 0.60, 64^2 1.90 / 0.70, 128^2 1.90 / 0.84, 256^2 2.05 / 1.42, 320^2 2.29 / 2.23, 500 x 333 3.33 / 2.97, 430^2 (756
//     tiles of 32 x 8, one wave is 760) 3.38 / 3.07, 440^2 (770) 3.37 / 3.58, 5000 x 33 (785) 3.38 / 3.66, 560^2 4.53 / 4.82, 700^2 6.05 / 7.01,
//     1000^2 12.1 / 14.1 (none of these taken), 1250^2 23.3 / 19.8, 2048^2 58.7 / 50.5; with tiles of 32 x 16 that stick out of 2 M to
//     3 M nodes by 60 % (100000 x 20) 29.9 / 36.3, 33 % (x 24) 35.5 / 38.9, 14 % (x 28) 40.7 / 41.3 (not taken), 7 % (x 30) 43.4 / 41.9;
//     D1Q3 4096 1.89 / 0.47, 10^5 1.96 / 1.13, 2 10^6 17.1 / 8.3;
//     D3Q19 8^3 1.93 / 1.14, 16^3 1.95 / 1.44, 24^3 1.94 / 1.75, 28^3 2.18 / 2.13 (not taken); FP64 D3Q19 16^3 2.89 / 2.82, 20^3 2.94 / 3.05 (not taken)
bool plan_multi(const Geom &g, bool dev, int sms, MultiPlan &best) {
  best = MultiPlan{};
  if (g.d > 3 || sms <= 0) return false;
  const int64_t S = g.S, share = (S + sms - 1) / sms;  // nodes per SM
  // (a region that wraps around the box once at most)
  auto fits = [&](int tx, int ty, int tz, int H) {
    return tx + H - 1 <= g.n[0] && (g.d < 2 || ty + H - 1 <= g.n[1]) && (g.d < 3 || tz + H - 1 <= g.n[2]);
  };
  // one tile per SM, the smallest first region
  auto search = [&](int H, int step, int most_x, int most_y, int most_z, int64_t most_nodes) {
    int64_t least = INT64_MAX;
    for (int tz = 1; tz <= most_z; ++tz)
      for (int ty = 1; ty <= most_y; ++ty)
        for (int tx = step; tx <= most_x; tx += step) {
          if (!fits(tx, ty, tz, H)) continue;
          const MultiPlan p = make_multi(g, dev, tx, ty, tz, H, multi_threads(g.d));
          if (p.grid > sms || p.nodes > most_nodes || p.nodes >= least || p.smem > (size_t)kMultiMaxSmem) continue;
          least = p.nodes;
          best = p;
        }
  };
  if (g.d == 1) {
    if (!dev && share > 200) return false;
    const int tx = (int)std::min<int64_t>(512, std::max<int64_t>(32, share));
    if (fits(tx, 1, 1, kMultiMaxSteps)) best = make_multi(g, dev, tx, 1, 1, kMultiMaxSteps, 256);
  } else if (g.d == 3) {
    if (dev && S <= 14000) search(S <= 4200 ? 3 : 2, 1, 24, 24, 24, 2048);
  } else if (share <= (dev ? 480 : 440)) {
    search(dev ? (share <= 160 ? 6 : 4) : (share <= 48 ? 4 : (share <= 160 ? 3 : 2)), 4, 64, 64, 1, kMultiThreads);
  } else if (dev && S <= 200000 && fits(32, 8, 1, 3)) {
    best = make_multi(g, dev, 32, 8, 1, 3, 192);
    if (best.grid > 5 * sms) best = MultiPlan{};  // more than one wave (40 KB of shared memory a CTA)
  } else if (dev && S >= 1500000 && fits(32, 16, 1, 2)) {
    best = make_multi(g, dev, 32, 16, 1, 2, 320);
    if ((int64_t)best.grid * best.own > S + S / 10) best = MultiPlan{};  // tiles that stick out compute for nothing
  }
  return best.H > 1;
}

MultiPlan shorter_multi(const Geom &g, bool dev, const MultiPlan &p, int H) {
  return H == p.H ? p : make_multi(g, dev, p.t[0], p.t[1], p.t[2], H, p.threads);
}

cudaError_t prepare_multi(int d, bool dev, const MultiPlan &p) {
  for (int i = 0; i < 4; ++i) {
    const cudaError_t e = cudaFuncSetAttribute(multi_kernel(d, dev, i & 1, i & 2), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               kMultiMaxSmem);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_multi(int d, bool dev, bool adjoint, const MultiArgs &m, cudaStream_t st) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)m.p.grid);
  cfg.blockDim = dim3((unsigned)m.p.threads);
  cfg.dynamicSmemBytes = m.p.smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = m.a.pdl ? 1u : 0u;
  void *args[] = {const_cast<MultiArgs *>(&m)};
  return cudaLaunchKernelExC(&cfg, multi_kernel(d, dev, adjoint, m.a.s == 2.0), args);
}

}  // namespace lhe
