// lhe_step_multi.cu -- several steps of a small or 32-bit periodic 1D / 2D box in one launch.
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
  int W, x0, y0, nx, ny, own_x, own_y;
  __device__ __forceinline__ explicit MultiTile(const StepArgs &a, const MultiPlan &p) {
    const int ty = D == 2 ? blockIdx.x / p.tiles_x : 0, tx = blockIdx.x - ty * p.tiles_x;
    W = p.w;
    nx = a.g.n[0];
    ny = D == 2 ? a.g.n[1] : 1;
    x0 = tx * p.tx - (p.H - 1);
    y0 = D == 2 ? ty * p.ty - (p.H - 1) : 0;
    // the tile's own nodes (a last tile may stick out of the box: the nodes beyond are another tile's)
    own_x = min(p.tx, nx - tx * p.tx);
    own_y = D == 2 ? min(p.ty, ny - ty * p.ty) : 1;
  }
  // node of the box at (ix, iy) of the first step's region
  __device__ __forceinline__ int32_t site(int ix, int iy, int &gx, int &gy) const {
    gx = wrap_once(x0 + ix, nx);
    gy = D == 2 ? wrap_once(y0 + iy, ny) : 0;
    return gx + nx * gy;
  }
};

// t = r w + rest for 0 <= t < 2^13, inv ~ 1 / w: the product is within 2^-21 t / w of (t + 1/2) / w, which is at
// least 1 / (2 w) from an integer.
__device__ __forceinline__ int row_of(int t, float inv) { return (int)(((float)t + 0.5f) * inv); }

// Calls node(ix, iy, t) for the nodes of step j (1 .. H) of the region, one after another per thread.
template <int D, class F>
__device__ __forceinline__ void multi_nodes(const MultiPlan &p, int j, F node) {
  const int o = j - 1, w = p.w - 2 * o, nodes = w * (D == 2 ? p.h - 2 * o : 1);
  const float inv = __fdividef(1.0f, (float)w);
  for (int t = threadIdx.x; t < nodes; t += blockDim.x) {
    const int r = D == 2 ? row_of(t, inv) : 0;
    node(t - r * w + o, D == 2 ? r + o : 0);
  }
}

// The two copies hold the nodes' populations together (Q consecutive values a node): a neighbour's address is one
// of three row addresses plus a constant, and Q is odd, so that the lanes of a warp fall on different banks.
// (With population-major copies each access took its own address arithmetic: 329 instructions a node and
// step in 32 bits, twice the arithmetic's.)
template <int D, bool ADJ, class T>
__device__ __forceinline__ void pull_shared(const T *__restrict__ from, int c, int W, T (&f)[Lattice<D>::Q]) {
  constexpr Lattice<D> L{};
  constexpr int Q = Lattice<D>::Q;
  const T *row[3];
  row[1] = from + c * Q;
  row[0] = D == 2 ? row[1] - W * Q : row[1];
  row[2] = D == 2 ? row[1] + W * Q : row[1];
#pragma unroll
  for (int k = 0; k < Q; ++k) {
    const int ex = ADJ ? L.e[k][0] : -L.e[k][0], ey = D == 2 ? (ADJ ? L.e[k][D - 1] : -L.e[k][D - 1]) : 0;
    f[k] = row[1 + ey][ex * Q + k];
  }
}

template <int D, bool ADJ, int MODE>
__global__ void __launch_bounds__(kMultiThreads) k_multi_fp64(const __grid_constant__ MultiArgs m) {
  constexpr Lattice<D> L{};
  constexpr int Q = Lattice<D>::Q;
  extern __shared__ __align__(16) unsigned char smem[];
  const StepArgs &a = m.a;
  const MultiPlan &p = m.p;
  const int H = p.H, N = p.w * p.h;
  double *buf = reinterpret_cast<double *>(smem);  // two copies of N x Q
  double *acc = buf + 2 * N * Q;                   // adjoint: dL/dR of the tile
  const MultiTile<D> tile(a, p);
  const int64_t S = a.g.S;
  // the collision of step o + 1 at (ix, iy): psi from the pulled populations, dL/dR on the way
  auto collide = [&](const double (&f)[Q], int o, int ix, int iy) {
    double psi;
    if (ADJ) {
      const double w2 = MODE == kModeS2 ? fixed_moment_sum<Q, 1>(f) : fixed_moment_sum<Q, 0>(f);
      psi = MODE == kModeS2 ? w2 : m.sig[o] * w2;
      const int lx = ix - (H - 1), ly = D == 2 ? iy - (H - 1) : 0;
      if (a.gR && lx >= 0 && lx < tile.own_x && ly >= 0 && ly < tile.own_y) {
        int gx, gy;
        const int32_t site = tile.site(ix, iy, gx, gy);
        const int c = lx + p.tx * ly;
        const double g = fma(MODE == kModeS2 ? a.half_dt : m.gsc[o], w2, o == 0 ? a.gR[site] : acc[c]);
        if (o == H - 1) a.gR[site] = g;
        else acc[c] = g;
      }
    } else {
      int gx, gy;
      const double R = a.Rfield ? __ldg(a.Rfield + tile.site(ix, iy, gx, gy)) : 0.0;
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
  multi_nodes<D>(p, 1, [&](int ix, int iy) {
    int x[D], gx, gy;
    const int32_t site = tile.site(ix, iy, gx, gy);
    x[0] = gx;
    if (D == 2) x[D - 1] = gy;
    int32_t om[D], op[D];
    axis_offsets<D, false>(a.g, x, om, op);
    double f[Q];
#pragma unroll
    for (int k = 0; k < Q; ++k) f[k] = __ldg(src + k * S + source_site<D, ADJ>(L, k, site, om, op));
    const double psi = collide(f, 0, ix, iy);
    double *to = buf + (ix + tile.W * iy) * Q;
#pragma unroll
    for (int k = 0; k < Q; ++k) to[k] = out(f[k], psi, 0, k);
  });
  __syncthreads();
  int cur = 0;
  for (int j = 2; j < H; ++j) {
    const double *from = buf + cur * N * Q;
    double *dst = buf + (cur ^ 1) * N * Q;
    multi_nodes<D>(p, j, [&](int ix, int iy) {
      const int c = ix + tile.W * iy;
      double f[Q];
      pull_shared<D, ADJ>(from, c, tile.W, f);
      const double psi = collide(f, j - 1, ix, iy);
      double *to = dst + c * Q;
#pragma unroll
      for (int k = 0; k < Q; ++k) to[k] = out(f[k], psi, j - 1, k);
    });
    __syncthreads();
    cur ^= 1;
  }
  const double *from = buf + cur * N * Q;
  double *__restrict__ dst = static_cast<double *>(a.dst);
  multi_nodes<D>(p, H, [&](int ix, int iy) {
    if (ix - (H - 1) >= tile.own_x || (D == 2 && iy - (H - 1) >= tile.own_y)) return;
    int gx, gy;
    const int32_t site = tile.site(ix, iy, gx, gy);
    double f[Q];
    pull_shared<D, ADJ>(from, ix + tile.W * iy, tile.W, f);
    const double psi = collide(f, H - 1, ix, iy);
#pragma unroll
    for (int k = 0; k < Q; ++k) dst[k * S + site] = out(f[k], psi, H - 1, k);
  });
}

template <int D, bool ADJ, bool S2>
__global__ void __launch_bounds__(kMultiThreads) k_multi_dev(const __grid_constant__ MultiArgs m) {
  constexpr Lattice<D> L{};
  constexpr int Q = Lattice<D>::Q;
  extern __shared__ __align__(16) unsigned char smem[];
  const StepArgs &a = m.a;
  const MultiPlan &p = m.p;
  const int H = p.H, N = p.w * p.h;
  double *acc = reinterpret_cast<double *>(smem);                           // adjoint: dL/dR of the tile
  float2 *bphi = reinterpret_cast<float2 *>(acc + (ADJ ? p.tx * p.ty : 0));  // two copies of N
  float *buf = reinterpret_cast<float *>(bphi + 2 * N);                     // two copies of N x Q
  const MultiTile<D> tile(a, p);
  const int64_t S = a.g.S;
  const bool field = !ADJ && a.Rfield != nullptr;
  const float oms = (float)a.oms;
  // step o + 1 at (ix, iy) from the pulled deviations and the differences of phi: the new pair of phi; gk becomes the new deviations
  auto collide = [&](float (&gk)[Q], const float (&dl)[Q], float2 p0, int o, int ix, int iy) {
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
      const int lx = ix - (H - 1), ly = D == 2 ? iy - (H - 1) : 0;
      if (a.gR && lx >= 0 && lx < tile.own_x && ly >= 0 && ly < tile.own_y) {
        int gx, gy;
        const int32_t site = tile.site(ix, iy, gx, gy);
        const int q = lx + p.tx * ly;
        const double g = fma(a.dt, df_value(pn), o == 0 ? a.gR[site] : acc[q]);
        if (o == H - 1) a.gR[site] = g;
        else acc[q] = g;
      }
    } else if (field) {
      int gx, gy;
      dtR = (float)(a.dt * __ldg(a.Rfield + tile.site(ix, iy, gx, gy)));
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
    pull_shared<D, ADJ>(from, c, tile.W, gk);
    const float2 *row[3];
    row[1] = pf + c;
    row[0] = D == 2 ? row[1] - tile.W : row[1];
    row[2] = D == 2 ? row[1] + tile.W : row[1];
    const float2 p0 = *row[1];
    dl[0] = 0.0f;
#pragma unroll
    for (int k = 1; k < Q; ++k) {
      const int ex = ADJ ? L.e[k][0] : -L.e[k][0], ey = D == 2 ? (ADJ ? L.e[k][D - 1] : -L.e[k][D - 1]) : 0;
      const float2 pk = row[1 + ey][ex];
      dl[k] = (pk.x - p0.x) + (pk.y - p0.y);
    }
    return p0;
  };
  pdl_wait();
  const float *__restrict__ src = static_cast<const float *>(a.src);
  const float2 *__restrict__ phis = a.phi_src;
  multi_nodes<D>(p, 1, [&](int ix, int iy) {
    int x[D], gx, gy;
    const int32_t site = tile.site(ix, iy, gx, gy);
    x[0] = gx;
    if (D == 2) x[D - 1] = gy;
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
    const int c = ix + tile.W * iy;
    bphi[c] = collide(gk, dl, p0, 0, ix, iy);
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
    multi_nodes<D>(p, j, [&](int ix, int iy) {
      const int c = ix + tile.W * iy;
      float gk[Q], dl[Q];
      const float2 p0 = pull(from, pf, c, gk, dl);
      pt[c] = collide(gk, dl, p0, j - 1, ix, iy);
#pragma unroll
      for (int k = 0; k < Q; ++k) to[c * Q + k] = gk[k];
    });
    __syncthreads();
    cur ^= 1;
  }
  const float *from = buf + cur * N * Q;
  const float2 *pf = bphi + cur * N;
  float *__restrict__ dst = static_cast<float *>(a.dst);
  multi_nodes<D>(p, H, [&](int ix, int iy) {
    if (ix - (H - 1) >= tile.own_x || (D == 2 && iy - (H - 1) >= tile.own_y)) return;
    int gx, gy;
    const int32_t site = tile.site(ix, iy, gx, gy);
    float gk[Q], dl[Q];
    const float2 p0 = pull(from, pf, ix + tile.W * iy, gk, dl);
    a.phi_dst[site] = collide(gk, dl, p0, H - 1, ix, iy);
#pragma unroll
    for (int k = 0; k < Q; ++k) dst[k * S + site] = gk[k];
  });
}

namespace {

// H steps over tiles of tx x ty nodes, a thread per node of the first region up to `most`.
MultiPlan make_multi(const Geom &g, bool dev, int tx, int ty, int H, int most) {
  MultiPlan p;
  p.H = H;
  p.tx = tx;
  p.ty = g.d == 2 ? ty : 1;
  p.w = tx + 2 * (H - 1);
  p.h = g.d == 2 ? ty + 2 * (H - 1) : 1;
  p.tiles_x = (g.n[0] + tx - 1) / tx;
  p.grid = p.tiles_x * (g.d == 2 ? (g.n[1] + ty - 1) / ty : 1);
  p.threads = std::min(most, (p.w * p.h + 31) / 32 * 32);
  const size_t Q = 2 * g.d * g.d + 1, N = (size_t)p.w * p.h;
  p.smem = 8 * (size_t)p.tx * p.ty + 2 * N * (dev ? 4 * Q + 8 : 8 * Q);
  return p;
}

template <int D>
const void *multi_kernel(bool dev, bool adjoint, bool s2) {
  if (dev)
    return adjoint ? (s2 ? (const void *)k_multi_dev<D, true, true> : (const void *)k_multi_dev<D, true, false>)
                   : (s2 ? (const void *)k_multi_dev<D, false, true> : (const void *)k_multi_dev<D, false, false>);
  return adjoint ? (s2 ? (const void *)k_multi_fp64<D, true, kModeS2> : (const void *)k_multi_fp64<D, true, kModeGeneral>)
                 : (s2 ? (const void *)k_multi_fp64<D, false, kModeS2> : (const void *)k_multi_fp64<D, false, kModeGeneral>);
}

const void *multi_kernel(int d, bool dev, bool adjoint, bool s2) {
  return d == 1 ? multi_kernel<1>(dev, adjoint, s2) : multi_kernel<2>(dev, adjoint, s2);
}

}  // namespace

// The plan of a periodic 1D / 2D box, or none (one step per launch). Small grids: one tile per SM, the one with the
// smallest first region, a thread per node of it, and as many steps as pay for the rings that the tiles share
// with their neighbours: FP64 is held back by the FP64 pipe (~2 operations per clock per SM, 10 a node), so that H
// falls with the tile's size, and none pays from ~260^2 on. 32 bits pay further on, where a launch is short beside a
// step, and again from 1.5 M nodes, where the two states leave L2 and H steps pass memory once.
// us per step, one step per launch / this rule (forward):
//   FP64 D2Q9 16^2 1.90 / 1.31, 64^2 2.14 / 1.39, 128^2 2.22 / 1.66, 200^2 3.08 / 2.46, 256^2 3.66 / 3.21, 270 x 260 3.68 / 3.52 with the
//     adjoint 3.52 / 3.69 (not taken), 500 x 333 5.9 / 7.1 (32 x 8, H = 2; not taken); D1Q3 64 1.92 / 0.74, 30000 2.01 / 1.03,
//     10^6 16.4 / 18.4 (not taken)
//   32 bits D2Q9 16^2 1.90 / 0.60, 64^2 1.90 / 0.70, 128^2 1.90 / 0.84, 256^2 2.05 / 1.42, 320^2 2.29 / 2.23, 500 x 333 3.33 / 2.97, 1000^2
//     11.7 / 12.1 (not taken), 1250^2 23.3 / 19.8, 2048^2 58.7 / 50.5; D1Q3 4096 1.89 / 0.47, 10^5 1.96 / 1.13, 2 10^6 17.1 / 8.3
bool plan_multi(const Geom &g, bool dev, int sms, MultiPlan &best) {
  best = MultiPlan{};
  if (g.d > 2 || sms <= 0) return false;
  const int64_t S = g.S, share = (S + sms - 1) / sms;  // nodes per SM
  const int ny = g.d == 2 ? g.n[1] : 1;
  // (a region that wraps around the box once at most)
  auto fits = [&](int tx, int ty, int H) { return tx + H - 1 <= g.n[0] && (g.d < 2 || ty + H - 1 <= ny); };
  if (g.d == 1) {
    if (!dev && share > 200) return false;
    const int tx = (int)std::min<int64_t>(512, std::max<int64_t>(32, share));
    if (fits(tx, 1, kMultiMaxSteps)) best = make_multi(g, dev, tx, 1, kMultiMaxSteps, 256);
  } else if (share <= (dev ? 480 : 440)) {
    const int H = dev ? (share <= 160 ? 6 : 4) : (share <= 48 ? 4 : (share <= 160 ? 3 : 2));
    int64_t least = INT64_MAX;
    for (int tx = 4; tx <= 64; tx += 4)
      for (int ty = 1; ty <= 64; ++ty) {
        if (!fits(tx, ty, H)) continue;
        const int64_t tiles = (int64_t)((g.n[0] + tx - 1) / tx) * ((ny + ty - 1) / ty);
        const int64_t region = (int64_t)(tx + 2 * (H - 1)) * (ty + 2 * (H - 1));
        if (tiles > sms || region > kMultiThreads || region >= least) continue;
        least = region;
        best = make_multi(g, dev, tx, ty, H, kMultiThreads);
      }
  } else if (dev && S <= 180000 && fits(32, 8, 3)) {
    best = make_multi(g, dev, 32, 8, 3, 192);
  } else if (dev && S >= 1500000 && fits(32, 16, 2)) {
    best = make_multi(g, dev, 32, 16, 2, 320);
  }
  return best.H > 1;
}

MultiPlan shorter_multi(const Geom &g, bool dev, const MultiPlan &p, int H) {
  return H == p.H ? p : make_multi(g, dev, p.tx, p.ty, H, p.threads);
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
