// lhe_stability.cu -- stability maps (Sec. 4): for a batch of velocities sigma and a grid of Fourier
// variables xi, the spectral radius of the amplification matrix of one step on a Fourier mode,
// G(xi) = T(xi) ((1 - s) I + s omega 1^T), T = diag(exp(-i e_k . xi)), in population space (Eq. (G)
// is the same matrix in moment space, G_moment = M G M^{-1}). The von Neumann (L2) condition is
// rho(G(xi)) <= 1 for every xi; Proposition 1's microscopic entropy condition is min_k omega_k > 0.
//
// The matrix is a diagonal plus a rank-one matrix: its eigenvalues are found from the secular equation
// (k_stability), with repeated phases deflated, so that the (Q-1)-fold eigenvalue 1 - s of G(0) comes out to
// rounding, where the roots of the characteristic polynomial would spread by eps^(1/(Q-1)). A matrix whose roots
// do not pass the trace checks takes the backward-stable QR route (radius_qr): the Q x Q complex matrix is reduced
// to upper Hessenberg form by Householder reflections, then its eigenvalues are found by the shifted
// QR iteration (Givens rotations, Wilkinson shifts, deflation on negligible subdiagonals), all in FP64.
// The radius per sigma is the maximum over its xi, reduced with an integer atomic max on the (non-negative)
// double bits.
#include <algorithm>

#include "lhe_internal.h"

namespace lhe {

namespace {

constexpr double kPi = 3.14159265358979323846;

struct cd {
  double re, im;
};
__device__ __forceinline__ cd mk(double r, double i) { return cd{r, i}; }
__device__ __forceinline__ cd operator+(cd a, cd b) { return cd{a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ cd operator-(cd a, cd b) { return cd{a.re - b.re, a.im - b.im}; }
__device__ __forceinline__ cd operator*(cd a, cd b) { return cd{a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re}; }
__device__ __forceinline__ cd operator*(double s, cd a) { return cd{s * a.re, s * a.im}; }
__device__ __forceinline__ cd cj(cd a) { return cd{a.re, -a.im}; }
__device__ __forceinline__ double ab2(cd a) { return a.re * a.re + a.im * a.im; }
__device__ __forceinline__ double ab(cd a) { return hypot(a.re, a.im); }
__device__ __forceinline__ double ab1(cd a) { return fabs(a.re) + fabs(a.im); }
// principal square root
__device__ __forceinline__ cd csqrt_(cd z) {
  const double r = ab(z);
  if (r == 0.0) return cd{0.0, 0.0};
  const double t = sqrt(0.5 * (r + fabs(z.re)));
  if (z.re >= 0.0) return cd{t, z.im / (2.0 * t)};
  return cd{fabs(z.im) / (2.0 * t), z.im >= 0.0 ? t : -t};
}

// Largest eigenvalue modulus of the N x N complex matrix A (destroyed). Returns NaN when the QR
// iteration does not converge within its iteration budget (80 sweeps per eigenvalue) and the
// remaining window is not triangular to 1e-10.
template <int N>
__device__ double spectral_radius(cd (&A)[N][N]) {
  // 1. upper Hessenberg form: for each column k, a reflection I - 2 v v^H / (v^H v) zeroes A[k+2.., k]
  for (int k = 0; k < N - 2; ++k) {
    double tail = 0.0;
    for (int i = k + 2; i < N; ++i) tail += ab2(A[i][k]);
    if (tail == 0.0) continue;
    const cd x0 = A[k + 1][k];
    const double xn = sqrt(ab2(x0) + tail), a0 = ab(x0);
    const cd ph = a0 > 0.0 ? mk(x0.re / a0, x0.im / a0) : mk(1.0, 0.0);
    cd v[N];
    v[k + 1] = x0 + xn * ph;
    for (int i = k + 2; i < N; ++i) v[i] = A[i][k];
    const double vv = ab2(v[k + 1]) + tail;
    for (int j = k; j < N; ++j) {  // A <- H A on rows k+1..N-1
      cd dot = mk(0.0, 0.0);
      for (int i = k + 1; i < N; ++i) dot = dot + cj(v[i]) * A[i][j];
      const cd f = (2.0 / vv) * dot;
      for (int i = k + 1; i < N; ++i) A[i][j] = A[i][j] - v[i] * f;
    }
    for (int i = 0; i < N; ++i) {  // A <- A H on columns k+1..N-1
      cd dot = mk(0.0, 0.0);
      for (int j = k + 1; j < N; ++j) dot = dot + A[i][j] * v[j];
      const cd f = (2.0 / vv) * dot;
      for (int j = k + 1; j < N; ++j) A[i][j] = A[i][j] - f * cj(v[j]);
    }
    for (int i = k + 2; i < N; ++i) A[i][k] = mk(0.0, 0.0);
  }
  // 2. shifted QR on the active window [lo, hi]
  double rho = 0.0;
  int hi = N - 1, iter = 0;
  cd gs[N];
  double gc[N];
  while (hi >= 0) {
    if (hi == 0) {
      rho = fmax(rho, ab(A[0][0]));
      break;
    }
    int lo = hi;
    for (; lo > 0; --lo) {
      const double tst = ab1(A[lo - 1][lo - 1]) + ab1(A[lo][lo]);
      if (ab1(A[lo][lo - 1]) <= 4.440892098500626e-16 * (tst > 0.0 ? tst : 1.0)) {  // 2 ulp
        A[lo][lo - 1] = mk(0.0, 0.0);
        break;
      }
    }
    if (lo == hi) {
      rho = fmax(rho, ab(A[hi][hi]));
      --hi;
      iter = 0;
      continue;
    }
    if (++iter > 80) {
      // budget spent: a window whose subdiagonal is at rounding level is triangular for our purpose
      for (int i = lo + 1; i <= hi; ++i)
        if (!(ab1(A[i][i - 1]) <= 1e-10 * (ab1(A[i - 1][i - 1]) + ab1(A[i][i]))))  // (not finite: not converged)
          return __longlong_as_double(0x7FF8000000000000ll);
      for (int i = lo; i <= hi; ++i) rho = fmax(rho, ab(A[i][i]));
      hi = lo - 1;
      iter = 0;
      continue;
    }
    // Wilkinson shift: the eigenvalue of the trailing 2 x 2 block nearer to its last entry
    const cd a = A[hi - 1][hi - 1], b = A[hi - 1][hi], c = A[hi][hi - 1], d = A[hi][hi];
    const cd half_tr = 0.5 * (a + d);
    const cd disc = csqrt_(half_tr * half_tr - (a * d - b * c));
    const cd m1 = half_tr + disc, m2 = half_tr - disc;
    cd mu = ab2(m1 - d) < ab2(m2 - d) ? m1 : m2;
    if (iter % 10 == 9) {  // exceptional shift, off the symmetric configurations that stall the iteration
      const double sc = ab1(c) + (hi - 1 > lo ? ab1(A[hi - 1][hi - 2]) : 0.0);
      mu = d + mk(0.75 * sc, 0.45 * sc);
    }
    for (int i = lo; i <= hi; ++i) A[i][i] = A[i][i] - mu;
    for (int k = lo; k < hi; ++k) {  // R = G_{hi-1} ... G_lo (H - mu I)
      const cd x = A[k][k], y = A[k + 1][k];
      double cc;
      cd ss;
      const double ax = ab(x), ay = ab(y);
      if (ay == 0.0) {
        cc = 1.0;
        ss = mk(0.0, 0.0);
      } else if (ax == 0.0) {
        cc = 0.0;
        ss = mk(y.re / ay, -y.im / ay);
      } else {
        const double r = hypot(ax, ay);
        cc = ax / r;
        ss = (1.0 / r) * (mk(x.re / ax, x.im / ax) * cj(y));
      }
      gc[k] = cc;
      gs[k] = ss;
      for (int j = k; j <= hi; ++j) {
        const cd p = A[k][j], q = A[k + 1][j];
        A[k][j] = cc * p + ss * q;
        A[k + 1][j] = cc * q - cj(ss) * p;
      }
    }
    for (int k = lo; k < hi; ++k) {  // R Q: apply each G_k^H from the right
      const double cc = gc[k];
      const cd ss = gs[k];
      const int top = min(k + 2, hi);
      for (int i = lo; i <= top; ++i) {
        const cd p = A[i][k], q = A[i][k + 1];
        A[i][k] = cc * p + cj(ss) * q;
        A[i][k + 1] = cc * q - ss * p;
      }
    }
    for (int i = lo; i <= hi; ++i) A[i][i] = A[i][i] + mu;
  }
  return rho;
}

// The radius of one matrix by the QR route, from the population-space matrix itself.
template <int D>
__device__ __noinline__ double radius_qr(const double *__restrict__ omega, const int (&j)[D], int32_t nxi, double s) {
  constexpr Lattice<D> L{};
  constexpr int Q = Lattice<D>::Q;
  double xi[D];
  for (int i = 0; i < D; ++i) xi[i] = -kPi + 2.0 * kPi * (double)j[i] / (double)nxi;
  cd A[Q][Q];
  for (int k = 0; k < Q; ++k) {
    double ph = 0.0;
    for (int i = 0; i < D; ++i) ph -= L.e[k][i] * xi[i];
    double sn, cs;
    sincos(ph, &sn, &cs);
    const cd tk = mk(cs, sn);  // exp(-i e_k . xi)
    const double wk = s * omega[k];
    for (int q = 0; q < Q; ++q) A[k][q] = (wk + (q == k ? 1.0 - s : 0.0)) * tk;
  }
  const double rho = spectral_radius<Q>(A);
  return rho == rho ? rho : __longlong_as_double(0x7FF0000000000000ll);  // not converged: report +inf
}

struct StabilityArgs {
  const double *omega;  // Q per velocity
  unsigned long long *rho_bits;
  int64_t npoints, nper;  // velocities; Fourier variables per velocity that are visited
  int32_t nxi;
  double s;
  StabilityRest rest;
  int8_t e[33][4];
};

// Velocity and Fourier indices of matrix t.
template <int D>
__device__ __forceinline__ int64_t matrix_of(const StabilityArgs &a, int64_t t, int (&j)[D]) {
  const int64_t pt = t / a.nper;
  int64_t r = t - pt * a.nper;
#pragma unroll
  for (int i = 0; i < D; ++i) {
    j[i] = (int)(i == D - 1 ? r : r % a.nxi);
    r /= a.nxi;
  }
  return pt;
}

// The bits of non-negative doubles order as integers; most matrices do not raise the maximum.
__device__ __forceinline__ void raise_radius(unsigned long long *out, double rho) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(rho);
  if (*(volatile unsigned long long *)out < bits) atomicMax(out, bits);
}

struct cf {
  float re, im;
};
__device__ __forceinline__ cf operator+(cf a, cf b) { return cf{a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ cf operator-(cf a, cf b) { return cf{a.re - b.re, a.im - b.im}; }
__device__ __forceinline__ cf operator*(cf a, cf b) { return cf{a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re}; }
__device__ __forceinline__ float ab2(cf a) { return fmaf(a.re, a.re, a.im * a.im); }
__device__ __forceinline__ cf rcp(cf a) {
  const float n = __fdividef(1.0f, ab2(a));
  return cf{a.re * n, -a.im * n};
}
// 1/n by one third-order Newton step, x (1 + e + e^2) with e = 1 - n x, from a seed of ~22 bits: three FP64
// operations (a division takes several times that), within one unit in the last place. For 2^-126 < n < 2^126.
__device__ __forceinline__ cd rcp(cd a) {
  const double n = ab2(a);
  const double x = float_to_double(__fdividef(1.0f, ff_split(n).x));
  const double e = fma(-n, x, 1.0);
  const double y = fma(x, fma(e, e, e), x);
  return cd{a.re * y, -a.im * y};
}

// G(xi) is a diagonal plus a rank-one matrix, T((1 - s) I + s omega 1^T), so its eigenvalues need no O(Q^3)
// reduction. Links with the same phase share a pole tau_p (the phases are multiples of pi / nxi: exact integers),
// whose weights add up to W_p; all but one of a shared pole's links, and poles of weight zero, have the eigenvalue
// (1 - s) tau_p. The others are (1 - s) z with z a root of the secular equation (Golub, "Some modified
// matrix eigenvalue problems", SIAM Review 15, 1973)
//   1 + kappa sum_p tau_p W_p / (tau_p - z) = 0,  kappa = s / (1 - s).
// All P <= Q roots are found together by the Ehrlich-Aberth iteration (Aberth, "Iteration methods for finding all
// zeros of a polynomial simultaneously", Math. Comp. 27, 1973) on the polynomial of which they are the
// zeros, each as an offset d from a pole b, z = tau_b + d, which keeps roots next to poles of small weight
// exact: with c_p = kappa tau_p W_p, S = 1 + sum_{p != b} c_p / (tau_p - z) and g = d S - c_b,
//   d -= g / (S + d S' + g (sum_{p != b} 1 / (z - tau_p) - sum_{other roots} 1 / (z - z_j))).
// FP32 iterations (the FP32 pipe runs 64 times the FP64 pipe's rate) bring the offsets to ~1e-6; then S and g
// in FP64, with the denominator still in FP32, until a step is below 2e-9 (the step's relative error
// is ~1e-6, so the next one would be below rounding): two as a rule. The roots are accepted if their sum and sum
// of squares match the matrix's traces, to 1e-10 of its size and of its square (absolute checks, or ones that grow with
// kappa^2, rejected velocities of order 100 and let anything pass for tau near 1); else, and without convergence, the matrix
// is left to the QR route (k_stability_qr, a thread per matrix; within this kernel one lane of a group ran it while the others
// waited: 24 velocities of order 100, D3Q19, 12^3 Fourier variables 134 ms, now 0.84 by the secular equation, 61 by QR).
// Weights above 1e6 and ones that are not finite go there at once: FP32 cannot hold their products.
// A group of G lanes holds a matrix, a lane a root (two for the 33rd pole of D = 4); G is the smallest of 8, 16
// and 32 that holds the poles, of which there are at most nxi (nxi even) or 2 nxi. G(-xi) is the conjugate of G(xi), so half
// of the last axis is visited. Bound by the FP64 pipe (85 % busy: S in the last two iterations, the poles' sines). Against roots
// refined in 80 bits (600 random D3Q19 matrices) the radius is within 6e-15, LAPACK's QR within 3e-14. 24 velocities of D3Q19,
// 12^3 Fourier variables: 29.2 ms by QR (one thread per matrix, in local memory) -> 0.50 ms; the whole call takes 0.55.
// (D4Q33 in groups of 8 on at least five CTAs an SM: at 114 registers and four it took a tenth longer. 0 leaves the others alone.)
template <int D, int G>
__global__ void __launch_bounds__(128, D == 4 && G == 8 ? 5 : 0) k_stability(const __grid_constant__ StabilityArgs a) {
  constexpr int Q = 2 * D * D + 1;
  constexpr int R = (Q + G - 1) / G;  // roots per lane at most
  constexpr int kGroups = 128 / G;
  __shared__ cd tau64[kGroups][Q], c64[kGroups][Q];  // poles and kappa tau_p W_p
  __shared__ float4 tauf[kGroups][Q];                // poles as float pairs (re, im, low parts)
  __shared__ cf cfl[kGroups][Q], off[kGroups][Q];    // the weights in FP32; offsets of the roots from their own poles
  __shared__ int ang[kGroups][Q];
  const int grp = threadIdx.x / G, lane = threadIdx.x % G, nxi = a.nxi;
  const unsigned shift = (threadIdx.x & 31u) / G * G, gmask = G == 32 ? 0xffffffffu : ((1u << (G & 31)) - 1u) << shift;
  const int64_t total = a.npoints * a.nper;
  for (int64_t t0 = blockIdx.x * (int64_t)kGroups; t0 < total; t0 += (int64_t)gridDim.x * kGroups) {
    int64_t t = t0 + grp;
    const bool idle = t >= total;  // surplus groups repeat the last matrix and write nothing
    if (idle) t = total - 1;
    __syncwarp();  // the last matrix's tables are read out
    int j[D];
    const int64_t pt = matrix_of(a, t, j);
    const double *__restrict__ omega = a.omega + pt * Q;
    // phases of the links, -e_k . xi = (pi / nxi) (nxi sum_i e_ki - 2 sum_i e_ki j_i)
    for (int k = lane; k < Q; k += G) {
      int v = 0;
#pragma unroll
      for (int i = 0; i < D; ++i) v += a.e[k][i] * (nxi - 2 * j[i]);
      v %= 2 * nxi;
      ang[grp][k] = v < 0 ? v + 2 * nxi : v;
    }
    __syncwarp();
    const double r1 = 1.0 - a.s, kappa = a.s / r1;
    int P = 0;
    bool deflated = false;
    cd trace = mk(0.0, 0.0);  // sum over the links of tau W
    for (int k0 = 0; k0 < Q; k0 += G) {
      const int k = k0 + lane;
      bool first = k < Q;
      double W = 0.0;
      if (k < Q)
        for (int q = 0; q < Q; ++q)
          if (ang[grp][q] == ang[grp][k]) {
            if (q < k) first = false;
            W += omega[q];
          }
      const bool keep = first && fabs(W) > 1e-15;
      const unsigned kept = __ballot_sync(0xffffffffu, keep) & gmask;
      if (__ballot_sync(0xffffffffu, k < Q && !keep) & gmask) deflated = true;
      if (keep) {
        const int p = P + __popc(kept & ((1u << (threadIdx.x & 31u)) - 1u));
        double sn, cs;
        sincospi((double)ang[grp][k] / (double)nxi, &sn, &cs);
        const cd c = (kappa * W) * mk(cs, sn);
        tau64[grp][p] = mk(cs, sn);
        c64[grp][p] = a.s == 1.0 ? W * mk(cs, sn) : c;
        cfl[grp][p] = cf{(float)c.re, (float)c.im};
        const float2 x = df_split(cs), y = df_split(sn);
        tauf[grp][p] = make_float4(x.x, y.x, x.y, y.y);
      }
      P += __popc(kept);
    }
    __syncwarp();
    float size = 0.0f;  // of the matrix over 1 - s, besides its diagonal
    for (int p = 0; p < P; ++p) {
      trace = trace + c64[grp][p];  // kappa sum tau W
      size += fabsf(cfl[grp][p].re) + fabsf(cfl[grp][p].im);
    }
    if (a.s == 1.0) {  // the matrix has rank one: its only eigenvalue besides 0 is sum tau W
      if (lane == 0 && !idle) atomicMax(a.rho_bits + pt, (unsigned long long)__double_as_longlong(ab(trace)));
      continue;
    }
    // pole i minus pole q in FP32
    auto pole_diff = [&](float4 ti, int q) {
      const float4 tq = tauf[grp][q];
      return cf{(ti.x - tq.x) + (ti.z - tq.z), (ti.y - tq.y) + (ti.w - tq.w)};
    };
    // first offsets: the other poles seen from the pole
    cf d[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int i = lane + r * G;
      d[r] = cf{0.0f, 0.0f};
      if (i >= P) continue;
      const float4 ti = tauf[grp][i];
      cf S{1.0f, 0.0f};
      for (int q = 0; q < P; ++q)
        if (q != i) S = S - cfl[grp][q] * rcp(pole_diff(ti, q));
      if (!(ab2(S) >= 0.0625f)) S = cf{0.25f, 0.0f};
      // a little off the symmetric starts from which the iteration cannot part two roots
      d[r] = cfl[grp][i] * rcp(S) * cf{1.0f + 0.02f * (float)((i * 5) % 7 - 3) * 0.33f, 0.02f * (float)((i * 3) % 5 - 2) * 0.5f};
      off[grp][i] = d[r];
    }
    __syncwarp();
    const float reach = fmaxf(0.5f, 0.5f * fabsf((float)kappa));
    for (int it = 0; it < 20; ++it) {
      float worst = 0.0f;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int i = lane + r * G;
        if (i >= P) continue;
        const float4 ti = tauf[grp][i];
        cf S{1.0f, 0.0f}, Sp{0.0f, 0.0f}, sum{0.0f, 0.0f};
        for (int q = 0; q < P; ++q) {
          if (q == i) continue;
          const cf z = pole_diff(ti, q) + d[r];
          const cf A = rcp(z), T = cfl[grp][q] * A;
          S = S - T;
          Sp = Sp + T * A;
          sum = sum + A - rcp(z - off[grp][q]);
        }
        const cf g = d[r] * S - cfl[grp][i];
        cf st = g * rcp(S + d[r] * Sp + g * sum);
        const float m = sqrtf(ab2(st)), lim = fmaxf(reach, sqrtf(ab2(d[r])));
        if (!(m < 1e30f)) st = cf{0.01f, 0.0f};
        else if (m > lim) st = cf{st.re * (lim / m), st.im * (lim / m)};
        worst = fmaxf(worst, m < 1e30f ? m / fmaxf(1.0f, sqrtf(ab2(d[r]))) : 1.0f);
        d[r] = d[r] - st;
      }
      __syncwarp();
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (lane + r * G < P) off[grp][lane + r * G] = d[r];
      __syncwarp();
      if (!__any_sync(0xffffffffu, worst > 4e-6f)) break;
    }
    // FP64: the offset from the nearest pole
    int b[R];
    cd d64[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int i = lane + r * G;
      b[r] = 0;
      d64[r] = mk(0.0, 0.0);
      if (i >= P) continue;
      const float4 ti = tauf[grp][i];
      float best = ab2(d[r]);
      b[r] = i;
      for (int q = 0; q < P; ++q) {
        const float m = ab2(pole_diff(ti, q) + d[r]);
        if (q != i && m < best) {
          best = m;
          b[r] = q;
        }
      }
      d64[r] = (tau64[grp][i] - tau64[grp][b[r]]) + mk((double)d[r].re, (double)d[r].im);
    }
    bool converged = false;
    for (int it = 0; it < 12; ++it) {
      bool small = true;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int i = lane + r * G;
        if (i >= P) continue;
        const float4 ti = tauf[grp][i];
        const cd tb = tau64[grp][b[r]];
        cd S = mk(1.0, 0.0);
        cf Sp{0.0f, 0.0f}, sum{0.0f, 0.0f};
        for (int q = 0; q < P; ++q) {
          const cf z = pole_diff(ti, q) + off[grp][i];
          if (q != i) sum = sum - rcp(z - off[grp][q]);
          if (q == b[r]) continue;
          S = S - c64[grp][q] * rcp((tb - tau64[grp][q]) + d64[r]);
          const cf A = rcp(z);
          Sp = Sp + cfl[grp][q] * A * A;
          sum = sum + A;
        }
        const cd g = d64[r] * S - c64[grp][b[r]];
        const cf gf{(float)g.re, (float)g.im}, df{(float)d64[r].re, (float)d64[r].im};
        const cf inv = rcp(cf{(float)S.re, (float)S.im} + df * Sp + gf * sum);
        const cd st = g * mk((double)inv.re, (double)inv.im);
        d64[r] = d64[r] - st;
        if (!(ab2(st) <= 4e-18 * fmax(1.0, ab2(d64[r])))) small = false;
      }
      __syncwarp();
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int i = lane + r * G;
        if (i >= P) continue;
        const cd o = (tau64[grp][b[r]] - tau64[grp][i]) + d64[r];
        off[grp][i] = cf{(float)o.re, (float)o.im};
      }
      __syncwarp();
      converged = (__ballot_sync(0xffffffffu, !small) & gmask) == 0u;
      if (__all_sync(0xffffffffu, converged)) break;
    }
    // traces: sum z = sum tau + kappa sum tau W; sum z^2 = sum tau^2 (1 + 2 kappa W) + (kappa sum tau W)^2
    cd s1 = mk(0.0, 0.0), s2 = mk(0.0, 0.0);
    double top = 0.0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int i = lane + r * G;
      if (i >= P) continue;
      const cd ti = tau64[grp][i], z = tau64[grp][b[r]] + d64[r], c = c64[grp][i];
      s1 = s1 + z - ti - c;
      s2 = s2 + z * z - ti * ti - 2.0 * (ti * c);
      top = fmax(top, ab2(z));
    }
    for (int o = G / 2; o > 0; o >>= 1) {
      s1 = s1 + mk(__shfl_xor_sync(0xffffffffu, s1.re, o), __shfl_xor_sync(0xffffffffu, s1.im, o));
      s2 = s2 + mk(__shfl_xor_sync(0xffffffffu, s2.re, o), __shfl_xor_sync(0xffffffffu, s2.im, o));
      top = fmax(top, __shfl_xor_sync(0xffffffffu, top, o));
    }
    s2 = s2 - trace * trace;
    // (the roots' rounding grows with the matrix: large weights, or s near 1)
    const double scale = fmax(1.0, (double)size), tol = 1e-10 * P * scale;
    const bool good = converged && ab1(s1) < tol && ab1(s2) < tol * scale;
    if (lane == 0 && !idle) {
      if (good) {
        const double rho = fabs(r1) * sqrt(top);
        raise_radius(a.rho_bits + pt, deflated ? fmax(rho, fabs(r1)) : rho);
      } else {
        const unsigned long long q = atomicAdd(a.rest.count, 1ull);
        if (q < (unsigned long long)a.rest.room) a.rest.list[q] = t;
      }
    }
  }
}

// The matrices that the secular equation left over, one thread each (in local memory): those on the list, or all of
// them when the list was too short.
template <int D>
__global__ void __launch_bounds__(128) k_stability_qr(const __grid_constant__ StabilityArgs a) {
  const int64_t n = (int64_t)*a.rest.count, total = a.npoints * a.nper;
  const bool listed = n <= a.rest.room;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < (listed ? n : total); q += (int64_t)gridDim.x * blockDim.x) {
    int j[D];
    const int64_t pt = matrix_of(a, listed ? a.rest.list[q] : q, j);
    raise_radius(a.rho_bits + pt, radius_qr<D>(a.omega + pt * Lattice<D>::Q, j, a.nxi, a.s));
  }
}

template <int D, int G>
cudaError_t stability_dg(const StabilityArgs &a, cudaStream_t st) {
  const int64_t groups = a.npoints * a.nper;
  const int64_t blocks = std::min<int64_t>((groups + 128 / G - 1) / (128 / G), 1 << 20);
  k_stability<D, G><<<(unsigned)blocks, 128, 0, st>>>(a);
  return cudaGetLastError();
}

template <int D>
cudaError_t stability_d(StabilityArgs &a, bool rest, cudaStream_t st) {
  constexpr Lattice<D> L{};
  constexpr int Q = Lattice<D>::Q;
  for (int k = 0; k < Q; ++k)
    for (int i = 0; i < D; ++i) a.e[k][i] = (int8_t)L.e[k][i];
  a.nper = a.nxi / 2 + 1;  // G(-xi) = conj G(xi): j_d <= nxi / 2 (and its partner nxi - j_d)
  if (a.nper > a.nxi) a.nper = a.nxi;
  for (int i = 0; i < D - 1; ++i) a.nper *= a.nxi;
  if (rest) {
    const int64_t blocks = std::min<int64_t>((a.npoints * a.nper + 127) / 128, 1 << 20);
    k_stability_qr<D><<<(unsigned)blocks, 128, 0, st>>>(a);
    return cudaGetLastError();
  }
  const int poles = std::min(Q, a.nxi % 2 ? 2 * a.nxi : a.nxi);
  if constexpr (Q > 16)
    if (poles > 16) return stability_dg<D, 32>(a, st);
  if constexpr (Q > 8)
    if (poles > 8) return stability_dg<D, 16>(a, st);
  return stability_dg<D, 8>(a, st);
}

}  // namespace

static cudaError_t stability(int d, const double *omega_dev, int64_t npoints, int32_t nxi, double s,
                             unsigned long long *rho_bits_dev, const StabilityRest &r, bool rest, cudaStream_t st) {
  if (npoints <= 0) return cudaSuccess;
  StabilityArgs a{};
  a.omega = omega_dev;
  a.rho_bits = rho_bits_dev;
  a.npoints = npoints;
  a.nxi = nxi;
  a.s = s;
  a.rest = r;
  switch (d) {
    case 1: return stability_d<1>(a, rest, st);
    case 2: return stability_d<2>(a, rest, st);
    case 3: return stability_d<3>(a, rest, st);
    case 4: return stability_d<4>(a, rest, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_stability(int d, const double *omega_dev, int64_t npoints, int32_t nxi, double s,
                             unsigned long long *rho_bits_dev, const StabilityRest &r, cudaStream_t st) {
  return stability(d, omega_dev, npoints, nxi, s, rho_bits_dev, r, false, st);
}

cudaError_t launch_stability_rest(int d, const double *omega_dev, int64_t npoints, int32_t nxi, double s,
                                  unsigned long long *rho_bits_dev, const StabilityRest &r, cudaStream_t st) {
  return stability(d, omega_dev, npoints, nxi, s, rho_bits_dev, r, true, st);
}

}  // namespace lhe
