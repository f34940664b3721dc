// lhe_device.cuh -- device-side building blocks shared by the kernels of the library:
// the DdQ(2d^2+1) lattice as compile-time tables, division by run-time invariant integers,
// the fixed-point moment sum and the integer double -> float-pair split.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace lhe {

constexpr int kMaxD = 5;
constexpr int kMaxQ = 51;
constexpr int kMaxModes = 16;

// Threads per block of the fused step kernels (one thread per lattice node).
#ifndef LHE_STEP_THREADS
#define LHE_STEP_THREADS 128
#endif

// ----------------------------------------------------------------------------------------------
// Lattice (Sec. 2.3, Eq. (DdQ-M)): k = 0 rest; k = 1..d: +e_i; k = d+1..2d: -e_i; then for each
// pair i<j (lexicographic) four velocities with component i from J1 = (1,-1,-1,1) and component
// j from J2 = (1,1,-1,-1). Built at compile time so unrolled loops see constant components.
template <int D>
struct Lattice {
  static constexpr int Q = 2 * D * D + 1;
  int e[Q][D];
  int opp[Q];
  int nnz[Q];
  int ax[Q][2];  // indices of the nonzero components (-1 if absent)
  __host__ __device__ constexpr Lattice() : e{}, opp{}, nnz{}, ax{} {
    const int J1[4] = {1, -1, -1, 1}, J2[4] = {1, 1, -1, -1};
    for (int k = 0; k < Q; ++k)
      for (int i = 0; i < D; ++i) e[k][i] = 0;
    int k = 1;
    for (int i = 0; i < D; ++i) e[k++][i] = 1;
    for (int i = 0; i < D; ++i) e[k++][i] = -1;
    for (int i = 0; i < D; ++i)
      for (int j = i + 1; j < D; ++j)
        for (int r = 0; r < 4; ++r) {
          e[k][i] = J1[r];
          e[k][j] = J2[r];
          ++k;
        }
    for (int a = 0; a < Q; ++a) {
      opp[a] = -1;
      for (int b = 0; b < Q; ++b) {
        bool same = true;
        for (int i = 0; i < D; ++i)
          if (e[b][i] != -e[a][i]) same = false;
        if (same) opp[a] = b;
      }
      nnz[a] = 0;
      ax[a][0] = ax[a][1] = -1;
      for (int i = 0; i < D; ++i)
        if (e[a][i] != 0) ax[a][nnz[a]++] = i;
    }
  }
};

// ----------------------------------------------------------------------------------------------
// Division of a 32-bit unsigned by a run-time invariant divisor with one multiply-high
// (Granlund & Montgomery, "Division by invariant integers using multiplication", PLDI 1994):
// q = (umulhi(n, m) + n) >> l with l = ceil(log2 d), m = floor(2^32 (2^l - d) / d) + 1.
struct FastDiv {
  uint32_t d = 1, m = 0;
  int32_t l = 0;
  FastDiv() = default;
  __host__ explicit FastDiv(uint32_t div) : d(div) {
    l = 0;
    while ((1ull << l) < div) ++l;
    m = (uint32_t)((((1ull << 32) * ((1ull << l) - div)) / div) + 1ull);
    if (div == 1) m = 0;
  }
  __device__ __forceinline__ uint32_t div(uint32_t n) const {
    return (uint32_t)(((uint64_t)__umulhi(n, m) + n) >> l);
  }
};

// ----------------------------------------------------------------------------------------------
// Powers of two built from their bit pattern (no FP64 arithmetic): valid for -1022 <= p <= 1023.
__device__ __forceinline__ double pow2_bits(int p) {
  return __hiloint2double((p + 1023) << 20, 0);
}

__host__ __device__ constexpr int ceil_log2(int q) {
  int l = 0;
  while ((1 << l) < q) ++l;
  return l;
}

// Moment sum of Q doubles, accumulated exactly in 64-bit fixed point on the integer pipes.
// Each term's 53-bit significand is placed, with G guard bits (G = 10 - ceil(log2 Q) keeps Q terms
// below 2^63), in the frame of the largest exponent present, rounding to nearest (ties up) when it
// is shifted right; the integer total is converted back to a correctly rounded double (ties to even)
// with integer operations only, times 2^P2. The error is below one unit in the last place of the
// largest |f_k| (sequential FP64 addition: up to (Q-1)/2 units). GB300 runs FP64 arithmetic and
// FP32<->FP64 conversions at ~2 per clock per SM and integer arithmetic far faster, so this takes
// the Q-1 additions of the moment sum (and the conversion) off the FP64 pipe.
// Subnormal terms beside a larger one count as zero (an error below 2^-1022 each), a sum of terms below 2^-954 is taken
// in FP64; any NaN or infinite term makes the result NaN.
constexpr unsigned kExpField = 0x7FF00000u;  // exponent field in the high word of a double

// One term in the frame of the largest exponent field emf (in place, at least kFixedLeast) with G guard bits, rounded to
// nearest (ties away from zero). With t = 2 |f| in the frame, truncated, and its sign applied as ~t = -t - 1, the
// rounded term is (t + 1) >> 1 for either sign. Zero and subnormal terms get an implicit bit too and fall
// below the frame, whose lowest bit is at least 2^(68 - 1023 - 52 - G). About 20 integer instructions a term (the
// direct form, half a unit added before the shift and the sign after it, took about 30: D3Q19 step, 994 -> 809
// instructions a node). LOW: for frames from 1 << 20 on, where subnormal terms count (two instructions more).
constexpr unsigned kFixedLeast = 68u << 20;

template <int G, bool LOW = false>
__device__ __forceinline__ long long fixed_align(double f, unsigned emf) {
  const unsigned hi = (unsigned)__double2hiint(f), lo = (unsigned)__double2loint(f), ef = hi & kExpField;
  const unsigned sh = min((emf - (LOW ? max(ef, 0x00100000u) : ef)) >> 20, 63u);
  const unsigned one = LOW ? min(ef, 0x00100000u) : 0x00100000u;  // the implicit bit
  const unsigned long long m = (((unsigned long long)((hi & 0x000FFFFFu) | one)) << 32 | lo) << (G + 1);
  const long long t = (long long)(m >> sh) ^ (long long)((int)hi >> 31);
  return (t + 1) >> 1;
}

// fixed_align of the double of a float; emaxf: largest exponent field of the floats (0 .. 254; the frame of the
// doubles is emf = (max(emaxf, 1) + 896) << 20). Truncates toward zero below the frame (2^-(53+G) of the largest).
template <int G>
__device__ __forceinline__ long long fixed_align(float f, unsigned emaxf) {
  const unsigned b = (unsigned)__float_as_int(f), e = (b >> 23) & 0xFFu;
  const unsigned m = (b & 0x007FFFFFu) | (e ? 0x00800000u : 0u);
  const unsigned sh = max(emaxf, 1u) - max(e, 1u);
  const unsigned long long v = sh < 64u ? ((unsigned long long)m << (29 + G)) >> sh : 0ull;
  const long long sg = (long long)((int)b >> 31);
  return ((long long)v ^ sg) - sg;
}

// The value of a total acc in that frame, correctly rounded (ties to even), times 2^P2.
template <int G, int P2>
__device__ __forceinline__ double fixed_value(long long acc, unsigned emf) {
  if (acc == 0) return 0.0;
  const unsigned long long sbit = acc < 0 ? 0x8000000000000000ull : 0ull;
  unsigned long long a = acc < 0 ? (unsigned long long)(-acc) : (unsigned long long)acc;
  const int lz = __clzll((long long)a);
  a <<= lz;                                  // leading one at bit 63
  unsigned long long mant = a >> 11;         // 53 bits with the leading one
  const unsigned rem = (unsigned)a & 0x7FFu; // dropped bits
  mant += (rem > 0x400u || (rem == 0x400u && (mant & 1ull))) ? 1ull : 0ull;
  int ex = (63 - lz) + (int)(emf >> 20) - 1075 - G + 1023 + P2;
  if (mant >> 53) {
    mant >>= 1;
    ++ex;
  }
  if (ex <= 0 || ex >= 2047) {  // result outside the normal range: convert and scale in two exact steps
    const int p = (int)(emf >> 20) - 1075 - G + P2;
    const int p1 = p / 2;
    return __ll2double_rn(acc) * pow2_bits(p1) * pow2_bits(p - p1);
  }
  return __longlong_as_double((long long)(sbit | ((unsigned long long)ex << 52) | (mant & 0xFFFFFFFFFFFFFull)));
}

// ZEROS: return at once for a sum of zeros (the latency of small grids' boundary kernels grows by it: adjoint of D2Q9 300^2 boxes
// in 32 bits 7.6 -> 8.2 us a step, so that k_adj_boundary does without).
template <int Q, int P2, bool ZEROS = true, class Get>
__device__ __forceinline__ double fixed_moment_sum_impl(Get f) {
  constexpr int G = 10 - ceil_log2(Q);
  static_assert(G >= 3, "too many terms for a 64-bit accumulator");
  unsigned emf = 0u;  // largest exponent field, in place (bits 20..30 of the high word)
#pragma unroll
  for (int k = 0; k < Q; ++k) emf = max(emf, (unsigned)__double2hiint(f(k)) & kExpField);
  if (emf == kExpField) return __longlong_as_double(0x7FF8000000000000ll);
  if constexpr (Q > 3) {
    if (emf < kFixedLeast) {
      // Every term below 2^-954. Zeros take no FP64 operation: summed as the tiny terms are, regions of them were stepped 1.4 to
      // 1.7 times slower than others (D3Q19 256^3: 1.26 ms, now 0.73; 1000^2: 40 us, now 23). Tiny terms in fixed point too,
      // here or in a function apart, made every step of small grids 1 to 3 % slower.
      if constexpr (ZEROS) {
        unsigned any = 0u;
#pragma unroll
        for (int k = 0; k < Q; ++k) any |= ((unsigned)__double2hiint(f(k)) & 0x7FFFFFFFu) | (unsigned)__double2loint(f(k));
        if (any == 0u) return 0.0;
      }
      double s = 0.0;
#pragma unroll
      for (int k = 0; k < Q; ++k) s += f(k);
      return s * (double)(1 << P2);
    }
  } else {  // three terms: the branch would be predicated, and its additions cost as much as if it were taken (D1Q3, 1.35 M nodes: 19.5 us a step, now 12.7)
    emf = max(emf, 0x00100000u);
  }
  long long acc = 0;
#pragma unroll
  for (int k = 0; k < Q; ++k) acc += fixed_align<G, (Q <= 3)>(f(k), emf);
  return fixed_value<G, P2>(acc, emf);
}

template <int Q, int P2, bool ZEROS = true>
__device__ __forceinline__ double fixed_moment_sum(const double (&f)[Q]) {
  return fixed_moment_sum_impl<Q, P2, ZEROS>([&](int k) { return f[k]; });
}

// Moment sum of the boundary nodes of FP32-deviation boxes in d = 4, 5: the first NFX terms in fixed point, the rest
// added on the FP64 pipe (their stored floats keep the rounding they had). The FP64 steps split their sums the same
// way while a fixed-point term took ~30 integer instructions; at ~20 the whole sum in fixed point is faster, us per step, split /
// whole: D5Q51 24^5 1021 / 930, 12^5 39.4 / 35.7, 8^5 8.8 / 8.4 (38 of 51 terms), D4Q33 boxes 32^4 106.5 / 102.0, 48^4 475 / 457 (29 of 33).
template <int Q>
constexpr int kNodeFixedTerms = Q == 51 ? 38 : (Q == 33 ? 29 : Q);

template <int Q, int NFX>
__device__ __forceinline__ double split_moment_sum(const double (&f)[Q]) {
  double s = fixed_moment_sum_impl<NFX, 0>([&](int k) { return f[k]; });
#pragma unroll
  for (int k = NFX; k < Q; ++k) s += f[k];
  return s;
}

// Double-float storage of the macroscopic variable of the FP32-deviation form: phi = h + l with h
// the value truncated to 24 significant bits and l the rounded residual (a 48-bit significand,
// relative spacing 2^-48). Neighbour differences are then plain FP32 arithmetic.
__device__ __forceinline__ double df_value(float2 p) { return (double)p.x + (double)p.y; }

__device__ __forceinline__ float2 df_split(double x) {
  const double hd = __hiloint2double(__double2hiint(x), __double2loint(x) & (int)0xE0000000);
  return make_float2((float)hd, (float)(x - hd));
}

// New pair for h + t, with h the leading part of a pair and t an FP32 increment: h' is the exact sum
// rounded toward zero to 24 significant bits, l' = (h + t) - h' rounded to nearest. TwoSum gives
// s + e = h + t exactly (s the rounded-to-nearest sum); when s was rounded away from zero it is moved
// one step toward zero, and s - h' (0 or one ulp) is exact. FP32 arithmetic only (the intrinsics
// keep the compiler from contracting or reordering the error terms).
__device__ __forceinline__ float2 df_add(float h, float t) {
  const float s = __fadd_rn(h, t);
  const float bp = __fsub_rn(s, h);
  const float e = __fadd_rn(__fsub_rn(h, __fsub_rn(s, bp)), __fsub_rn(t, bp));
  const bool away = (s > 0.0f && e < 0.0f) || (s < 0.0f && e > 0.0f);
  const float hn = away ? __int_as_float(__float_as_int(s) - 1) : s;
  return make_float2(hn, __fadd_rn(__fsub_rn(s, hn), e));
}

// The double of a float, by its bits (FP32 -> FP64 conversions retire at the FP64 pipe's ~2 per clock per SM);
// subnormals are scaled by 2^64 first. Branch-free: a branch to the conversion would be predicated, and a
// predicated conversion costs as much as one that runs.
__device__ __forceinline__ double float_to_double(float f) {
  const bool tiny = ((unsigned)__float_as_int(f) & 0x7F800000u) == 0u;
  const unsigned b = (unsigned)__float_as_int(tiny ? __fmul_rn(f, 0x1p64f) : f), mag = b & 0x7FFFFFFFu;
  const unsigned bias = tiny ? 0x34000000u : (mag >= 0x7F800000u ? 0x70000000u : 0x38000000u);
  const unsigned hi = mag == 0u ? 0u : (mag >> 3) + bias;
  return __hiloint2double((int)((b & 0x80000000u) | hi), (int)(b << 29));
}

// Arithmetic on unevaluated pairs h + l of floats (Dekker, "A floating-point technique for extending the
// available precision", Numer. Math. 18, 1971; Knuth's TwoSum): ~2^-46 of the operands, on the FP32
// pipe, which runs 64 times the FP64 pipe's rate here. The intrinsics keep the compiler from contracting.
__device__ __forceinline__ float2 ff_quick(float a, float b) {  // |a| >= |b| or a = 0
  const float s = __fadd_rn(a, b);
  return make_float2(s, __fsub_rn(b, __fsub_rn(s, a)));
}

__device__ __forceinline__ float2 ff_add(float2 a, float2 b) {
  const float s = __fadd_rn(a.x, b.x);
  const float bp = __fsub_rn(s, a.x);
  const float e = __fadd_rn(__fsub_rn(a.x, __fsub_rn(s, bp)), __fsub_rn(b.x, bp));
  return ff_quick(s, __fadd_rn(e, __fadd_rn(a.y, b.y)));
}

__device__ __forceinline__ float2 ff_neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 ff_sub(float2 a, float2 b) { return ff_add(a, ff_neg(b)); }

__device__ __forceinline__ float2 ff_mul(float2 a, float2 b) {
  const float p = __fmul_rn(a.x, b.x);
  const float e = __fmaf_rn(a.x, b.x, -p);
  return ff_quick(p, __fmaf_rn(a.x, b.y, __fmaf_rn(a.y, b.x, e)));
}

// Exponent of a double: 2^E <= |x| < 2^(E+1); -1023 for zero and subnormals, 1024 for infinities and NaN.
__device__ __forceinline__ int double_exponent(double x) { return (int)(((unsigned)__double2hiint(x) & kExpField) >> 20) - 1023; }

// df_split by integer operations, for E = double_exponent(x) <= 126: h the value truncated to 24 bits, l the rest
// rounded to nearest. Below 2^-70 the low part and below 2^-126 the whole value is taken as zero.
__device__ __forceinline__ float2 ff_split(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int E = (int)((hi & kExpField) >> 20) - 1023;
  if (E < -126) return make_float2(0.0f, 0.0f);
  const unsigned sign = hi & 0x80000000u;
  const float h = __int_as_float((int)(sign | ((unsigned)(E + 127) << 23) | ((hi & 0x000FFFFFu) << 3) | (lo >> 29)));
  const float r = (float)(lo & 0x1FFFFFFFu);
  const float sc = E >= -70 ? __int_as_float((int)(sign | ((unsigned)(E - 52 + 127) << 23))) : 0.0f;
  return make_float2(h, __fmul_rn(r, sc));
}

// Stores of the new state with the default cache policy. The evict-first hint (st.global.cs) was
// measured 0.6-1.7 % slower on every step kernel (D3Q19 256^3 FP64 744.6 vs 739.8 us, D4Q33 48^4 FP32
// deviations 252.9 vs 248.6 us), bitwise the same results.
__device__ __forceinline__ void st_stream(double *p, double v) { *p = v; }
__device__ __forceinline__ void st_stream(float *p, float v) { *p = v; }

// Programmatic dependent launch. A step kernel lets the next kernel of its stream be scheduled once
// every CTA of this one has reached pdl_trigger, and waits for the kernel before it to
// complete, with its memory visible, before it touches global memory (pdl_wait). When the kernel was
// launched without the programmatic-serialization attribute both are no-ops. A trigger on entry puts the
// next grid's CTAs wherever a place is left beside this grid's, so that a grid of about one wave ends up
// two deep on some SMs. The register kernels therefore trigger just before their stores; the FP64 step, in grids of
// about one wave (at most kTriggerCtasPerSM CTAs per SM), not before it ends. us per step with the trigger on entry /
// before the stores / at the end: FP64 D2Q9 256^2 5.93 / 3.93 / 3.66, 500 x 333 (8.6 CTAs per SM) 7.16 / 6.76 / 6.01,
// 1000^2 (51) 23.7 / 23.4 / 25.3, D3Q19 32^3 8.94 / 4.86 / 4.03, 45 x 37 x 51 9.52 / 8.12 / 6.87, 64^3 (13.5) 13.5 / 13.5 / 14.0;
// 128^3 and larger the same (the adjoint, which also updates dL/dR, is faster with the trigger at the end at every size:
// 64^3 13.7 / 13.3, 128^3 100.4 / 99.2); FP32 deviations: lhe_step_dev.cu. (A run-time choice in
// one kernel measured like the trigger at the end everywhere, so the two are separate instantiations.)
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

}  // namespace lhe
