// FP64 arithmetic of the kernels, arranged around an FP64 pipe of 2 lanes a clock and SM (1/64 of the
// FP32 rate): reciprocals and roots by short iterations, the nonlinear weights on the integer pipe.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace weno {
namespace dev {

// The special-function unit's single-precision reciprocal (1 ulp, subnormals flushed).
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

__device__ __forceinline__ uint32_t hi_word(double x) { return (uint32_t)__double2hiint(x); }

// 1/x by the third-order Householder iteration x0 (1 + e + e^2), e = 1 - x x0 (the series of 1/(1 - e)
// cut after e^2), from the seed of rcp.approx.ftz.f64 (20 bits, so e^3 < 2^-60): three FP64
// instructions, last-bit accurate.  Valid where rcp_safe(hi_word(x)); outside it the caller divides.
__device__ __forceinline__ double rcp_seed(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  return r;
}
__device__ __forceinline__ double rcp_f64(double x) {
  const double r = rcp_seed(x), e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}
// Positive normal numbers well inside the exponent range (2^-1021 <= x < 2^1021): one unsigned compare
// that zeros, subnormals, infinities, NaN and negative numbers fail.
constexpr uint32_t kHiMin = 0x00200000u, kHiMax = 0x7fc00000u;
__device__ __forceinline__ bool rcp_safe(uint32_t hi_min, uint32_t hi_max) { return hi_min >= kHiMin && hi_max < kHiMax; }

// 1/sqrt(x), last-bit accurate: with e = 1 - x y0^2 from the 20-bit seed y0 of rsqrt.approx.ftz.f64,
// 1/sqrt(x) = y0 (1 + e/2 + 3/8 e^2 + ...), the binomial series of (1 - e)^(-1/2) cut below 2^-60.
__device__ __forceinline__ double rsqrt_f64(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-(x * y), y, 1.0);
  return fma(y * e, fma(e, 0.375, 0.5), y);
}
// sqrt(x) = x / sqrt(x), from the same seed: s0 = x y0, sqrt(x) = s0 (1 + e/2 + 3/8 e^2 + ...).
__device__ __forceinline__ double sqrt_f64(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double s = x * y, e = fma(-s, y, 1.0);
  return fma(s * e, fma(e, 0.375, 0.5), s);
}
// Guarded forms: IEEE outside the range the iterations are valid in.
__device__ __noinline__ double rcp_ieee(double x) { return 1.0 / x; }
__device__ __noinline__ double sqrt_ieee(double x) { return sqrt(x); }
__device__ __noinline__ double quotient_ieee(double a, double b) { return a / b; }
__device__ __noinline__ double rsqrt_ieee(double x) { return 1.0 / sqrt(x); }
__device__ __forceinline__ double rcp_any(double x) {
  const uint32_t h = hi_word(x) & 0x7fffffffu;
  return rcp_safe(h, h) ? rcp_f64(x) : rcp_ieee(x);
}
__device__ __forceinline__ double sqrt_any(double x) {
  const uint32_t h = hi_word(x);
  return rcp_safe(h, h) ? sqrt_f64(x) : sqrt_ieee(x);
}
__device__ __forceinline__ double rsqrt_any(double x) {
  const uint32_t h = hi_word(x);
  return rcp_safe(h, h) ? rsqrt_f64(x) : rsqrt_ieee(x);
}

// Members of candidate j (slot numbers 1..M), four bits each, for a j known at run time only.
template <int M> struct SubBits;
template <> struct SubBits<12> { static constexpr uint64_t A = 0x422433114321ull, B = 0xcba987651432ull; };
template <> struct SubBits<9> { static constexpr uint64_t A = 0x213321321ull, B = 0x987654132ull; };
template <int M> __device__ __forceinline__ int sub_a(int j) { return (int)(SubBits<M>::A >> (4 * j)) & 15; }
template <int M> __device__ __forceinline__ int sub_b(int j) { return (int)(SubBits<M>::B >> (4 * j)) & 15; }

// What a Gauss point needs of one candidate: gradient, beta + eps, beta^2, beta^3.
struct CandF64 { double gx, gy, be, b2, b3; };

// beta + eps is set to infinity where beta^3 overflows, so that face_points_f64 sees it.
__device__ __forceinline__ CandF64 candidate_f64(double gx, double gy, double a0, double eps) {
  const double b = a0 * (gx * gx + gy * gy), b2 = b * b, b3 = b2 * b;
  return CandF64{gx, gy, hi_word(b3) < 0x7ff00000u ? b + eps : __longlong_as_double(0x7ff0000000000000ll), b2, b3};
}

// Positive numbers t 2^(e - 1086) with a 64-bit t (the value of a biased FP64 exponent e and a mantissa
// left-justified in t; t may have a few leading zeros): the indicators, the nonlinear weights and their
// sums are formed on the integer pipe, which the FP64 pipe never sees.  Each operation below loses less
// than 2^-58 of its result; all numbers are positive, so nothing cancels.
struct PosNum { uint64_t t; int e; };

// A positive FP64 number; zero and subnormals become about 2^-1023.
__device__ __forceinline__ PosNum pos_of(double x) {
  const uint32_t h = hi_word(x), l = (uint32_t)__double2loint(x);
  return PosNum{(uint64_t)(0x80000000u | __funnelshift_l(l, h, 11)) << 32 | (l << 11), (int)(h >> 20)};
}
// The same number in one word, for tables and shared memory: t, whose low 11 bits are zero, with the biased
// exponent in them.  Two instructions unpack it where pos_of takes four, which saves ten of the about 110 integer
// instructions a point and candidate.  33k-cell vortex step 584.8 -> 575.7 us, 53k-cell
// residual 293.6 -> 290.1, 8k-quad CFL step 245.1 -> 241.5; in characteristic variables, where no thread shares
// its indicators, 434.1 -> 437.4: it keeps FP64 weights.
struct PosWord { uint64_t bits; };
__device__ __forceinline__ PosWord pos_word(double x) {
  const uint64_t u = (uint64_t)__double_as_longlong(x);
  return PosWord{1ull << 63 | u << 11 | (u >> 52 & 0x7ffu)};
}
__device__ __forceinline__ PosNum pos_of(PosWord w) { return PosNum{w.bits & ~0x7ffull, (int)(w.bits & 0x7ffu)}; }
__device__ __forceinline__ double f64_of(PosWord w) {
  return __longlong_as_double((long long)((w.bits & 0x7ffu) << 52 | (w.bits << 1) >> 12));
}
__device__ __forceinline__ double f64_of(double x) { return x; }
struct PosPair { PosWord x, y; };  // (gamma+, gamma-)
// A candidate with its indicators in that form.
struct CandPos { double gx, gy; PosWord be, b2, b3; };

__device__ __forceinline__ PosNum pos_mul(PosNum a, PosNum b) {
  const uint32_t ah = (uint32_t)(a.t >> 32), al = (uint32_t)a.t, bh = (uint32_t)(b.t >> 32), bl = (uint32_t)b.t;
  return PosNum{(uint64_t)ah * bh + __umulhi(ah, bl) + __umulhi(al, bh), a.e + b.e - 1022};
}
__device__ __forceinline__ PosNum pos_sum(PosNum a, PosNum b) {
  const int de = a.e - b.e;
  const uint64_t big = de < 0 ? b.t : a.t, small = de < 0 ? a.t : b.t;
  return PosNum{(big >> 1) + (small >> min(abs(de) + 1, 63)), max(a.e, b.e) + 1};
}

// 2^64 / m for m = (mh, ml) / 2^63 in [1, 2), low by at most 2^-58: Newton's iteration r <- r + r (1 - r m)
// from the single-precision reciprocal's seed, biased to stay below 1/m (so that 1 - r m >= 0 and all
// products are unsigned), to 2^-38 cut to 32 bits and on to 2^-58.
__device__ __forceinline__ uint64_t recip_fixed(uint32_t mh, uint32_t ml) {
  const float seed = rcp_approx(__uint_as_float(0x3f800000u | ((mh >> 8) & 0x7fffffu)));
  const uint32_t r0 = __float_as_uint(fmaf(seed, 1.0f - 0x1p-20f, 1.0f)) << 9;  // low by 2^-21 to 2^-19
  const uint64_t e1 = (1ull << 63) - (uint64_t)r0 * mh;                         // < 2^44
  const uint32_t r1 = r0 + (__umulhi(r0, (uint32_t)(e1 >> 12)) >> 19) - 2u;     // low by at most 2^-29
  const uint64_t e2 = (1ull << 63) - ((uint64_t)r1 * mh + __umulhi(r1, ml));    // < 2^34
  return ((uint64_t)r1 << 32) + (((uint64_t)r1 * (uint32_t)(e2 >> 2)) >> 29);
}

// FP64 value of t 2^(e - 1086) with the top bit of t set, rounded to nearest (halves away from zero);
// zero below the normal range.
__device__ __forceinline__ double pos_to_f64(uint64_t t, int e) {
  const uint64_t bits = (t >> 11) + ((t >> 10) & 1u) + ((uint64_t)(uint32_t)(e - 1) << 52);
  return e <= 0 ? 0.0 : __longlong_as_double((long long)bits);
}

// gamma / d^2 for 0 <= gamma <= 1 and d in [2^-510, 2^400), good to 2^-56, with a normalised t; e_d gets
// the biased exponent of d.  gamma below 2^-1022 comes out smaller than 2^-900 of any weight that matters.
__device__ __forceinline__ PosNum pos_alpha(PosNum gamma, PosNum d, int& e_d) {
  const int ld = __clzll((long long)d.t);
  const uint64_t m = d.t << ld, r = recip_fixed((uint32_t)(m >> 32), (uint32_t)m);
  const uint32_t rh = (uint32_t)(r >> 32), rl = (uint32_t)r;
  e_d = d.e - ld;
  const PosNum s{(uint64_t)rh * rh + (((uint64_t)rh * rl) >> 31), 3068 - 2 * e_d};  // 1 / d^2
  const PosNum a = pos_mul(s, gamma);                                              // t in [2^61, 2^64)
  const int lz = __clz((int)(uint32_t)(a.t >> 32));
  return PosNum{a.t << lz, a.e - lz};
}
// The range of d above, as biased exponents.
constexpr int kAlphaExpMin = 1023 - 510, kAlphaExpMax = 1023 + 400;

// Sum of up to 16 weights: four bits of headroom in t instead of a carry, so 2^-59 of the sum is lost.
__device__ __forceinline__ PosNum pos_first(PosNum a) { return PosNum{a.t >> 4, a.e}; }
__device__ __forceinline__ PosNum pos_add(PosNum s, PosNum a) {
  const int de = s.e - a.e;
  const uint64_t t = a.t >> 4;
  const uint64_t big = de < 0 ? t : s.t, small = de < 0 ? s.t : t;
  return PosNum{big + (small >> min(abs(de), 63)), max(s.e, a.e)};
}
// Reciprocal of such a sum.
__device__ __forceinline__ double pos_rcp(PosNum s) {
  const int lz = __clzll((long long)s.t);
  const uint64_t m = s.t << lz;
  uint64_t r = recip_fixed((uint32_t)(m >> 32), (uint32_t)m);
  const int low = (int)(r >> 63) ^ 1;  // r falls just short of 2^63 where m is next to 2
  return pos_to_f64(r << low, 2041 - s.e + lz - low);
}

// Increments R(x_G) - W0 at PTS Gauss points of one face (Section 3.4), from the candidates cand(j) and
// the split weights wt(h, j) = (gamma+, gamma-) of point h (indicators and weights as FP64 or as PosWord):
//   alpha+- = gamma+- / (beta~+- + eps)^2,  beta~+- + eps = (beta + eps) + gamma (beta^2 + gamma beta^3),
//   R - W0 = sigma+ sum alpha+ p / sum alpha+  -  sigma- sum alpha- p / sum alpha-.
// Only p and the sums of alpha p are FP64, 4 instructions per point and candidate.  Returns false if an
// indicator left the range of pos_alpha (or was NaN): the increments are then redone by face_points_ieee.
template <int M, int PTS, typename Cand, typename Weights>
__device__ __forceinline__ bool face_points_f64(Cand cand, Weights wt, const double* dx, const double* dy,
                                                const double2* sig, double* incr) {
  PosNum Ap[PTS], Am[PTS];
  double Bp[PTS], Bm[PTS];
  int lo = kAlphaExpMax, hi = 0;
  auto weight = [&](auto g, PosNum be, PosNum b2, PosNum b3) {
    const PosNum gamma = pos_of(g);
    int e;
    const PosNum a = pos_alpha(gamma, pos_sum(be, pos_mul(gamma, pos_sum(b2, pos_mul(gamma, b3)))), e);
    lo = min(lo, e);
    hi = max(hi, e);
    return a;
  };
  auto one = [&](int j, bool first) {
    const auto c = cand(j);
    const PosNum be = pos_of(c.be), b2 = pos_of(c.b2), b3 = pos_of(c.b3);
#pragma unroll
    for (int h = 0; h < PTS; ++h) {
      const auto g = wt(h, j);
      const double p = c.gx * dx[h] + c.gy * dy[h];
      const PosNum ap = weight(g.x, be, b2, b3), an = weight(g.y, be, b2, b3);
      const double vp = pos_to_f64(ap.t, ap.e), vn = pos_to_f64(an.t, an.e);
      Ap[h] = first ? pos_first(ap) : pos_add(Ap[h], ap);
      Am[h] = first ? pos_first(an) : pos_add(Am[h], an);
      Bp[h] = first ? vp * p : fma(vp, p, Bp[h]);
      Bm[h] = first ? vn * p : fma(vn, p, Bm[h]);
    }
  };
  one(0, true);
#pragma unroll 2
  for (int j = 1; j < M; ++j) one(j, false);
#pragma unroll
  for (int h = 0; h < PTS; ++h) incr[h] = sig[h].x * (Bp[h] * pos_rcp(Ap[h])) - sig[h].y * (Bm[h] * pos_rcp(Am[h]));
  return lo >= kAlphaExpMin && hi < kAlphaExpMax;
}

// The same with IEEE division and the indicator as printed, beta (1 + q + q^2) with q = gamma beta:
// for indicators whose powers leave the FP64 range, and NaN states.
template <int M, int PTS, typename Cand, typename Weights>
__device__ __forceinline__ void face_points_ieee(Cand cand, Weights wt, const double* dx, const double* dy,
                                                 const double2* sig, double a0, double eps, double* incr) {
#pragma unroll
  for (int h = 0; h < PTS; ++h) {
    double Ap = 0.0, Bp = 0.0, Am = 0.0, Bm = 0.0;
#pragma unroll 1
    for (int j = 0; j < M; ++j) {
      const auto c = cand(j);
      const auto w = wt(h, j);
      const double2 g = make_double2(f64_of(w.x), f64_of(w.y));
      const double p = c.gx * dx[h] + c.gy * dy[h], b = a0 * (c.gx * c.gx + c.gy * c.gy);
      const double qp = g.x * b, qn = g.y * b;
      const double dp = b * (1.0 + qp + qp * qp) + eps, dn = b * (1.0 + qn + qn * qn) + eps;
      const double ap = g.x / (dp * dp), an = g.y / (dn * dn);
      Ap += ap;
      Bp += ap * p;
      Am += an;
      Bm += an * p;
    }
    incr[h] = sig[h].x * (Bp / Ap) - sig[h].y * (Bm / Am);
  }
}

}  // namespace dev
}  // namespace weno
