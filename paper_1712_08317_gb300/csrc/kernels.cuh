// sm_103a kernels of the WENO3 residual and the SSP-RK3 stage update.
//
//   K1 (reconstruction, Sections 3.1-3.4): candidate gradients from gathered
//                  stencil averages, smoothness indicators, split linear weights,
//                  new indicator, nonlinear weights and the Gauss-point values:
//     k_reconstruct_tma       FP32C Euler, tables staged in shared memory by TMA, one
//                             thread per (cell, variable); in characteristic variables
//                             the four lanes of a cell exchange variables by shuffles
//     k_reconstruct_f32c      FP32C scalar advection, one thread per cell
//     k_reconstruct_f64, k_reconstruct_char_f64   FP64 (kernels_f64.cuh): a
//                             thread per (cell, variable, Gauss points)
//   K2 (face fluxes, Eqs. 5-6): two Gauss points a face, rotated HLLC (Euler) or
//                  upwind (scalar), |l|/2 (F1 + F2); at reflective walls the outer
//                  state is the inner one mirrored, at inflow faces the prescribed
//                  state at the stage time: k_face_f64, k_face_f32, k_face_scalar.
//   K3 k_gather    one thread per cell: signed gather of its face fluxes
//                  (Eq. 4, no atomics) fused with the RK3 stage (Section 4).
//   K2 + K3 k_update_f32c   FP32C Euler, small meshes: fluxes, gather and stage
//                  in one pass.
//   k_advance_time after the third stage of a step: t += dt per instance.
// The reconstruction kernels take WALLS = true on meshes with reflective walls:
// stencil entries then carry momentum flips for mirror images.
//
// Layouts: state U[cell][v] (cell-major), Gauss values Wg[point][v] with the
// points of a quad at 8q..8q+7 and of a triangle at 8 nQ + 6t.., face fluxes
// F[face][v]; per-cell tables are structure-of-arrays with the cell index
// fastest, so the 4 variable threads of a cell share each table sector.
#pragma once

#include <cstdint>
#include <type_traits>
#include <cuda.h>
#include <cuda_runtime.h>

#include "arith_f64.cuh"

namespace weno {
namespace dev {

// Candidate sub-stencils S_j = {i0, a, b} (Sections 3.1 and 3.2).
template <int M> struct Sub;
template <> struct Sub<12> {
  static __device__ __forceinline__ int a(int j) { constexpr int t[12] = {1, 2, 3, 4, 1, 1, 3, 3, 4, 2, 2, 4}; return t[j]; }
  static __device__ __forceinline__ int b(int j) { constexpr int t[12] = {2, 3, 4, 1, 5, 6, 7, 8, 9, 10, 11, 12}; return t[j]; }
};
template <> struct Sub<9> {
  static __device__ __forceinline__ int a(int j) { constexpr int t[9] = {1, 2, 3, 1, 2, 3, 3, 1, 2}; return t[j]; }
  static __device__ __forceinline__ int b(int j) { constexpr int t[9] = {2, 3, 1, 4, 5, 6, 7, 8, 9}; return t[j]; }
};

// Programmatic dependent launch.  The kernels of a residual or a step are launched so that each may start
// while the one before it in the stream still runs: kernel_begin lets the next one start as soon as all
// blocks of this one have, and kernel_wait returns when everything before has finished and its writes are
// visible.  Before kernel_wait a kernel touches nothing but the solver's constant tables.  Whatever a
// kernel of the chain writes is read with plain loads (no __ldg, no __restrict__: the read-only path is
// for data constant over the kernel's life, which now begins before its predecessor's end).
// Only short kernels call kernel_begin: the FP32C fluxes, k_advance_time and the first level of the
// reductions.  A kernel that starts early fills the first SMs with room instead of spreading over all of
// them, which costs a reconstruction more than the early start brings (8,051 FP64
// quads with it in every kernel: 292 us a step instead of 272).  Before / after: 10,000 triangles in
// characteristic variables 41.0 -> 38.9 us a step, 800 triangles 22.5 -> 20.5, 133k cells 139.6 -> 136.8,
// 1.0M cells 798 -> 790, a residual of 53k FP64 cells 364 -> 349.
__device__ __forceinline__ void kernel_begin() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void kernel_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Loads of what an earlier kernel of the chain wrote, for the stencil gathers: ordinary (coherent) loads
// that the compiler may schedule freely among the other work, through a pointer that only exists after
// kernel_wait.
template <typename T>
__device__ __forceinline__ const T* after_wait(const T* p) {
  asm volatile("" : "+l"(p)::"memory");
  return p;
}
__device__ __forceinline__ float gather(const float* p) {
  float x;
  asm("ld.global.f32 %0, [%1];" : "=f"(x) : "l"(p));
  return x;
}
__device__ __forceinline__ double gather(const double* p) {
  double x;
  asm("ld.global.f64 %0, [%1];" : "=d"(x) : "l"(p));
  return x;
}

// Products that the compiler may not merge into a following addition.
__device__ __forceinline__ float mulr(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mulr(double a, double b) { return __dmul_rn(a, b); }

// Vector loads / stores of one cell's NV values.
template <typename T, int NV>
__device__ __forceinline__ void load_vec(const T* p, T w[NV]) {
#pragma unroll
  for (int v = 0; v < NV; ++v) w[v] = p[v];
}
template <>
__device__ __forceinline__ void load_vec<float, 4>(const float* p, float w[4]) {
  const float4 x = *reinterpret_cast<const float4*>(p);
  w[0] = x.x; w[1] = x.y; w[2] = x.z; w[3] = x.w;
}
template <>
__device__ __forceinline__ void load_vec<double, 4>(const double* p, double w[4]) {
  const double2 x = reinterpret_cast<const double2*>(p)[0], y = reinterpret_cast<const double2*>(p)[1];
  w[0] = x.x; w[1] = x.y; w[2] = y.x; w[3] = y.y;
}
template <typename T, int NV>
__device__ __forceinline__ void store_vec(T* p, const T w[NV]) {
#pragma unroll
  for (int v = 0; v < NV; ++v) p[v] = w[v];
}
template <>
__device__ __forceinline__ void store_vec<float, 4>(float* p, const float w[4]) {
  *reinterpret_cast<float4*>(p) = make_float4(w[0], w[1], w[2], w[3]);
}
template <>
__device__ __forceinline__ void store_vec<double, 4>(double* p, const double w[4]) {
  reinterpret_cast<double2*>(p)[0] = make_double2(w[0], w[1]);
  reinterpret_cast<double2*>(p)[1] = make_double2(w[2], w[3]);
}

// Stencil table entries: cell id in the low 29 bits; on meshes with reflective walls
// bit 30 / bit 29 mark a mirror image whose x / y momentum is reversed.
constexpr int32_t kDevFlipX = 1 << 30, kDevFlipY = 1 << 29, kDevSlotCell = (1 << 29) - 1;

// Flip mask of variable v (Euler: rho u -> bit 30, rho v -> bit 29).
template <bool WALLS, int NV>
__device__ __forceinline__ int32_t flip_mask(int v) {
  return (WALLS && NV == 4) ? (v == 1 ? kDevFlipX : (v == 2 ? kDevFlipY : 0)) : 0;
}

// Value of variable v of stencil entry `raw` (hi and, compensated, lo), momentum reversed for
// mirror images across walls.
template <typename T, int NV, bool WALLS, bool COMP>
__device__ __forceinline__ T slot_delta(const T* U, const T* Ulo, int32_t raw, int v,
                                        int32_t fm, T w0, T l0) {
  const int64_t cs = WALLS ? (raw & kDevSlotCell) : raw;
  T a = gather(U + cs * NV + v);
  T b = COMP ? gather(Ulo + cs * NV + v) : T(0);
  if (WALLS && (raw & fm)) { a = -a; b = -b; }
  return COMP ? (a - w0) + (b - l0) : a - w0;
}

// All variables of stencil entry `raw` (hi only), momentum reversed across walls.
template <typename T, bool WALLS>
__device__ __forceinline__ void slot_state4(const T* U, int32_t raw, T w[4]) {
  const int64_t cs = WALLS ? (raw & kDevSlotCell) : raw;
  load_vec<T, 4>(U + cs * 4, w);
  if (WALLS) {
    if (raw & kDevFlipX) w[1] = -w[1];
    if (raw & kDevFlipY) w[2] = -w[2];
  }
}

// Error-free sum (Knuth TwoSum): s + e = a + b exactly.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// Double-float numbers (hi + lo, |lo| <= ulp(hi)/2): ~48-bit arithmetic from FP32
// error-free transformations (Dekker / Knuth; products via fused multiply-add).
struct df { float hi, lo; };

__device__ __forceinline__ df df_norm(float s, float e) {  // fast two-sum, |s| >= |e|
  const float h = __fadd_rn(s, e);
  return df{h, __fsub_rn(e, __fsub_rn(h, s))};
}
__device__ __forceinline__ df df_add(df a, df b) {
  float s, e;
  two_sum(a.hi, b.hi, s, e);
  e = __fadd_rn(e, __fadd_rn(a.lo, b.lo));
  return df_norm(s, e);
}
__device__ __forceinline__ df df_mul(df a, df b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
  return df_norm(p, e);
}

// ---------------------------------------------------------------- K1
// FP32C variant of K1 (same arithmetic in FP32 with approximate reciprocals).
// Tables: gop4[j][q] = (o0 o1 o2 o3) of D_j^+, dg2[g][q] = x_G - c0,
// gam4[g][k][q] = gamma_{4k..4k+3}, gam1[g][q] = gamma_8 (triangles).

#ifndef WENO_K1_MIN_BLOCKS
#define WENO_K1_MIN_BLOCKS 2  // resident 256-thread blocks' worth of threads per SM the register budget is sized for
#endif

// Paired FP32 arithmetic (Blackwell f32x2): candidates j = 2k, 2k+1 share one
// instruction.  Odd M is padded with a candidate of weight 0 (it adds nothing).
__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ float2 rcp2(float2 x) { return make_float2(rcp_approx(x.x), rcp_approx(x.y)); }
__device__ __forceinline__ float2 abs2(float2 x) { return make_float2(fabsf(x.x), fabsf(x.y)); }

// Per-candidate quantities of one (cell, variable) that do not depend on the
// Gauss point, as candidate pairs: gradient (gx, gy), beta and be = beta + eps.
template <int P>
struct CandPairs {
  float2 gx[P], gy[P], b[P], be[P];
};

// Increment of one Gauss point as in gauss_increment below with every step of the nonlinear
// weights in FP64 (IEEE division), from the n candidates' (beta, p = P^1_j(x_G) - W0, gamma+,
// gamma-) in v[4n]: the fallback for weights outside the FP32 range.  Not inlined and looping at
// run time, so the FP32 path keeps its registers; it runs only at Gauss points that need it.
__device__ __noinline__ float nonlinear_increment_fp64(const float* __restrict__ v, int n, float sp, float sm,
                                                      float eps_f) {
  const double eps = eps_f;
  double Ap = 0.0, Bp = 0.0, Am = 0.0, Bm = 0.0;
  for (int j = 0; j < n; ++j) {
    const double b = v[4 * j], p = v[4 * j + 1], gp = v[4 * j + 2], gn = v[4 * j + 3];
    const double qp = gp * b, qn = gn * b;
    const double dp = b * (1.0 + qp + qp * qp) + eps, dn = b * (1.0 + qn + qn * qn) + eps;
    const double ap = gp / (dp * dp), an = gn / (dn * dn);
    Ap += ap;
    Bp += ap * p;
    Am += an;
    Bm += an * p;
  }
  return (float)((double)sp * (Bp / Ap) - (double)sm * (Bm / Am));
}

constexpr float kAlphaMin = 1e-30f;  // smallest sum of alpha the FP32 weights accept (see gauss_increment)

// Nonlinear weights of one candidate pair (or, scalar, of one candidate) at one Gauss point:
// alpha+- = gamma+- / (beta~+- + eps)^2 with beta~+- = beta (1 + q + q^2), q = gamma+- beta.
__device__ __forceinline__ void pair_alpha(float2 gp, float2 gn, float2 b, float2 be, float2& ap, float2& an) {
  const float2 qp = __fmul2_rn(gp, b), qn = __fmul2_rn(gn, b);
  const float2 dp = __ffma2_rn(b, __ffma2_rn(qp, qp, qp), be);   // beta~+ + eps
  const float2 dn = __ffma2_rn(b, __ffma2_rn(qn, qn, qn), be);   // beta~- + eps
  ap = __fmul2_rn(gp, rcp2(__fmul2_rn(dp, dp)));
  an = __fmul2_rn(gn, rcp2(__fmul2_rn(dn, dn)));
}
__device__ __forceinline__ void one_alpha(float gp, float gn, float b, float be, float& ap, float& an) {
  const float qp = gp * b, qn = gn * b;
  const float dp = fmaf(b, fmaf(qp, qp, qp), be), dn = fmaf(b, fmaf(qn, qn, qn), be);
  ap = gp * rcp_approx(dp * dp);
  an = gn * rcp_approx(dn * dn);
}

// Increment R(x_G) - W0 of one Gauss point (Section 3.4, FP32) from the
// candidate pairs and the split linear weights gamma+ (gpos), gamma- (gneg)
// with their sums sigma+- (sp, sm), which depend on geometry only and are
// precomputed in FP64:
//   R - W0 = sigma+ sum delta+ p - sigma- sum delta- p,
//   delta+-_j = alpha+-_j / sum alpha+-, alpha+-_j = gamma+-_j / (beta~+-_j + eps)^2,
//   beta~+-_j = beta_j (1 + q + q^2), q = gamma+-_j beta_j.
// The linear scheme is R - W0 = sum gamma_j p_j = sigma+ sum gamma+ p - sigma- sum gamma- p.
// With M odd the last candidate (the .x lane of the last pair) is evaluated in scalar arithmetic.
template <int M>
__device__ __forceinline__ float gauss_increment(const CandPairs<(M + 1) / 2>& c, const float2* gpos,
                                                 const float2* gneg, float dx, float dy, float sp, float sm,
                                                 int linear, float& amin) {
  constexpr int P = (M + 1) / 2, FULL = M / 2;
  amin = 1.0f;
  const float2 dx2 = f2(dx, dx), dy2 = f2(dy, dy);
  if (linear) {
    float2 ap = f2(0.f, 0.f), an = f2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < P; ++k) {
      const float2 p = __ffma2_rn(c.gx[k], dx2, __fmul2_rn(c.gy[k], dy2));
      ap = __ffma2_rn(gpos[k], p, ap);
      an = __ffma2_rn(gneg[k], p, an);
    }
    return sp * (ap.x + ap.y) - sm * (an.x + an.y);
  }
  // sums of alpha+- and alpha+- p: pair 0 initialises them, later pairs add
  float2 Ap, Bp, Am, Bm;
#pragma unroll
  for (int k = 0; k < FULL; ++k) {
    const float2 p = __ffma2_rn(c.gx[k], dx2, __fmul2_rn(c.gy[k], dy2));  // P^1_j(x_G) - W0
    float2 ap, an;
    pair_alpha(gpos[k], gneg[k], c.b[k], c.be[k], ap, an);
    if (k == 0) {
      Ap = ap; Bp = __fmul2_rn(ap, p);
      Am = an; Bm = __fmul2_rn(an, p);
    } else {
      Ap = __fadd2_rn(Ap, ap); Bp = __ffma2_rn(ap, p, Bp);
      Am = __fadd2_rn(Am, an); Bm = __ffma2_rn(an, p, Bm);
    }
  }
  float As = Ap.x + Ap.y, Bs = Bp.x + Bp.y, Ams = Am.x + Am.y, Bms = Bm.x + Bm.y;
  if constexpr (M % 2 == 1) {
    const float p = fmaf(c.gx[P - 1].x, dx, c.gy[P - 1].x * dy);
    float ap, an;
    one_alpha(gpos[P - 1].x, gneg[P - 1].x, c.b[P - 1].x, c.be[P - 1].x, ap, an);
    As += ap; Bs = fmaf(ap, p, Bs);
    Ams += an; Bms = fmaf(an, p, Bms);
  }
  // The smaller sum of alpha of the two groups: the caller redoes the Gauss point in FP64 when it
  // falls below kAlphaMin (indicators of order 1e6 and more, whose (beta~ + eps)^2 overflows FP32
  // or whose reciprocal flushes).  Above it every candidate that matters is far from both limits;
  // the sums never exceed 1 / eps^2 <= 1e30, since eps >= 1e-15 for FP32 weights.
  amin = fminf(As, Ams);
  return sp * Bs * rcp_approx(As) - sm * Bms * rcp_approx(Ams);
}

// gauss_increment with the nonlinear weights in FP64, whose range holds every finite FP32
// beta; delta = alpha / sum alpha is the same function, so only rounding differs.
template <int P>
__device__ __forceinline__ float gauss_increment_fp64(const CandPairs<P>& c, const float2* gpos, const float2* gneg,
                                                      float dx, float dy, float sp, float sm, float eps) {
  const float2 dx2 = f2(dx, dx), dy2 = f2(dy, dy);
  float v[8 * P];
#pragma unroll
  for (int k = 0; k < P; ++k) {
    const float2 p = __ffma2_rn(c.gx[k], dx2, __fmul2_rn(c.gy[k], dy2));
    v[8 * k + 0] = c.b[k].x; v[8 * k + 1] = p.x; v[8 * k + 2] = gpos[k].x; v[8 * k + 3] = gneg[k].x;
    v[8 * k + 4] = c.b[k].y; v[8 * k + 5] = p.y; v[8 * k + 6] = gpos[k].y; v[8 * k + 7] = gneg[k].y;
  }
  return nonlinear_increment_fp64(v, 2 * P, sp, sm, eps);
}

// Candidate gradients and smoothness indicators of one (cell, variable), as
// candidate pairs (the padding candidate of odd M has g = 0, beta = 0).
template <int NV, int M, bool WALLS>
__device__ __forceinline__ void cell_gradients(const float* U, const float* Ulo,
                                               const int32_t* __restrict__ slot, int64_t slot_pitch,
                                               const float4* __restrict__ gop4, int64_t pitch, int64_t q, int64_t c,
                                               int v, float a0, float eps, float& w0, float& l0,
                                               CandPairs<(M + 1) / 2>& cp) {
  w0 = gather(U + c * NV + v);
  l0 = gather(Ulo + c * NV + v);
  float dW[M + 1];
  dW[0] = 0.0f;
  const int32_t fm = flip_mask<WALLS, NV>(v);
#pragma unroll
  for (int s = 1; s <= M; ++s)
    dW[s] = slot_delta<float, NV, WALLS, true>(U, Ulo, __ldg(slot + (int64_t)(s - 1) * slot_pitch + q), v, fm, w0, l0);
  float gx[2 * ((M + 1) / 2)], gy[2 * ((M + 1) / 2)], b[2 * ((M + 1) / 2)];
#pragma unroll
  for (int j = 0; j < M; ++j) {
    const float da = dW[Sub<M>::a(j)], db = dW[Sub<M>::b(j)];
    const float4 m = __ldg(gop4 + (int64_t)j * pitch + q);
    gx[j] = fmaf(m.x, da, m.y * db);
    gy[j] = fmaf(m.z, da, m.w * db);
    b[j] = a0 * fmaf(gx[j], gx[j], gy[j] * gy[j]);
  }
  if (M % 2) { gx[M] = 0.f; gy[M] = 0.f; b[M] = 0.f; }
#pragma unroll
  for (int k = 0; k < (M + 1) / 2; ++k) {
    cp.gx[k] = f2(gx[2 * k], gx[2 * k + 1]);
    cp.gy[k] = f2(gy[2 * k], gy[2 * k + 1]);
    const float2 bb = f2(b[2 * k], b[2 * k + 1]);
    cp.b[k] = bb;
    cp.be[k] = __fadd2_rn(bb, f2(eps, eps));
  }
}

// FP32C tables (rows of `pitch` cells): gop4[j] = D_j^+ entries; dgs[g] =
// (x_G - c0, sigma+, sigma-); gpm4[g][k] = gamma+_{4k..4k+3} for k < M/4 and
// gamma-_{4(k-M/4)..} after them; g1[g] = (gamma+_8, gamma-_8) for triangles.
template <int NV, int M, int G>
__global__ void __launch_bounds__(256, WENO_K1_MIN_BLOCKS) k_reconstruct_f32c(
    const float* U, const float* Ulo, const int32_t* __restrict__ slot,
    const float4* __restrict__ gop4, const float4* __restrict__ dgs, const float4* __restrict__ gpm4,
    const float2* __restrict__ g1, const float* __restrict__ area, int64_t N, int64_t pitch, int64_t first,
    int64_t gbase, float* Wg, float eps, int linear) {
  constexpr int M4 = M / 4, P = (M + 1) / 2;
  kernel_wait();
  U = after_wait(U);
  Ulo = after_wait(Ulo);
  const int64_t total = N * NV;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t q = t / NV;
    const int v = (int)(t - q * NV);
    const int64_t c = first + q;
    float w0, l0;
    CandPairs<P> cp;
    cell_gradients<NV, M, false>(U, Ulo, slot, N, gop4, pitch, q, c, v, __ldg(area + c), eps, w0, l0, cp);
    float* out = Wg + (gbase + q * G) * NV + v;
    // (x_G - c0, sigma+-) and the split weights of Gauss point g
    auto tables = [&](int g, float4& d, float2* gp, float2* gn) {
      d = __ldg(dgs + (int64_t)g * pitch + q);
#pragma unroll
      for (int k = 0; k < M4; ++k) {
        const float4 x = __ldg(gpm4 + (int64_t)(g * 2 * M4 + k) * pitch + q);
        const float4 y = __ldg(gpm4 + (int64_t)(g * 2 * M4 + M4 + k) * pitch + q);
        gp[2 * k] = f2(x.x, x.y); gp[2 * k + 1] = f2(x.z, x.w);
        gn[2 * k] = f2(y.x, y.y); gn[2 * k + 1] = f2(y.z, y.w);
      }
      if (M % 4) {
        const float2 e = __ldg(g1 + (int64_t)g * pitch + q);
        gp[P - 1] = f2(e.x, 0.f);
        gn[P - 1] = f2(e.y, 0.f);
      }
    };
    float amin = 1.0f;  // smallest sum of alpha over the Gauss points
#pragma unroll 1
    for (int g = 0; g < G; ++g) {
      float4 d;
      float2 gp[P], gn[P];
      tables(g, d, gp, gn);
      float am;
      const float incr = gauss_increment<M>(cp, gp, gn, d.x, d.y, d.z, d.w, linear, am);
      amin = fminf(amin, am);
      out[(int64_t)g * NV] = w0 + (l0 + incr);
    }
    if (!(amin >= kAlphaMin)) {  // weights outside the FP32 range (rare): every point again in FP64
#pragma unroll 1
      for (int g = 0; g < G; ++g) {
        float4 d;
        float2 gp[P], gn[P];
        tables(g, d, gp, gn);
        out[(int64_t)g * NV] = w0 + (l0 + gauss_increment_fp64<P>(cp, gp, gn, d.x, d.y, d.z, d.w, eps));
      }
    }
  }
}

// ---------------------------------------------------------------- K1 with TMA-staged tables
// Euler FP32C, one block per tile or persistent: a tile is TILE consecutive cells of one type,
// one (cell, variable) per thread.  One elected thread loads the tile's split
// linear weights, Gauss offsets and gradient operators into shared memory with
// 2D TMA copies (cp.async.bulk.tensor) completing on an mbarrier; the stencil
// gathers of the tile are issued before the wait.  The next tile's copy starts
// when the block has finished reading the current one, and the other resident
// blocks hide its latency.  Every wait is bounded: on timeout the block
// records *err = 1 and exits (its one copy has completed or is abandoned with
// the block's shared memory).
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ uint64_t globaltimer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
constexpr uint64_t kWaitLimitNs = 1000000000ull;  // 1 s: far beyond any copy's latency
// Waits for the barrier phase; gives up after kWaitLimitNs (or 2^26 polls) and returns false.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = globaltimer_ns();
  for (int it = 1; it < (1 << 26); ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((it & 255) == 0 && globaltimer_ns() - t0 > kWaitLimitNs) return false;
  }
  return false;
}
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          smem_addr(dst)),
      "l"((uint64_t)map), "r"(x), "r"(y), "r"(smem_addr(bar))
      : "memory");
}

// The same; the lines are the first to leave L2.
__device__ __forceinline__ void tma_load_2d_once(void* dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
  uint64_t policy;
  asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3}], "
      "[%4], %5;" ::"r"(smem_addr(dst)),
      "l"((uint64_t)map), "r"(x), "r"(y), "r"(smem_addr(bar)), "l"(policy)
      : "memory");
}

#ifndef WENO_K1_TILE
#define WENO_K1_TILE 16  // cells per block tile of the TMA reconstruction (8, 16, 32 or 64)
#endif
#ifndef WENO_K1_DG_LDS
#define WENO_K1_DG_LDS 0  // 1: the TMA reconstruction re-reads the Gauss offsets from shared memory
#endif
static_assert(WENO_K1_TILE == 8 || WENO_K1_TILE == 16 || WENO_K1_TILE == 32 || WENO_K1_TILE == 64, "tile of 8, 16, 32 or 64 cells");

// Tables of the Euler FP32C reconstruction, staged per tile: the G Gauss points of a cell are taken
// as G/2 pairs (the two points of one face), whose values share a float2.  Rows of TILE float4:
//   gam [k][j]  (gamma+_j, gamma+_j', gamma-_j, gamma-_j') at points 2k and 2k+1 (split, normalised)
//   dg  [2k]    (dx, dx', dy, dy')    x_G - c0 of the two points
//   dg  [2k+1]  (sigma+, sigma+', sigma-, sigma-')
//   gop [j]     D_j^+ (the 2x2 operator from the sub-stencil's differences to the gradient)
template <int M, int G>
struct PairTile {
  static constexpr int TILE = WENO_K1_TILE;  // cells per tile; TILE x 4 threads (one per variable)
  static constexpr int THREADS = TILE * 4;
  static constexpr int NP = G / 2;
  static constexpr int GAM = NP * M * TILE * 16;
  static constexpr int DG = G * TILE * 16;
  static constexpr int GOP = M * TILE * 16;
  static constexpr int STAGE = GAM + DG + GOP;  // bytes, multiple of 128
};

// Indicators are clamped to kBetaMax before beta^2 and beta^3 are formed (below).  A candidate
// with beta that large has alpha = gamma / (beta~ + eps)^2 < 1e-40 whether clamped or not, i.e.
// zero in FP32; where every candidate of a group is that large, the sum of alpha is zero and the
// cell is redone with FP64 weights, from the unclamped value.
constexpr float kBetaMax = 1e12f;

// All G Gauss values of one (cell, variable) from its stencil differences dW (dW[0] = 0) and the
// tile's tables, FP32 arithmetic (Sections 3.1-3.4):
//   g_j = D_j^+ (dW_a, dW_b),  beta_j = |Omega| |g_j|^2,  p_j = g_j . (x_G - c0) = P^1_j(x_G) - W0,
//   beta~+-_j + eps = beta (1 + q + q^2) + eps, q = gamma+-_j beta, evaluated as the polynomial
//   (beta + eps) + gamma (beta^2 + gamma beta^3) in gamma,
//   alpha+-_j = gamma+-_j / (beta~+-_j + eps)^2,
//   R - W0 = sigma+ sum alpha+ p / sum alpha+  -  sigma- sum alpha- p / sum alpha-
// (the linear scheme: sigma+ sum gamma+ p - sigma- sum gamma- p).  Candidates are the outer loop,
// and the two points of a face share the paired FP32 instructions, so the per-point sums are the
// only state kept across candidates.  Returns false if a sum of alpha fell below kAlphaMin: the
// caller then has the cell redone with FP64 weights.  From finite inputs the sums are finite (the
// clamp below keeps beta^3 finite, and an overflowing square gives alpha = 0); a NaN sum comes from
// a NaN state, which FP64 weights cannot mend, and is left to the caller's state check.
template <int M, int G>
__device__ __forceinline__ bool pair_points(const float4* __restrict__ sgam, const float4* __restrict__ sdg,
                                            const float4* __restrict__ sgo, int cl, const float* dW, float a0,
                                            float eps, int linear, float w0, float l0, float* __restrict__ out) {
  constexpr int NP = G / 2, TILE = WENO_K1_TILE;
  float2 Ap[NP], Bp[NP], Am[NP], Bm[NP];
#if WENO_K1_DG_LDS
  // the offsets of face k's points, read from shared memory where they are used (fewer registers)
  auto DX = [&](int k) { const float4 r = sdg[(2 * k) * TILE + cl]; return f2(r.x, r.y); };
  auto DY = [&](int k) { const float4 r = sdg[(2 * k) * TILE + cl]; return f2(r.z, r.w); };
#else
  float2 dx[NP], dy[NP];
#pragma unroll
  for (int k = 0; k < NP; ++k) {
    const float4 r = sdg[(2 * k) * TILE + cl];
    dx[k] = f2(r.x, r.y);
    dy[k] = f2(r.z, r.w);
  }
  auto DX = [&](int k) { return dx[k]; };
  auto DY = [&](int k) { return dy[k]; };
#endif
#pragma unroll
  for (int k = 0; k < NP; ++k) {
    Ap[k] = f2(0.f, 0.f); Bp[k] = f2(0.f, 0.f);
    Am[k] = f2(0.f, 0.f); Bm[k] = f2(0.f, 0.f);
  }
  if (linear) {
#pragma unroll
    for (int j = 0; j < M; ++j) {
      const float4 m = sgo[j * TILE + cl];
      const float da = dW[Sub<M>::a(j)], db = dW[Sub<M>::b(j)];
      const float gx = fmaf(m.x, da, m.y * db), gy = fmaf(m.z, da, m.w * db);
      const float2 GX = f2(gx, gx), GY = f2(gy, gy);
#pragma unroll
      for (int k = 0; k < NP; ++k) {
        const float4 g4 = sgam[(k * M + j) * TILE + cl];
        const float2 p = __ffma2_rn(GX, DX(k), __fmul2_rn(GY, DY(k)));
        Bp[k] = __ffma2_rn(f2(g4.x, g4.y), p, Bp[k]);
        Bm[k] = __ffma2_rn(f2(g4.z, g4.w), p, Bm[k]);
      }
    }
#pragma unroll
    for (int k = 0; k < NP; ++k) {
      const float4 s = sdg[(2 * k + 1) * TILE + cl];
      out[(2 * k) * 4] = w0 + (l0 + (s.x * Bp[k].x - s.z * Bm[k].x));
      out[(2 * k + 1) * 4] = w0 + (l0 + (s.y * Bp[k].y - s.w * Bm[k].y));
    }
    return true;
  }
#pragma unroll
  for (int j = 0; j < M; ++j) {
    const float4 m = sgo[j * TILE + cl];
    const float da = dW[Sub<M>::a(j)], db = dW[Sub<M>::b(j)];
    const float gx = fmaf(m.x, da, m.y * db), gy = fmaf(m.z, da, m.w * db);
    const float b0 = a0 * fmaf(gx, gx, gy * gy);
    const float b = b0 > kBetaMax ? kBetaMax : b0;  // keeps a NaN (fminf would drop it)
    const float b2 = b * b, b3 = b2 * b, be = b + eps;
    const float2 GX = f2(gx, gx), GY = f2(gy, gy), C0 = f2(be, be), C1 = f2(b2, b2), C2 = f2(b3, b3);
#pragma unroll
    for (int k = 0; k < NP; ++k) {
      const float4 g4 = sgam[(k * M + j) * TILE + cl];
      const float2 gp = f2(g4.x, g4.y), gn = f2(g4.z, g4.w);
      const float2 p = __ffma2_rn(GX, DX(k), __fmul2_rn(GY, DY(k)));
      const float2 dp = __ffma2_rn(gp, __ffma2_rn(gp, C2, C1), C0);  // beta~+ + eps at both points
      const float2 dn = __ffma2_rn(gn, __ffma2_rn(gn, C2, C1), C0);
      const float2 ap = __fmul2_rn(gp, rcp2(__fmul2_rn(dp, dp)));
      const float2 an = __fmul2_rn(gn, rcp2(__fmul2_rn(dn, dn)));
      Ap[k] = __fadd2_rn(Ap[k], ap);
      Bp[k] = __ffma2_rn(ap, p, Bp[k]);
      Am[k] = __fadd2_rn(Am[k], an);
      Bm[k] = __ffma2_rn(an, p, Bm[k]);
    }
  }
  // Above kAlphaMin every candidate that matters is far from both FP32 limits; the sums never
  // exceed 1 / eps^2 <= 1e30, since eps >= 1e-15 for FP32 weights.
  bool ok = true;
#pragma unroll
  for (int k = 0; k < NP; ++k) {
    const float4 s = sdg[(2 * k + 1) * TILE + cl];
    ok = ok && !(Ap[k].x < kAlphaMin) && !(Ap[k].y < kAlphaMin) && !(Am[k].x < kAlphaMin) && !(Am[k].y < kAlphaMin);
    const float i0 = s.x * Bp[k].x * rcp_approx(Ap[k].x) - s.z * Bm[k].x * rcp_approx(Am[k].x);
    const float i1 = s.y * Bp[k].y * rcp_approx(Ap[k].y) - s.w * Bm[k].y * rcp_approx(Am[k].y);
    out[(2 * k) * 4] = w0 + (l0 + i0);
    out[(2 * k + 1) * 4] = w0 + (l0 + i1);
  }
  return ok;
}

// The tables of one cell type as 2D tensor maps (rows of PairTile).
struct TileMaps { CUtensorMap gam, dg, gop; };

// What the tiles of one cell type work on; q counts the cells of the type, cell q is first + q and its
// Gauss values start at point gbase + q G.
struct TileCells {
  const float *U, *Ulo, *area;
  const int32_t* slot;  // [slot - 1][q]
  int64_t N, first, gbase;
  float* Wg;
  float eps, gas_gamma;
  int linear;
};

// Copies of a tile's tables into shared memory, completing on the barrier.  A pass reads each table once:
// with `once` they leave L2 before what the kernels of a stage hand to one another (see tables_once).
template <int M, int G>
__device__ __forceinline__ void load_tile(unsigned char* smem, const TileMaps* maps, int64_t tile, uint64_t* bar, int once) {
  using L = PairTile<M, G>;
  const int x = (int)(tile * L::TILE * 4);
  mbar_expect_tx(bar, L::STAGE);
  if (once) {
    tma_load_2d_once(smem, &maps->gam, x, 0, bar);
    tma_load_2d_once(smem + L::GAM, &maps->dg, x, 0, bar);
    tma_load_2d_once(smem + L::GAM + L::DG, &maps->gop, x, 0, bar);
  } else {
    tma_load_2d(smem, &maps->gam, x, 0, bar);
    tma_load_2d(smem + L::GAM, &maps->dg, x, 0, bar);
    tma_load_2d(smem + L::GAM + L::DG, &maps->gop, x, 0, bar);
  }
}

// The cells whose sums of alpha left the FP32 range are redone with FP64 weights within the pass, each by
// its whole warp: lane (variable v = lane % 4, Gauss point lane / 4), so that a cell costs about 300 FP64
// instructions in a row and not 8 times as many in 4 lanes.  The warp comes here together; the tile's
// tables are still in shared memory and the stencil is gathered again (fix_cell, fix_cell_char; not
// inlined, so that the pass keeps its registers: 122 and 80 as without it).  A launch of its own for the
// marked cells cost 3 to 4 us a pass where nothing was marked, which is most passes.  dU(s) is the lane's
// difference of stencil slot s.
template <int M, int G, typename Diff>
__device__ __forceinline__ float fix_increment(const float4* __restrict__ sgam, const float4* __restrict__ sdg,
                                               const float4* __restrict__ sgo, int cl, int g, Diff dU, float a0,
                                               float eps) {
  constexpr int TILE = WENO_K1_TILE;
  const int k = g >> 1;
  const bool h = g & 1;
  const float4 r = sdg[(2 * k) * TILE + cl], s = sdg[(2 * k + 1) * TILE + cl];
  const double dx = h ? r.y : r.x, dy = h ? r.w : r.z;
  const double2 sig = make_double2(h ? s.y : s.x, h ? s.w : s.z);
  auto cand = [&](int j) {
    const float4 m = sgo[j * TILE + cl];
    const float da = dU(sub_a<M>(j)), db = dU(sub_b<M>(j));
    const float gx = fmaf(m.x, da, m.y * db), gy = fmaf(m.z, da, m.w * db);
    return candidate_f64((double)gx, (double)gy, (double)a0, (double)eps);
  };
  auto weights = [&](int, int j) {
    const float4 w = sgam[(k * M + j) * TILE + cl];
    return h ? make_double2(w.y, w.w) : make_double2(w.x, w.z);
  };
  double incr;
  if (!face_points_f64<M, 1>(cand, weights, &dx, &dy, &sig, &incr))
    face_points_ieee<M, 1>(cand, weights, &dx, &dy, &sig, (double)a0, (double)eps, &incr);
  return (float)incr;
}

template <int M, int G, bool WALLS>
__device__ __noinline__ void fix_cell(const unsigned char* smem, const TileCells& t, int64_t q, int cl) {
  using L = PairTile<M, G>;
  const int lane = threadIdx.x & 31, v = lane & 3, g = min(lane >> 2, G - 1);
  const int64_t c = t.first + q;
  const float *U = after_wait(t.U), *Ulo = after_wait(t.Ulo);
  const float w0 = gather(U + c * 4 + v), l0 = gather(Ulo + c * 4 + v);
  const int32_t fm = flip_mask<WALLS, 4>(v);
  float dW[M + 1];
#pragma unroll 1
  for (int s = 1; s <= M; ++s)
    dW[s] = slot_delta<float, 4, WALLS, true>(U, Ulo, __ldg(t.slot + (int64_t)(s - 1) * t.N + q), v, fm, w0, l0);
  const float4* sgam = reinterpret_cast<const float4*>(smem);
  const float incr = fix_increment<M, G>(sgam, sgam + L::GAM / 16, sgam + (L::GAM + L::DG) / 16, cl, g,
                                         [&](int s) { return dW[s]; }, __ldg(t.area + c), t.eps);
  if (lane < 4 * G) t.Wg[(t.gbase + q * G + g) * 4 + v] = w0 + (l0 + incr);
}

// Calls fix(q, cell of the tile) for each cell of the tile with a lane that has `bad` set, on the warp of the
// first TILE x 4 threads that holds it: lanes 4i..4i+3 of warp w hold cell 8w + i of the tile.  With PARTS > 1
// the block has that many warps for every such cell, which agree on it first.  The redone values go to the
// addresses of the cell's regular ones and are stored by other lanes; the barriers (a vote orders no memory)
// put them after those.
template <int PARTS, typename Fix>
__device__ __forceinline__ void fix_marked(bool bad, int64_t q0, Fix fix) {
  constexpr int WARPS = WENO_K1_TILE / 8;
  uint32_t m = __ballot_sync(0xffffffffu, bad);
  const int w = threadIdx.x >> 5;
  if constexpr (PARTS > 1) {
    if (!__syncthreads_or((int)m)) return;
    __shared__ uint32_t marks[PARTS * WARPS];
    if ((threadIdx.x & 31) == 0) marks[w] = m;
    __syncthreads();
    if (w >= WARPS) return;
    for (int i = 1; i < PARTS; ++i) m |= marks[w + i * WARPS];
  }
  if (m) __syncwarp();
  while (m) {
    const int i = (__ffs(m) - 1) >> 2;
    m &= ~(0xfu << (4 * i));
    const int cl = 8 * w + i;
    fix(q0 + cl, cl);
  }
}

// One tile, component-wise.  Returns false if the wait for its tables timed out.
template <int M, int G, bool WALLS>
__device__ __forceinline__ bool tile_points(const unsigned char* smem, uint64_t* bar, uint32_t phase, const TileCells& t,
                                            int64_t tile) {
  using L = PairTile<M, G>;
  const int cl = threadIdx.x >> 2, v = threadIdx.x & 3;
  const int64_t q = tile * L::TILE + cl;
  const bool act = q < t.N;
  const float4* sgam = reinterpret_cast<const float4*>(smem);
  const float4* sdg = sgam + L::GAM / 16;
  const float4* sgo = sdg + L::DG / 16;
  // stencil gathers (independent of the staged tables) before the wait
  float w0 = 0.f, l0 = 0.f, a0 = 0.f, dW[M + 1];
  dW[0] = 0.f;
  const float *U = after_wait(t.U), *Ulo = after_wait(t.Ulo);
  if (act) {
    const int64_t c = t.first + q;
    w0 = gather(U + c * 4 + v);
    l0 = gather(Ulo + c * 4 + v);
    const int32_t fm = flip_mask<WALLS, 4>(v);
#pragma unroll
    for (int s = 1; s <= M; ++s)
      dW[s] = slot_delta<float, 4, WALLS, true>(U, Ulo, __ldg(t.slot + (int64_t)(s - 1) * t.N + q), v, fm, w0, l0);
    a0 = __ldg(t.area + c);
  }
  const bool ok = mbar_wait_bounded(bar, phase);
  if (__syncthreads_or(!ok)) return false;
  bool bad = false;
  if (act)
    bad = !pair_points<M, G>(sgam, sdg, sgo, cl, dW, a0, t.eps, t.linear, w0, l0, t.Wg + (t.gbase + q * G) * 4 + v);
  fix_marked<1>(bad, tile * L::TILE, [&](int64_t qf, int cf) { fix_cell<M, G, WALLS>(smem, t, qf, cf); });
  return true;
}

// Euler (Section 4): the Gauss points of local face k are reconstructed in the
// characteristic variables of the normal flux Jacobian at the Roe average of
// the cell and its neighbour across face k (stencil slot k+1; the cell itself
// at an outflow boundary).  Four consecutive lanes hold one cell; lane l
// gathers variable l of the stencil, projects the stencil differences onto
// field l with row l of R^-1 (lane shuffles bring the other variables),
// reconstructs field l, and returns variable l of W0 + R dU with row l of R.
// Reconstructing the increment dU (zero for constant data) keeps constant
// states exact whatever the rounding of R R^-1.
// Products here are rounded or inside an explicit fma, so that the instances of the kernel (one that walks
// the faces and keeps the cell's part of a frame, one with a thread for each) give the same bits.
__device__ __forceinline__ float lane_sum4(const float c[4], float x, int base) {
  float r = mulr(c[0], __shfl_sync(0xffffffffu, x, base));
#pragma unroll
  for (int i = 1; i < 4; ++i) r = fmaf(c[i], __shfl_sync(0xffffffffu, x, base + i), r);
  return r;
}

// Roe frame of one face for lane l: row l of R^-1 (Lr) and row l of R (Rr), fields ordered
// q_n - a, entropy, shear, q_n + a, from the two cells' averages and the outward unit normal.
__device__ __forceinline__ void roe_rows(const float Wl[4], const float Wr[4], float nx, float ny, float gm1, int l,
                                         float Lr[4], float Rr[4]) {
  const float rl = Wl[0], ul = Wl[1] / rl, vl = Wl[2] / rl;
  const float hl = fmaf(gm1, fmaf(-mulr(0.5f, rl), fmaf(ul, ul, mulr(vl, vl)), Wl[3]), Wl[3]) / rl;
  const float rr = Wr[0], ur = Wr[1] / rr, vr = Wr[2] / rr;
  const float hr = fmaf(gm1, fmaf(-mulr(0.5f, rr), fmaf(ur, ur, mulr(vr, vr)), Wr[3]), Wr[3]) / rr;
  const float sl = sqrtf(rl), sr = sqrtf(rr), iw = 1.f / (sl + sr);
  const float u = mulr(fmaf(sl, ul, mulr(sr, ur)), iw), v = mulr(fmaf(sl, vl, mulr(sr, vr)), iw);
  const float H = mulr(fmaf(sl, hl, mulr(sr, hr)), iw);
  const float kin = mulr(0.5f, fmaf(u, u, mulr(v, v)));
  const float a = sqrtf(mulr(gm1, H - kin)), ia = 1.f / a;
  const float qn = fmaf(u, nx, mulr(v, ny)), qt = fmaf(v, nx, -mulr(u, ny));
  const float b1 = mulr(mulr(gm1, ia), ia), b2 = mulr(b1, kin);
  if (l == 0) {
    Lr[0] = mulr(0.5f, fmaf(qn, ia, b2)); Lr[1] = mulr(-0.5f, fmaf(b1, u, mulr(nx, ia)));
    Lr[2] = mulr(-0.5f, fmaf(b1, v, mulr(ny, ia))); Lr[3] = mulr(0.5f, b1);
    Rr[0] = 1.f; Rr[1] = 1.f; Rr[2] = 0.f; Rr[3] = 1.f;
  } else if (l == 1) {
    Lr[0] = 1.f - b2; Lr[1] = mulr(b1, u); Lr[2] = mulr(b1, v); Lr[3] = -b1;
    Rr[0] = fmaf(-a, nx, u); Rr[1] = u; Rr[2] = -ny; Rr[3] = fmaf(a, nx, u);
  } else if (l == 2) {
    Lr[0] = -qt; Lr[1] = -ny; Lr[2] = nx; Lr[3] = 0.f;
    Rr[0] = fmaf(-a, ny, v); Rr[1] = v; Rr[2] = nx; Rr[3] = fmaf(a, ny, v);
  } else {
    Lr[0] = mulr(0.5f, fmaf(-qn, ia, b2)); Lr[1] = mulr(0.5f, fmaf(nx, ia, -mulr(b1, u)));
    Lr[2] = mulr(0.5f, fmaf(ny, ia, -mulr(b1, v))); Lr[3] = mulr(0.5f, b1);
    Rr[0] = fmaf(-a, qn, H); Rr[1] = kin; Rr[2] = qt; Rr[3] = fmaf(a, qn, H);
  }
}

#ifndef WENO_KCHAR_MIN_BLOCKS
#define WENO_KCHAR_MIN_BLOCKS 2  // resident 256-thread blocks per SM the characteristic kernel's registers allow
#endif

// Increments R(x_G) - W0 of one field at the two Gauss points of face k from that field's stencil
// differences dU (dU[0] = 0) and the tile's point-pair tables (PairTile rows), FP32: the arithmetic
// of pair_points for a single face, candidates outer, both points in one paired instruction.
// Returns false if a sum of alpha fell below kAlphaMin (the cell is then redone, fix_cell_char).
template <int M>
__device__ __forceinline__ bool face_pair(const float4* __restrict__ sgam, const float4* __restrict__ sdg,
                                          const float4* __restrict__ sgo, int cl, int k, const float* dU, float a0,
                                          float eps, int linear, float2& incr) {
  constexpr int TILE = WENO_K1_TILE;
  const float4 r = sdg[(2 * k) * TILE + cl], s = sdg[(2 * k + 1) * TILE + cl];
  const float2 dx = f2(r.x, r.y), dy = f2(r.z, r.w);
  float2 Ap = f2(0.f, 0.f), Bp = f2(0.f, 0.f), Am = f2(0.f, 0.f), Bm = f2(0.f, 0.f);
  if (linear) {
#pragma unroll
    for (int j = 0; j < M; ++j) {
      const float4 m = sgo[j * TILE + cl];
      const float da = dU[Sub<M>::a(j)], db = dU[Sub<M>::b(j)];
      const float gx = fmaf(m.x, da, m.y * db), gy = fmaf(m.z, da, m.w * db);
      const float4 g4 = sgam[(k * M + j) * TILE + cl];
      const float2 p = __ffma2_rn(f2(gx, gx), dx, __fmul2_rn(f2(gy, gy), dy));
      Bp = __ffma2_rn(f2(g4.x, g4.y), p, Bp);
      Bm = __ffma2_rn(f2(g4.z, g4.w), p, Bm);
    }
    incr = f2(s.x * Bp.x - s.z * Bm.x, s.y * Bp.y - s.w * Bm.y);
    return true;
  }
#pragma unroll
  for (int j = 0; j < M; ++j) {
    const float4 m = sgo[j * TILE + cl];
    const float da = dU[Sub<M>::a(j)], db = dU[Sub<M>::b(j)];
    const float gx = fmaf(m.x, da, m.y * db), gy = fmaf(m.z, da, m.w * db);
    const float b0 = a0 * fmaf(gx, gx, gy * gy);
    const float b = b0 > kBetaMax ? kBetaMax : b0;  // keeps a NaN
    const float b2 = b * b, b3 = b2 * b, be = b + eps;
    const float2 C0 = f2(be, be), C1 = f2(b2, b2), C2 = f2(b3, b3);
    const float4 g4 = sgam[(k * M + j) * TILE + cl];
    const float2 gp = f2(g4.x, g4.y), gn = f2(g4.z, g4.w);
    const float2 p = __ffma2_rn(f2(gx, gx), dx, __fmul2_rn(f2(gy, gy), dy));
    const float2 dp = __ffma2_rn(gp, __ffma2_rn(gp, C2, C1), C0);  // beta~+ + eps at both points
    const float2 dn = __ffma2_rn(gn, __ffma2_rn(gn, C2, C1), C0);
    const float2 ap = __fmul2_rn(gp, rcp2(__fmul2_rn(dp, dp)));
    const float2 an = __fmul2_rn(gn, rcp2(__fmul2_rn(dn, dn)));
    Ap = __fadd2_rn(Ap, ap);
    Bp = __ffma2_rn(ap, p, Bp);
    Am = __fadd2_rn(Am, an);
    Bm = __ffma2_rn(an, p, Bm);
  }
  incr = f2(fmaf(mulr(s.x, Bp.x), rcp_approx(Ap.x), -mulr(mulr(s.z, Bm.x), rcp_approx(Am.x))),
            fmaf(mulr(s.y, Bp.y), rcp_approx(Ap.y), -mulr(mulr(s.w, Bm.y), rcp_approx(Am.y))));
  return !(Ap.x < kAlphaMin) && !(Ap.y < kAlphaMin) && !(Am.x < kAlphaMin) && !(Am.y < kAlphaMin);
}

// fix_cell in characteristic variables: the lane's field is lane % 4.
template <int M, int G, bool WALLS>
__device__ __noinline__ void fix_cell_char(const unsigned char* smem, const TileCells& t, int64_t q, int cl) {
  using L = PairTile<M, G>;
  const int lane = threadIdx.x & 31, base = lane & ~3, l = lane & 3, g = min(lane >> 2, G - 1), k = g >> 1;
  const int64_t c = t.first + q;
  const float4* sgam = reinterpret_cast<const float4*>(smem);
  const float4* sdg = sgam + L::GAM / 16;
  const float *U = after_wait(t.U), *Ulo = after_wait(t.Ulo);
  float W0[4], Wn[4], Lr[4], Rr[4];
  load_vec<float, 4>(U + c * 4, W0);
  const float w0 = gather(U + c * 4 + l), l0 = gather(Ulo + c * 4 + l);
  slot_state4<float, WALLS>(U, __ldg(t.slot + (int64_t)k * t.N + q), Wn);
  const float4 d0 = sdg[(2 * k) * L::TILE + cl];
  const float tx = d0.y - d0.x, ty = d0.w - d0.z, it = rsqrtf(fmaf(tx, tx, mulr(ty, ty)));
  roe_rows(W0, Wn, ty * it, -tx * it, t.gas_gamma - 1.f, l, Lr, Rr);
  const int32_t fm = flip_mask<WALLS, 4>(l);
  float dU[M + 1];
#pragma unroll 1
  for (int s = 1; s <= M; ++s)
    dU[s] = lane_sum4(Lr, slot_delta<float, 4, WALLS, true>(U, Ulo, __ldg(t.slot + (int64_t)(s - 1) * t.N + q), l,
                                                            fm, w0, l0), base);
  const float incr = fix_increment<M, G>(sgam, sdg, sdg + L::DG / 16, cl, g, [&](int s) { return dU[s]; },
                                         __ldg(t.area + c), t.eps);
  const float dWl = lane_sum4(Rr, incr, base);  // variable l of R dU
  if (lane < 4 * G) t.Wg[(t.gbase + q * G + g) * 4 + l] = w0 + (l0 + dWl);
}

// One tile in characteristic variables.  Per face, each lane builds the Roe frame, projects the stencil
// differences onto its field and evaluates the face's two Gauss points with face_pair; lanes of cells
// past the end compute on the last cell's data and store nothing.
template <int M, int G, int PARTS, bool WALLS>
__device__ __forceinline__ bool tile_points_char(const unsigned char* smem, uint64_t* bar, uint32_t phase,
                                                 const TileCells& t, int64_t tile) {
  using L = PairTile<M, G>;
  const int tid = threadIdx.x % L::THREADS, part = threadIdx.x / L::THREADS;
  const int base = (tid & 31) & ~3, l = tid & 3, cl = tid >> 2;
  const int64_t qr = tile * L::TILE + cl;
  const bool act = qr < t.N;
  const int64_t q = act ? qr : t.N - 1;
  const int64_t c = t.first + q;
  const float4* sgam = reinterpret_cast<const float4*>(smem);
  const float4* sdg = sgam + L::GAM / 16;
  const float4* sgo = sdg + L::DG / 16;
  // stencil gathers (independent of the staged tables) before the wait
  const float *U = after_wait(t.U), *Ulo = after_wait(t.Ulo);
  float W0[4];
  load_vec<float, 4>(U + c * 4, W0);
  const float w0 = W0[l], l0 = gather(Ulo + c * 4 + l);
  float dW[M + 1];
  dW[0] = 0.f;
  const int32_t fm = flip_mask<WALLS, 4>(l);
#pragma unroll
  for (int s = 1; s <= M; ++s)
    dW[s] = slot_delta<float, 4, WALLS, true>(U, Ulo, __ldg(t.slot + (int64_t)(s - 1) * t.N + q), l, fm, w0, l0);
  const float a0 = __ldg(t.area + c);
  const bool ok = mbar_wait_bounded(bar, phase);
  if (__syncthreads_or(!ok)) return false;
  bool inrange = true;  // every sum of alpha of this lane's Gauss points within the FP32 range
#pragma unroll 1
  for (int k = part; k < G / 2; k += PARTS) {
    // the frame of face k: the neighbour across it (slot k + 1) and the unit normal from the
    // direction x_G' - x_G of its two Gauss points
    float Wn[4];
    slot_state4<float, WALLS>(U, __ldg(t.slot + (int64_t)k * t.N + q), Wn);
    const float4 d0 = sdg[(2 * k) * L::TILE + cl];
    const float tx = d0.y - d0.x, ty = d0.w - d0.z, it = rsqrtf(fmaf(tx, tx, mulr(ty, ty)));
    float Lr[4], Rr[4];
    roe_rows(W0, Wn, ty * it, -tx * it, t.gas_gamma - 1.f, l, Lr, Rr);
    float dU[M + 1];
    dU[0] = 0.f;
#pragma unroll
    for (int s = 1; s <= M; ++s) dU[s] = lane_sum4(Lr, dW[s], base);
    float2 incr;
    inrange = face_pair<M>(sgam, sdg, sgo, cl, k, dU, a0, t.eps, t.linear, incr) && inrange;
    const float d0l = lane_sum4(Rr, incr.x, base), d1l = lane_sum4(Rr, incr.y, base);  // variable l of R dU
    if (act) {
      t.Wg[(t.gbase + q * G + 2 * k) * 4 + l] = w0 + (l0 + d0l);
      t.Wg[(t.gbase + q * G + 2 * k + 1) * 4 + l] = w0 + (l0 + d1l);
    }
  }
  // a cell's four lanes mix all fields, so it is redone whole; lanes past the end read the zero fill of
  // the tables and are left out
  fix_marked<PARTS>(act && !inrange, tile * L::TILE, [&](int64_t qf, int cf) { fix_cell_char<M, G, WALLS>(smem, t, qf, cf); });
  return true;
}

// FP32C Euler K1 over the tiles of both cell types (KINDS bit 0: quads, bit 1: triangles; a mesh of one
// type has the instance sized for it), quads first.
#ifndef WENO_K1_BLOCKS_Q
#define WENO_K1_BLOCKS_Q (WENO_K1_MIN_BLOCKS * 64 / WENO_K1_TILE)  // resident blocks per SM, quads
#endif
#ifndef WENO_K1_BLOCKS_T
// triangles: 80 registers without spills, 24 warps per SM (measured 2.6 % faster per pass than at
// the quads' 16 warps, whose 122 registers spill when cut to 96)
#define WENO_K1_BLOCKS_T (WENO_K1_MIN_BLOCKS * 96 / WENO_K1_TILE)  // resident blocks per SM, triangles
#endif
// Threads of a block.  SPLIT (characteristic variables on small meshes): TILE x 4 threads for every face instead
// of threads that walk the faces, whose frames, projections and candidates are one serial chain of about
// 600 instructions a face; what is repeated is the gathers.  80 registers (768 threads an SM; with 64, which
// spill more, 6,400 quads take 33.0 us a step instead of 30.9).
template <int KINDS, bool SPLIT> struct K1Threads {
  static constexpr int value = WENO_K1_TILE * 4 * (!SPLIT ? 1 : KINDS & 1 ? 4 : 3);
};
// The register budget: 65,536 / (blocks x threads) per thread.
template <int KINDS, bool CHAR, bool SPLIT> struct K1Blocks {
  static constexpr int value = SPLIT ? 768 / K1Threads<KINDS, true>::value
      : CHAR ? WENO_KCHAR_MIN_BLOCKS * 64 / WENO_K1_TILE : KINDS == 2 ? WENO_K1_BLOCKS_T : WENO_K1_BLOCKS_Q;
};
template <int KINDS> struct K1Smem {
  static constexpr int quad = PairTile<12, 8>::STAGE, tri = PairTile<9, 6>::STAGE;
  static constexpr int stage = (KINDS & 1) ? quad : tri, bytes = stage + 16;  // one buffer + one mbarrier (padded)
};

template <int KINDS, bool CHAR, bool WALLS, bool SPLIT>
__global__ void __launch_bounds__(K1Threads<KINDS, SPLIT>::value, K1Blocks<KINDS, CHAR, SPLIT>::value) k_reconstruct_tma(
    const __grid_constant__ TileMaps mq, const __grid_constant__ TileMaps mt, const __grid_constant__ TileCells tq,
    const __grid_constant__ TileCells tt, int* __restrict__ err, int stall, int once) {
  constexpr int TILE = WENO_K1_TILE, PARTS = K1Threads<KINDS, SPLIT>::value / (TILE * 4);
  extern __shared__ __align__(128) unsigned char smem[];
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + K1Smem<KINDS>::stage);
  const int tid = threadIdx.x;
  const int64_t nq = KINDS & 1 ? (tq.N + TILE - 1) / TILE : 0, ntiles = nq + (KINDS & 2 ? (tt.N + TILE - 1) / TILE : 0);
  if (tid == 0) {
    mbar_init(bar, stall ? 2 : 1);  // stall != 0 (testing aid): the wait runs out
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  __syncthreads();
  auto quads = [&](int64_t tile) { return KINDS == 1 || (KINDS == 3 && tile < nq); };
  auto issue = [&](int64_t tile) {
    if (quads(tile)) load_tile<12, 8>(smem, &mq, tile, bar, once);
    else load_tile<9, 6>(smem, &mt, tile - nq, bar, once);
  };
  if (tid == 0 && blockIdx.x < ntiles) issue(blockIdx.x);
  kernel_wait();
  uint32_t phase = 0u;
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    bool ok;
    if (quads(tile)) {
      if constexpr (CHAR) ok = tile_points_char<12, 8, PARTS, WALLS>(smem, bar, phase, tq, tile);
      else ok = tile_points<12, 8, WALLS>(smem, bar, phase, tq, tile);
    } else {
      if constexpr (CHAR) ok = tile_points_char<9, 6, PARTS, WALLS>(smem, bar, phase, tt, tile - nq);
      else ok = tile_points<9, 6, WALLS>(smem, bar, phase, tt, tile - nq);
    }
    if (!ok) {  // the whole block: tile_points agrees on it
      if (tid == 0) *err = 1;
      return;
    }
    phase ^= 1u;
    const int64_t next = tile + gridDim.x;
    if (next < ntiles) {
      __syncthreads();  // the buffer is free for the next tile's copy
      if (tid == 0) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        issue(next);
      }
    }
  }
}

// ---------------------------------------------------------------- K2
template <typename T>
struct Prm { T gas_gamma, ax, ay; };

#ifndef WENO_K2_FAST
#define WENO_K2_FAST 1  // FP32 flux with approximate reciprocal / square root (FP64 always exact); 0: IEEE-rounded
#endif

// Division and square root of the flux: IEEE-rounded, or for FP32 with WENO_K2_FAST the
// hardware approximations (rcp.approx / sqrt.approx, a few ulp), which FP32 rounding of the
// Gauss values already dominates.
template <typename T> struct FluxMath {
  static __device__ __forceinline__ T rcp(T x) { return T(1) / x; }
  static __device__ __forceinline__ T div(T a, T b) { return a / b; }
  static __device__ __forceinline__ T sqr(T x) { return sqrt(x); }
};
#if WENO_K2_FAST
template <> struct FluxMath<float> {
  static __device__ __forceinline__ float rcp(float x) { return rcp_approx(x); }
  static __device__ __forceinline__ float div(float a, float b) { return __fmul_rn(a, rcp_approx(b)); }
  static __device__ __forceinline__ float sqr(float x) {
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
  }
};
#endif

// HLLC in the frame of the unit normal (nx, ny); returns the flux rotated back.  The side of the contact
// is taken by selection, not by branches: a warp's faces rarely agree on one.  Every product is either
// inside an explicit fma or rounded, so that a flux has the same bits in whichever kernel it is inlined
// (k_face_f32 and k_update_f32c: a mesh alone and as part of a larger batch give the same results).
template <typename T>
__device__ __forceinline__ void hllc(const T wl[4], const T wr[4], T nx, T ny, T gam, T out[4], bool& bad) {
  using FM = FluxMath<T>;
  const T gm1 = gam - T(1);
  const T rl = wl[0], rr = wr[0], El = wl[3], Er = wr[3];
  const T il = FM::rcp(rl), ir = FM::rcp(rr);
  const T nl = fma(wl[1], nx, mulr(wl[2], ny)), tl = fma(wl[2], nx, -mulr(wl[1], ny));  // normal and tangential
  const T nr = fma(wr[1], nx, mulr(wr[2], ny)), tr = fma(wr[2], nx, -mulr(wr[1], ny));  // momentum
  const T ul = mulr(nl, il), vl = mulr(tl, il), ur = mulr(nr, ir), vr = mulr(tr, ir);
  const T pl = mulr(gm1, fma(-mulr(T(0.5), rl), fma(ul, ul, mulr(vl, vl)), El));
  const T pr = mulr(gm1, fma(-mulr(T(0.5), rr), fma(ur, ur, mulr(vr, vr)), Er));
  bad |= !(rl > T(0) && rr > T(0) && pl > T(0) && pr > T(0));  // a NaN fails; a NaN energy shows in p
  const T cl = FM::sqr(mulr(mulr(gam, pl), il)), cr = FM::sqr(mulr(mulr(gam, pr), ir));
  // Roe averages
  const T sl = FM::sqr(rl), sr = FM::sqr(rr), iw = FM::rcp(sl + sr);
  const T ua = mulr(fma(sl, ul, mulr(sr, ur)), iw), va = mulr(fma(sl, vl, mulr(sr, vr)), iw);
  const T Ha = mulr(fma(sl, mulr(El + pl, il), mulr(sr, mulr(Er + pr, ir))), iw);
  const T ca = FM::sqr(mulr(gm1, fma(T(-0.5), fma(ua, ua, mulr(va, va)), Ha)));
  const T SL = fmin(ul - cl, ua - ca), SR = fmax(ur + cr, ua + ca);
  const T ml = mulr(rl, SL - ul), mr = mulr(rr, SR - ur);
  const T SS = FM::div(fma(-ur, mr, fma(ul, ml, pr - pl)), ml - mr);
  const bool left = SL >= T(0) || SS >= T(0);
  const T S = left ? SL : SR, m = left ? ml : mr, r = left ? rl : rr, E = left ? El : Er;
  const T mn = left ? nl : nr, mt = left ? tl : tr, un = left ? ul : ur, ut = left ? vl : vr;
  const T p = left ? pl : pr, ri = left ? il : ir;
  const T id = FM::rcp(S - SS), k = mulr(m, id);  // k: rho* of this side's star state
  const T Es = fma(k, fma(SS - un, SS, mulr(E, ri)), mulr(SS - un, mulr(p, id)));
  const bool star = left ? !(SL >= T(0)) : SR > T(0);  // between the outer waves
  const T b1 = fma(mn, un, p), b2 = mulr(mn, ut), b3 = mulr(E + p, un);
  const T f0 = star ? fma(S, k - r, mn) : mn, f1 = star ? fma(S, fma(k, SS, -mn), b1) : b1;
  const T f2 = star ? fma(S, fma(k, ut, -mt), b2) : b2, f3 = star ? fma(S, Es - E, b3) : b3;
  out[0] = f0;
  out[1] = fma(f1, nx, -mulr(f2, ny));
  out[2] = fma(f1, ny, mulr(f2, nx));
  out[3] = f3;
}

// Prescribed outer state of the inflow faces (gr = -3 - q for inflow face q): wa at
// the Gauss points whose xi = n . x_G - c0 (FP64, [q][2]) lies below speed * t_stage,
// wb elsewhere; t_stage = t[instance] + c dt[instance] with c = 0, 1, 1/2 for the
// three RK3 stages (Section 4).  The comparison is made in FP64 in both precisions.
template <typename T>
struct Inflow {
  T wa[4], wb[4];
  const double* xi;
  const double* t;
  const double* dt;
  double speed, c;
};

__device__ __forceinline__ int64_t cell_of_gauss(int64_t g, int64_t nQ) {
  return g < 8 * nQ ? g / 8 : nQ + (g - 8 * nQ) / 6;
}

// Euler state outside a boundary face at its point k (code: -1 outflow, -2 wall, -3 - q inflow face q)
// from the state w inside; i is the instance.
template <typename T, bool INFLOW>
__device__ __forceinline__ void outer_state(const T w[4], int64_t code, T nx, T ny, int k, const Inflow<T>& inf, int i,
                                            T out[4]) {
#pragma unroll
  for (int v = 0; v < 4; ++v) out[v] = w[v];
  if (code == -2) {  // reflective wall: normal momentum reversed
    const T mn = T(-2) * fma(w[1], nx, mulr(w[2], ny));
    out[1] = fma(mn, nx, w[1]);
    out[2] = fma(mn, ny, w[2]);
  }
  if constexpr (INFLOW) {
    if (code <= -3) {
      const bool a = __ldg(inf.xi + 2 * (-3 - code) + k) < inf.speed * (inf.t[i] + inf.c * inf.dt[i]);
#pragma unroll
      for (int v = 0; v < 4; ++v) out[v] = a ? inf.wa[v] : inf.wb[v];
    }
  }
}

// Flags: flag[instance] is set when a Gauss-point state of a face of that instance is non-physical;
// nQ and inst map a Gauss-value index back to its cell's instance (inst == nullptr: a single instance).

// Scalar upwind flux, FP32C: one thread per face.
__global__ void __launch_bounds__(256) k_face_scalar(
    const float* Wg, const int32_t* __restrict__ gl, const int32_t* __restrict__ gr,
    const float* __restrict__ fnx, const float* __restrict__ fny, const float* __restrict__ flen, int64_t nF,
    float* F, Prm<float> prm, int* flag, const int32_t* __restrict__ inst, int64_t nQ) {
  kernel_begin();
  kernel_wait();
  for (int64_t f = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; f < nF; f += (int64_t)gridDim.x * blockDim.x) {
    const int64_t il = __ldg(gl + f), ir = __ldg(gr + f);
    const float an = prm.ax * __ldg(fnx + f) + prm.ay * __ldg(fny + f), len = __ldg(flen + f);
    float acc = 0.f;
    bool bad = false;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const float wl = Wg[il + k], wr = ir >= 0 ? Wg[ir + 1 - k] : wl;
      const float fk = an * (an >= 0.f ? wl : wr);
      bad |= !(fk == fk);
      acc += fk;
    }
    F[f] = acc * (0.5f * len);
    if (bad) flag[inst ? __ldg(inst + cell_of_gauss(il, nQ)) : 0] = 1;  // every writer stores the same value
  }
}

// Euler HLLC flux, FP32C: one thread per face.
template <bool INFLOW>
__global__ void __launch_bounds__(256) k_face_f32(
    const float* Wg, const int32_t* __restrict__ gl, const int32_t* __restrict__ gr,
    const float* __restrict__ fnx, const float* __restrict__ fny, const float* __restrict__ flen, int64_t nF,
    float* F, Prm<float> prm, int* flag, const int32_t* __restrict__ inst, int64_t nQ,
    Inflow<float> inf) {
  kernel_begin();
  for (int64_t f = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; f < nF; f += (int64_t)gridDim.x * blockDim.x) {
    const int64_t il = __ldg(gl + f), ir = __ldg(gr + f);
    const float nx = __ldg(fnx + f), ny = __ldg(fny + f), len = __ldg(flen + f);
    const int i = INFLOW && ir <= -3 && inst ? __ldg(inst + cell_of_gauss(il, nQ)) : 0;
    kernel_wait();
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    bool bad = false;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      float wl[4], wr[4], fk[4];
      load_vec<float, 4>(Wg + (il + k) * 4, wl);
      // the right cell meets the left cell's point k at its point 1 - k
      if (ir >= 0) load_vec<float, 4>(Wg + (ir + 1 - k) * 4, wr);
      else outer_state<float, INFLOW>(wl, ir, nx, ny, k, inf, i, wr);
      hllc<float>(wl, wr, nx, ny, prm.gas_gamma, fk, bad);
#pragma unroll
      for (int v = 0; v < 4; ++v) acc[v] += fk[v];
    }
#pragma unroll
    for (int v = 0; v < 4; ++v) acc[v] *= 0.5f * len;
    store_vec<float, 4>(F + f * 4, acc);
    if (bad) flag[inst ? __ldg(inst + cell_of_gauss(il, nQ)) : 0] = 1;  // every writer stores the same value
  }
}

// The time steps of the next step: dt[i] = src[i] (src may be dt), or v for every instance (src == nullptr), and for the
// FP32C stages split[i] = (hi, lo) with hi + lo ~ dt[i] to 2^-48 (split once here: every cell would spend
// FP64 instructions on it).
__global__ void k_set_dt(double* dt, float2* __restrict__ split, const double* src, double v, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double d = src ? src[i] : v;
  const float hi = (float)d;
  dt[i] = d;
  split[i] = make_float2(hi, (float)(d - (double)hi));
}

// t[i] += dt[i] for every instance (after the third stage of a step).
__global__ void k_advance_time(double* t, const double* dt, int n) {
  kernel_begin();
  kernel_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) t[i] += dt[i];
}

// ---------------------------------------------------------------- K3
// MODE 0: R = L(U).  MODE 1..3: SSP-RK3 stage s written as
//   W(s) = W^n + c_s ((W(s-1) - W^n) + dt L(W(s-1))), c = 1, 1/4, 2/3, W(0) = W^n,
// i.e. the stages of Section 4 with the combination regrouped around W^n.
// Stages 1, 2 write the stage buffer Ws; stage 3 writes U (= W^{n+1}).
// COMP (FP32 fluxes, compensated state): the face sum is accumulated error-free
// (compensated two-sum), and 1/|Omega|, dt, the RK coefficient and the state
// update use double-float arithmetic, so that sum_i |Omega_i| dW_i telescopes
// to ~1e-14 of the fluxes and the hi + lo state keeps its ~48-bit precision.
// Quads (cells below nQ, face lists qcf [k][nQ]) and triangles (tcf [k][nT]) in one launch.
template <typename T, int NV, bool COMP, int MODE>
__global__ void __launch_bounds__(256) k_gather(
    const T* F, const int32_t* __restrict__ qcf, const int32_t* __restrict__ tcf,
    const T* __restrict__ inv_area, const T* __restrict__ inv_area_lo, int64_t nQ, int64_t nT, T* U,
    T* Ulo, T* Ws, T* Wslo, T* R, const double* dt, const float2* dt_split, const int32_t* __restrict__ inst) {
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < nQ + nT; c += (int64_t)gridDim.x * blockDim.x) {
    const bool quad = c < nQ;
    const int32_t* cf = quad ? qcf + c : tcf + (c - nQ);
    const int64_t row = quad ? nQ : nT;
    int32_t ef[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) ef[k] = k < 3 || quad ? __ldg(cf + k * row) : 0;
    const T ia = __ldg(inv_area + c);
    const T ial = COMP ? __ldg(inv_area_lo + c) : T(0);
    const int i = inst ? __ldg(inst + c) : 0;
    kernel_wait();
    T acc[NV], comp[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) { acc[v] = T(0); comp[v] = T(0); }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (k == 3 && !quad) break;
      const int32_t e = ef[k];
      const int64_t f = e >= 0 ? e : ~e;
      T fv[NV];
      load_vec<T, NV>(F + f * NV, fv);
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const T x = e >= 0 ? -fv[v] : fv[v];  // outward flux leaves the L cell
        if (COMP) {
          float s, err;
          two_sum((float)acc[v], (float)x, s, err);
          acc[v] = s;
          comp[v] = __fadd_rn((float)comp[v], err);
        } else {
          acc[v] += x;
        }
      }
    }
    if (MODE == 0) {
      T res[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) res[v] = COMP ? (acc[v] + comp[v]) * ia : acc[v] * ia;
      store_vec<T, NV>(R + c * NV, res);
    } else {
      T un[NV], ws[NV], out[NV];
      load_vec<T, NV>(U + c * NV, un);
      if (MODE > 1) load_vec<T, NV>(Ws + c * NV, ws);
      if (!COMP) {
        const T h = (T)dt[i];
        const T cs = MODE == 1 ? T(1) : (MODE == 2 ? T(0.25) : T(2.0 / 3.0));
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          const T d = (MODE > 1 ? ws[v] - un[v] : T(0)) + h * (acc[v] * ia);
          out[v] = un[v] + cs * d;
        }
        store_vec<T, NV>(MODE == 3 ? U + c * NV : Ws + c * NV, out);
      } else {
        const float2 dts = dt_split[i];
        const df h{dts.x, dts.y};
        const df iad{(float)ia, (float)ial};
        const df cs = MODE == 1 ? df{1.0f, 0.0f} : (MODE == 2 ? df{0.25f, 0.0f} : df{0.6666667f, -1.9868216e-08f});
        T unl[NV], wsl[NV], outl[NV];
        load_vec<T, NV>(Ulo + c * NV, unl);
        if (MODE > 1) load_vec<T, NV>(Wslo + c * NV, wsl);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          const df res = df_mul(df_norm((float)acc[v], (float)comp[v]), iad);
          df d = df_mul(h, res);
          if (MODE > 1) {
            float s, e;
            two_sum((float)ws[v], -(float)un[v], s, e);
            d = df_add(d, df_norm(s, __fadd_rn(e, __fsub_rn((float)wsl[v], (float)unl[v]))));
          }
          const df o = df_add(df{(float)un[v], (float)unl[v]}, df_mul(cs, d));
          out[v] = o.hi;
          outl[v] = o.lo;
        }
        store_vec<T, NV>(MODE == 3 ? U + c * NV : Ws + c * NV, out);
        store_vec<T, NV>(MODE == 3 ? Ulo + c * NV : Wslo + c * NV, outl);
      }
    }
  }
}

// ---------------------------------------------------------------- K2 + K3, FP32C Euler
// One face of a cell as its cell sees it: the neighbour's Gauss value that meets the face's first point
// of the cell (its own local point index; -1 outflow, -2 wall, -3 - q inflow face q), the face's unit
// normal (L to R) and its length, negative where the cell is the face's R cell.
struct CellFace { int32_t other; float nx, ny, slen; };

// Face fluxes, gather and RK3 stage of the FP32C Euler path in one pass: four lanes per cell, lane k
// with face k computes that face's flux, then (after a 4 x 4 transposition by shuffles) lane v sums and
// updates variable v.  A flux is thus computed by both of the face's cells, from the same operands in
// the same order (the cell's place on the face decides which is left), so both get the same bits and
// sum_i |Omega_i| dW_i telescopes as if it had been stored once; what is saved is a launch and the wait
// between the two kernels.  The sum and the stage are those of k_gather (COMP), operation by operation.
// MODE as k_gather.  Used while all its lanes are resident at once (use_fused): computing every flux twice
// costs 90 us a pass on 1.0M cells where k_face_f32 and k_gather take 37 + 27, but an 800-triangle step
// takes 25.3 us instead of 30.7 (10,000 triangles in characteristic variables 43.7 instead of 47.1;
// 51,200 triangles 61.5 either way).
template <int MODE, bool INFLOW>
__global__ void __launch_bounds__(256) k_update_f32c(
    const float* Wg, const CellFace* __restrict__ cf, const float* __restrict__ inv_area,
    const float* __restrict__ inv_area_lo, int64_t nQ, int64_t N, float* U, float* Ulo, float* Ws, float* Wslo, float* R,
    const float2* dt, const int32_t* __restrict__ inst, float gas_gamma, int* flag, Inflow<float> inf) {
  // uniform over a warp, whose lanes exchange fluxes; lanes past the end repeat the last cell
  for (int64_t t0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); t0 < 4 * N;
       t0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t t = t0 + (threadIdx.x & 31);
    const bool act = t < 4 * N;
    const int64_t c = act ? t >> 2 : N - 1;
    const int k = (int)(t & 3);
    const bool quad = c < nQ;
    const int i = inst ? __ldg(inst + c) : 0;
    const float ia = __ldg(inv_area + c), ial = __ldg(inv_area_lo + c);
    float4 e = make_float4(0.f, 0.f, 0.f, 0.f);
    if (quad || k < 3)
      e = __ldg(reinterpret_cast<const float4*>(cf) + (quad ? 4 * c + k : 4 * nQ + 3 * (c - nQ) + k));
    kernel_wait();
    float x[4] = {0.f, 0.f, 0.f, 0.f};
    if (quad || k < 3) {
      const int32_t other = __float_as_int(e.x);
      const float nx = e.y, ny = e.z, slen = e.w;
      const float4* own = reinterpret_cast<const float4*>(Wg) + (quad ? 8 * c : 8 * nQ + 6 * (c - nQ)) + 2 * k;
      float a[2][4], b[2][4];  // own and outer states at the cell's points 2k, 2k + 1
#pragma unroll
      for (int h = 0; h < 2; ++h) load_vec<float, 4>(reinterpret_cast<const float*>(own + h), a[h]);
      if (other >= 0) {
#pragma unroll
        for (int h = 0; h < 2; ++h) load_vec<float, 4>(Wg + ((int64_t)other - h) * 4, b[h]);
      } else {
#pragma unroll
        for (int h = 0; h < 2; ++h) outer_state<float, INFLOW>(a[h], other, nx, ny, h, inf, i, b[h]);
      }
      const bool left = slen > 0.f;
      bool bad = false;
#pragma unroll
      for (int h = 0; h < 2; ++h) {  // the face's points in the order of its L cell
        float wl[4], wr[4], fk[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          wl[v] = left ? a[h][v] : b[1 - h][v];
          wr[v] = left ? b[h][v] : a[1 - h][v];
        }
        hllc<float>(wl, wr, nx, ny, gas_gamma, fk, bad);
#pragma unroll
        for (int v = 0; v < 4; ++v) x[v] += fk[v];
      }
      const float w = -0.5f * slen;  // outward flux leaves the L cell
#pragma unroll
      for (int v = 0; v < 4; ++v) x[v] *= w;
      if (bad && act) flag[i] = 1;  // every writer stores the same value
    }
    // x[v] of lane k becomes x[k] of lane v: exchange across bit 0, then bit 1 of the lane
#pragma unroll
    for (int bit = 1; bit <= 2; bit *= 2) {
      const bool up = (k & bit) != 0;
#pragma unroll
      for (int m = 0; m < 2; ++m) {
        const int lo = bit == 1 ? 2 * m : m, hi = lo + bit;
        const float give = up ? x[lo] : x[hi];
        const float got = __shfl_xor_sync(0xffffffffu, give, bit);
        if (up) x[lo] = got;
        else x[hi] = got;
      }
    }
    const int64_t at = 4 * c + k;  // this lane's variable from here on
    float acc = 0.f, comp = 0.f;
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      float s, err;
      two_sum(acc, x[f], s, err);
      if (f < 3 || quad) {
        acc = s;
        comp = __fadd_rn(comp, err);
      }
    }
    if constexpr (MODE == 0) {
      if (act) R[at] = (acc + comp) * ia;
    } else {
      const float2 dts = dt[i];
      const df h{dts.x, dts.y};
      const df iad{ia, ial};
      const df cs = MODE == 1 ? df{1.0f, 0.0f} : (MODE == 2 ? df{0.25f, 0.0f} : df{0.6666667f, -1.9868216e-08f});
      const float un = U[at], unl = Ulo[at];
      df d = df_mul(h, df_mul(df_norm(acc, comp), iad));
      if (MODE > 1) {
        float s, e;
        two_sum(Ws[at], -un, s, e);
        d = df_add(d, df_norm(s, __fadd_rn(e, __fsub_rn(Wslo[at], unl))));
      }
      const df o = df_add(df{un, unl}, df_mul(cs, d));
      if (act) {
        (MODE == 3 ? U : Ws)[at] = o.hi;
        (MODE == 3 ? Ulo : Wslo)[at] = o.lo;
      }
    }
  }
}

// ---------------------------------------------------------------- K4 (reductions, not on the hot path)
// Largest stable step min 2|Omega| / sum_p (|v.n_p| + c)|l_p| and integrals sum |Omega| (U + U_lo) of each
// instance, in FP64 and in two levels over a fixed partition (`chunks`), so that results do not depend on
// scheduling.  What bounds them is the FP64 pipe (2 lanes a clock and SM) and, on small meshes, latency:
// the time step is formed and reduced in one kernel with the reciprocals and roots of arith_f64.cuh (48
// FP64 instructions a quad, not about 110 with IEEE division), FP32 states are widened on the integer
// pipe, minima are taken on the bits of the numbers, and a chunk is as many cells as spread a mesh over
// all SMs.
// 260k FP32C cells, both results: 170 -> 80 us (k_chunk_dt 29, k_chunk_sum 13, the rest launches and waits for
// the host); 8k FP64 quads, time step: 27 us less.

// A float as a double by integer operations, except for subnormals, infinities and NaN.
__device__ __forceinline__ double widen(float x) {
  const uint32_t b = __float_as_uint(x), m = b & 0x7fffffffu;
  if (m - 0x00800000u < 0x7f000000u)
    return __hiloint2double((int)((b & 0x80000000u) | ((m >> 3) + 0x38000000u)), (int)(b << 29));
  return m == 0 ? __hiloint2double((int)b, 0) : (double)x;
}
__device__ __forceinline__ double widen(double x) { return x; }

// Whether the cells of a state start on 16-byte boundaries, as load_vec needs it.  The reductions take a state
// that starts at any element of a buffer.
template <typename T, bool COMP>
__device__ __forceinline__ bool vec_aligned(const T* U, const T* Ulo) {
  return ((reinterpret_cast<uintptr_t>(U) | (COMP ? reinterpret_cast<uintptr_t>(Ulo) : 0)) & 15) == 0;
}

// The state of cell c in FP64; vec as vec_aligned (the same for all cells of a launch).
template <typename T, int NV, bool COMP>
__device__ __forceinline__ void state_f64(const T* __restrict__ U, const T* __restrict__ Ulo, int64_t c, bool vec, double w[NV]) {
  T h[NV], l[NV];
  if (NV == 1 || vec) {
    load_vec<T, NV>(U + c * NV, h);
    if (COMP) load_vec<T, NV>(Ulo + c * NV, l);
  } else {
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      h[v] = U[c * NV + v];
      if (COMP) l[v] = Ulo[c * NV + v];
    }
  }
#pragma unroll
  for (int v = 0; v < NV; ++v) w[v] = COMP ? widen(h[v]) + widen(l[v]) : widen(h[v]);
}

// a / b from r = rcp_any(b), corrected with the remainder to the rounded quotient (but for near ties), so that
// a step is as close to the exact one as with IEEE division.
__device__ __forceinline__ double quotient(double a, double b, double r) {
  const uint32_t h = hi_word(b) & 0x7fffffffu;
  const double q = a * r;
  if (!rcp_safe(h, h) || (hi_word(q) & 0x7fffffffu) >= 0x7ff00000u) return quotient_ieee(a, b);
  return fma(fma(-q, b, a), r, q);
}
// Half of a cell's stable step, |Omega| / sum_p (|v.n_p| + c)|l_p|; never negative, NaN for a negative pressure.
template <int NV, int NFACE>
__device__ __forceinline__ double half_dt(const double w[NV], const int32_t* __restrict__ cf, int64_t row,
                                          const double* __restrict__ fnx, const double* __restrict__ fny,
                                          const double* __restrict__ flen, double area, double gas_gamma, double ax,
                                          double ay) {
  double u = ax, vv = ay, snd = 0.0;
  if constexpr (NV == 4) {
    const double r = rcp_any(w[0]);
    u = quotient(w[1], w[0], r);
    vv = quotient(w[2], w[0], r);
    const double p = (gas_gamma - 1.0) * (w[3] - 0.5 * w[0] * (u * u + vv * vv));
    snd = sqrt_any(quotient(gas_gamma * p, w[0], r));
  }
  double s = 0.0;
#pragma unroll
  for (int k = 0; k < NFACE; ++k) {
    const int32_t e = __ldg(cf + k * row);
    const int64_t f = e >= 0 ? e : ~e;
    s += (fabs(u * __ldg(fnx + f) + vv * __ldg(fny + f)) + snd) * __ldg(flen + f);
  }
  return quotient(area, s, rcp_any(s));
}

// Smaller of two numbers that are >= 0 or NaN, by their bits: a NaN of either sign is above every number,
// so it is left out like by fmin.
__device__ __forceinline__ uint64_t bits_of(double x) { return (uint64_t)__double_as_longlong(x); }
__device__ __forceinline__ uint64_t block_min(uint64_t m) {
  __shared__ uint64_t sh[8];
#pragma unroll
  for (int o = 16; o; o >>= 1) m = min(m, (uint64_t)__shfl_xor_sync(0xffffffffu, (unsigned long long)m, o));
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = m;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 8; ++i) m = min(m, sh[i]);
  return m;
}
constexpr double kNoDt = 0.5e300;  // where no cell has a step

// Level 1, time step: one block per chunk [c0, c1) of cells of one instance and one type.
template <typename T, int NV, bool COMP>
__global__ void __launch_bounds__(256) k_chunk_dt(
    const T* __restrict__ U, const T* __restrict__ Ulo, const int32_t* __restrict__ qcf,
    const int32_t* __restrict__ tcf, const double* __restrict__ fnx, const double* __restrict__ fny,
    const double* __restrict__ flen, const double* __restrict__ area, const int64_t* __restrict__ chunks, int64_t nQ,
    int64_t nT, double gas_gamma, double ax, double ay, double* __restrict__ partial) {
  kernel_begin();
  const int64_t c0 = __ldg(chunks + 2 * blockIdx.x), c1 = __ldg(chunks + 2 * blockIdx.x + 1);
  const bool vec = vec_aligned<T, COMP>(U, Ulo);
  uint64_t m = bits_of(kNoDt);
  for (int64_t c = c0 + threadIdx.x; c < c1; c += 256) {
    double w[NV];
    state_f64<T, NV, COMP>(U, Ulo, c, vec, w);
    const double a = __ldg(area + c);
    const double h = c < nQ ? half_dt<NV, 4>(w, qcf + c, nQ, fnx, fny, flen, a, gas_gamma, ax, ay)
                            : half_dt<NV, 3>(w, tcf + (c - nQ), nT, fnx, fny, flen, a, gas_gamma, ax, ay);
    m = min(m, bits_of(h));
  }
  m = block_min(m);
  if (threadIdx.x == 0) partial[blockIdx.x] = __longlong_as_double((long long)m);
}

// Level 1, integrals.
template <int NV>
__device__ __forceinline__ void block_sum_store(const double acc[NV], double* __restrict__ out) {
  __shared__ double sh[256 * NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) sh[v * 256 + threadIdx.x] = acc[v];
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s)
      for (int v = 0; v < NV; ++v) sh[v * 256 + threadIdx.x] += sh[v * 256 + threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x < NV) out[threadIdx.x] = sh[threadIdx.x * 256];
}
template <typename T, int NV, bool COMP>
__global__ void __launch_bounds__(256) k_chunk_sum(const T* __restrict__ U, const T* __restrict__ Ulo,
                                                   const double* __restrict__ area,
                                                   const int64_t* __restrict__ chunks, double* __restrict__ partial) {
  kernel_begin();
  const int64_t c0 = __ldg(chunks + 2 * blockIdx.x), c1 = __ldg(chunks + 2 * blockIdx.x + 1);
  const bool vec = vec_aligned<T, COMP>(U, Ulo);
  double acc[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) acc[v] = 0.0;
  for (int64_t c = c0 + threadIdx.x; c < c1; c += 256) {
    double w[NV];
    state_f64<T, NV, COMP>(U, Ulo, c, vec, w);
    const double a = __ldg(area + c);
#pragma unroll
    for (int v = 0; v < NV; ++v) acc[v] += a * w[v];
  }
  block_sum_store<NV>(acc, partial + (int64_t)blockIdx.x * NV);
}

// Level 2: one block per instance over its chunks' partials [k0, k1); out is in the host's memory.
__global__ void __launch_bounds__(256) k_instance_dt(const double* partial, const int64_t* __restrict__ chunk_off,
                                                     double* out) {
  const int64_t k0 = __ldg(chunk_off + blockIdx.x), k1 = __ldg(chunk_off + blockIdx.x + 1);
  kernel_wait();
  uint64_t m = bits_of(kNoDt);
  for (int64_t k = k0 + threadIdx.x; k < k1; k += 256) m = min(m, bits_of(partial[k]));
  m = block_min(m);
  if (threadIdx.x == 0) out[blockIdx.x] = 2.0 * __longlong_as_double((long long)m);
}
template <int NV>
__global__ void __launch_bounds__(256) k_instance_sum(const double* partial, const int64_t* __restrict__ chunk_off,
                                                      double* out) {
  const int64_t k0 = __ldg(chunk_off + blockIdx.x), k1 = __ldg(chunk_off + blockIdx.x + 1);
  kernel_wait();
  double acc[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) acc[v] = 0.0;
  for (int64_t k = k0 + threadIdx.x; k < k1; k += 256)
#pragma unroll
    for (int v = 0; v < NV; ++v) acc[v] += partial[k * NV + v];
  block_sum_store<NV>(acc, out + (int64_t)blockIdx.x * NV);
}

__global__ void k_fill(double* __restrict__ p, double v, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) p[i] = v;
}

}  // namespace dev
}  // namespace weno
