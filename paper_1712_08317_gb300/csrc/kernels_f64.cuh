// FP64 kernels and their arithmetic: reconstruction (K1), component-wise and in characteristic
// variables, and face fluxes (K2).
//
// What bounds them: the FP64 pipe.  GB300 has 2 FP64 lanes per clock and SM, 1/64 of its FP32 rate
// (0.62 T FMA/s measured), so a double-precision instruction costs what about sixty others do, and
// the tables' bytes are small beside it.  Hence every choice below removes FP64 instructions, at the
// price of integer work, shuffles, shared-memory traffic or larger tables:
//   - the splitting of the linear weights (geometry only) is done once per solver (k_split_weights),
//   - differences, gradients and indicators are computed once per (cell, variable) and shared through
//     shared memory by the threads of the cell's faces,
//   - the indicators, the nonlinear weights and their sums are formed on the integer pipe (PosNum),
//   - other reciprocals start from the special-function unit's 20-bit seed and take one third-order step.
// K1 measured (one pass; first: one thread per (cell, variable), IEEE division, the splitting repeated
// by every variable, 5,350 FP64 issue slots a (cell, variable) of quads; then: as here with all of the
// weights in FP64, 2,140 slots; then: gamma / d^2 on the integer pipe, 1,200; their sums too, 940; now: the
// indicators d too, 560): 17,920 Euler quads 662 -> 277 -> 154 -> 124 -> 100 us, 15,360 triangles
// 384 -> 144 -> 83 -> 68 -> 56 us, 1,600 scalar quads 332 -> 30 us and now 16.  On 343k quads and 295k triangles
// the FP64 pipe is 72 and 76 %, the integer pipe 67 and 64 % busy: the two balance, and what is left is how
// well they overlap.
#pragma once

#include "kernels.cuh"

namespace weno {
namespace dev {

// Split linear weights of a group from its linear weights gam [g][j][q] (Section 3.4):
// gt+ = (gamma + theta |gamma|) / 2, gt- = gt+ - gamma, sigma+- = sum gt+-, gamma+- = gt+- / sigma+-.
// wt [g][j][q] = (gamma+, gamma-) and sig [g][q] = (sigma+, sigma-), rows of `pitch` cells; wt as PosPair for
// the component-wise kernel (W = PosPair), as double2 in characteristic variables.
__device__ __forceinline__ void put(PosPair* p, double x, double y) { *p = PosPair{pos_word(x), pos_word(y)}; }
__device__ __forceinline__ void put(double2* p, double x, double y) { *p = make_double2(x, y); }
template <int M, typename W>
__global__ void k_split_weights(const double* __restrict__ gam, int64_t N, int G, double theta, int64_t pitch,
                                W* __restrict__ wt, double2* __restrict__ sig) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= N * G) return;
  const int64_t g = t / N, q = t - g * N;
  double tp[M], tm[M], sp = 0.0, sm = 0.0;
#pragma unroll
  for (int j = 0; j < M; ++j) {
    const double x = gam[(g * M + j) * N + q];
    tp[j] = 0.5 * (x + theta * fabs(x));
    tm[j] = tp[j] - x;
    sp += tp[j];
    sm += tm[j];
  }
  sig[g * pitch + q] = make_double2(sp, sm);
  const double isp = 1.0 / sp, ism = 1.0 / sm;
#pragma unroll
  for (int j = 0; j < M; ++j) put(wt + (g * M + j) * pitch + q, tp[j] * isp, tm[j] * ism);
}

__device__ __forceinline__ PosPair pos_pair(const PosPair* p) {
  const ulonglong2 w = __ldg(reinterpret_cast<const ulonglong2*>(p));
  return PosPair{{w.x}, {w.y}};
}

// Layout of a block of either kernel: `width` = cells x variables of its tile; thread t holds column
// t % width (cell (t % width) / NV, variable or field t % NV) and, of the cell's G Gauss points, one, or
// in characteristic variables PTS, from PTS (t / width) on.
constexpr int kF64MaxWidth = 32;

// Component-wise FP64 K1.  The threads of a column share out its M stencil differences, then its M
// candidates, both into shared memory; then each evaluates its Gauss point.  A thread a point: no FP64
// instruction is repeated (a warp takes whole shares of the candidates), 64 registers leave 30 warps an
// SM, and the last wave is short (with both points of a face in a thread, 96 registers and 16 to 19
// warps: triangles 79 us a pass on the mesh above against 68, quads 124 either way).
template <int NV, int M, int G, bool WALLS>
__global__ void __launch_bounds__(kF64MaxWidth * G) k_reconstruct_f64(
    const double* U, const int32_t* __restrict__ slot, const double* __restrict__ gop,
    const double* __restrict__ dg, const double* __restrict__ gam, const PosPair* __restrict__ wt,
    const double2* __restrict__ sigma, const double* __restrict__ area, int64_t N, int64_t pitch, int64_t first,
    int64_t gbase, double* Wg, double eps, int linear, int width) {
  constexpr int PER = (M + G - 1) / G;
  extern __shared__ double sm[];
  double* dW = sm;                                      // [slot - 1][column]
  double *gx = sm + M * width, *gy = gx + M * width;    // [candidate][column]
  PosWord* be = reinterpret_cast<PosWord*>(gy + M * width);
  PosWord *b2 = be + M * width, *b3 = b2 + M * width;
  const int col = threadIdx.x % width, g = threadIdx.x / width, v = col % NV;
  const int64_t qr = (int64_t)blockIdx.x * (width / NV) + col / NV;
  const int64_t q = qr < N ? qr : N - 1;  // columns past the end work on the last cell and store nothing
  const int64_t c = first + q;
  kernel_wait();
  U = after_wait(U);
  const double w0 = gather(U + c * NV + v), a0 = __ldg(area + c);
  const int32_t fm = flip_mask<WALLS, NV>(v);
#pragma unroll
  for (int i = 0; i < PER; ++i) {
    const int s = g + i * G;
    if (s < M) dW[s * width + col] =
        slot_delta<double, NV, WALLS, false>(U, nullptr, __ldg(slot + (int64_t)s * N + q), v, fm, w0, 0.0);
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < PER; ++i) {
    const int j = g + i * G;
    if (j >= M) break;
    const double* o = gop + (int64_t)(j * 4) * N + q;
    const double da = dW[(sub_a<M>(j) - 1) * width + col], db = dW[(sub_b<M>(j) - 1) * width + col];
    const CandF64 cd =
        candidate_f64(__ldg(o) * da + __ldg(o + N) * db, __ldg(o + 2 * N) * da + __ldg(o + 3 * N) * db, a0, eps);
    const int k = j * width + col;
    gx[k] = cd.gx; gy[k] = cd.gy;
    be[k] = pos_word(cd.be); b2[k] = pos_word(cd.b2); b3[k] = pos_word(cd.b3);
  }
  __syncthreads();
  const double dx = __ldg(dg + (int64_t)(2 * g) * N + q), dy = __ldg(dg + (int64_t)(2 * g + 1) * N + q);
  double incr = 0.0;
  if (linear) {
    const double* gg = gam + (int64_t)(g * M) * N + q;
#pragma unroll 3
    for (int j = 0; j < M; ++j)
      incr += __ldg(gg + (int64_t)j * N) * (gx[j * width + col] * dx + gy[j * width + col] * dy);
  } else {
    auto cand = [&](int j) {
      const int k = j * width + col;
      return CandPos{gx[k], gy[k], be[k], b2[k], b3[k]};
    };
    const PosPair* w = wt + (int64_t)(g * M) * pitch + q;
    const double2 sig = __ldg(sigma + (int64_t)g * pitch + q);
    auto weights = [&](int, int j) { return pos_pair(w + j * pitch); };
    if (!face_points_f64<M, 1>(cand, weights, &dx, &dy, &sig, &incr))
      face_points_ieee<M, 1>(cand, weights, &dx, &dy, &sig, a0, eps, &incr);
  }
  if (qr < N) Wg[(gbase + q * G + g) * NV + v] = w0 + incr;
}

// Roe frame of one face: R^-1 (fr[4 f + v]) and R (fr[16 + 4 v + f]), fields f ordered q_n - a, entropy,
// shear, q_n + a, from the two cells' averages and the outward normal (tx, ty rotated by -90 degrees).
__device__ __forceinline__ void roe_frame_f64(const double Wl[4], const double Wr[4], double tx, double ty, double gm1,
                                              double* __restrict__ fr) {
  const double it = rsqrt_any(tx * tx + ty * ty), nx = ty * it, ny = -tx * it;
  const double il = rcp_any(Wl[0]), ir = rcp_any(Wr[0]);
  const double ul = Wl[1] * il, vl = Wl[2] * il, ur = Wr[1] * ir, vr = Wr[2] * ir;
  const double hl = (Wl[3] + gm1 * (Wl[3] - 0.5 * Wl[0] * (ul * ul + vl * vl))) * il;
  const double hr = (Wr[3] + gm1 * (Wr[3] - 0.5 * Wr[0] * (ur * ur + vr * vr))) * ir;
  const double sl = sqrt_any(Wl[0]), sr = sqrt_any(Wr[0]), iw = rcp_any(sl + sr);
  const double u = (sl * ul + sr * ur) * iw, v = (sl * vl + sr * vr) * iw, H = (sl * hl + sr * hr) * iw;
  const double kin = 0.5 * (u * u + v * v), a2 = gm1 * (H - kin), ia = rsqrt_any(a2), a = a2 * ia;
  const double qn = u * nx + v * ny, qt = v * nx - u * ny;
  const double b1 = gm1 * ia * ia, b2 = b1 * kin;
  fr[0] = 0.5 * (b2 + qn * ia); fr[1] = -0.5 * (b1 * u + nx * ia); fr[2] = -0.5 * (b1 * v + ny * ia); fr[3] = 0.5 * b1;
  fr[4] = 1.0 - b2; fr[5] = b1 * u; fr[6] = b1 * v; fr[7] = -b1;
  fr[8] = -qt; fr[9] = -ny; fr[10] = nx; fr[11] = 0.0;
  fr[12] = 0.5 * (b2 - qn * ia); fr[13] = 0.5 * (nx * ia - b1 * u); fr[14] = 0.5 * (ny * ia - b1 * v); fr[15] = 0.5 * b1;
  fr[16] = 1.0; fr[17] = 1.0; fr[18] = 0.0; fr[19] = 1.0;
  fr[20] = u - a * nx; fr[21] = u; fr[22] = -ny; fr[23] = u + a * nx;
  fr[24] = v - a * ny; fr[25] = v; fr[26] = nx; fr[27] = v + a * ny;
  fr[28] = H - a * qn; fr[29] = kin; fr[30] = qt; fr[31] = H + a * qn;
}

// FP64 K1 in characteristic variables (see the comment at the FP32C kernels below for the method).
// Thread (cell, field l, PTS points of a face): the two points share the projection and the candidates,
// 168 of about 470 FP64 instructions, so they go to two threads only on meshes too small to fill the
// FP64 pipe otherwise (f64_grid).  The block's first threads build the Roe frames, one thread a frame
// instead of four lanes each repeating it; every thread projects the shared stencil differences onto
// its field with row l of R^-1, evaluates its points, and returns variable l of R dU there.
constexpr int kFrame = 33;  // doubles a frame takes in shared memory (32, padded against bank conflicts)

template <int M, int G, int PTS, bool WALLS>
__global__ void __launch_bounds__(kF64MaxWidth * G / PTS) k_reconstruct_char_f64(
    const double* U, const int32_t* __restrict__ slot, const double* __restrict__ gop,
    const double* __restrict__ dg, const double* __restrict__ gam, const double2* __restrict__ wt,
    const double2* __restrict__ sigma, const double* __restrict__ area, int64_t N, int64_t pitch, int64_t first,
    int64_t gbase, double* Wg, double eps, double gas_gamma, int linear, int width) {
  constexpr int F = G / 2, PARTS = G / PTS, PER = (M + PARTS - 1) / PARTS;
  extern __shared__ double sm[];
  const int tile = width / 4, threads = width * PARTS;
  double* dW = sm;                      // [slot - 1][column]
  double* dU = dW + M * width;          // [slot - 1][thread]
  double* fr = dU + M * threads;        // [face][cell] frames
  double* inc = fr + kFrame * tile * F; // [point][thread]
  const int t = threadIdx.x, col = t % width, part = t / width, l = col % 4, cl = col / 4;
  const int64_t q0 = (int64_t)blockIdx.x * tile, qr = q0 + cl;
  const int64_t q = qr < N ? qr : N - 1;  // columns past the end work on the last cell and store nothing
  const int64_t c = first + q;
  kernel_wait();
  U = after_wait(U);
  const double w0 = gather(U + c * 4 + l), a0 = __ldg(area + c);
  const int32_t fm = flip_mask<WALLS, 4>(l);
#pragma unroll
  for (int i = 0; i < PER; ++i) {
    const int s = part + i * PARTS;
    if (s < M) dW[s * width + col] =
        slot_delta<double, 4, WALLS, false>(U, nullptr, __ldg(slot + (int64_t)s * N + q), l, fm, w0, 0.0);
  }
  if (t < tile * F) {  // frame of face t / tile of cell t % tile; the neighbour across face k is slot k + 1
    const int k = t / tile;
    const int64_t fq = q0 + t % tile < N ? q0 + t % tile : N - 1;
    double Wl[4], Wn[4];
    load_vec<double, 4>(U + (first + fq) * 4, Wl);
    slot_state4<double, WALLS>(U, __ldg(slot + (int64_t)k * N + fq), Wn);
    const double* d = dg + (int64_t)(4 * k) * N + fq;
    roe_frame_f64(Wl, Wn, __ldg(d + 2 * N) - __ldg(d), __ldg(d + 3 * N) - __ldg(d + N), gas_gamma - 1.0, fr + kFrame * t);
  }
  __syncthreads();
  const double* f0 = fr + kFrame * (part * PTS / 2 * tile + cl);
  const double L0 = f0[4 * l], L1 = f0[4 * l + 1], L2 = f0[4 * l + 2], L3 = f0[4 * l + 3];
#pragma unroll 4
  for (int s = 0; s < M; ++s) {
    const double* x = dW + s * width + 4 * cl;
    dU[s * threads + t] = L0 * x[0] + L1 * x[1] + L2 * x[2] + L3 * x[3];
  }
  const int g = PTS * part;
  const double* d = dg + (int64_t)(2 * g) * N + q;
  double dx[PTS], dy[PTS], incr[PTS];
#pragma unroll
  for (int h = 0; h < PTS; ++h) {
    dx[h] = __ldg(d + 2 * h * N);
    dy[h] = __ldg(d + (2 * h + 1) * N);
    incr[h] = 0.0;
  }
  auto cand = [&](int j) {
    const double* o = gop + (int64_t)(j * 4) * N + q;
    const double da = dU[(sub_a<M>(j) - 1) * threads + t], db = dU[(sub_b<M>(j) - 1) * threads + t];
    return candidate_f64(__ldg(o) * da + __ldg(o + N) * db, __ldg(o + 2 * N) * da + __ldg(o + 3 * N) * db, a0, eps);
  };
  if (linear) {
    const double* gg = gam + (int64_t)(g * M) * N + q;
#pragma unroll 3
    for (int j = 0; j < M; ++j) {
      const CandF64 x = cand(j);
#pragma unroll
      for (int h = 0; h < PTS; ++h) incr[h] += __ldg(gg + (int64_t)(h * M + j) * N) * (x.gx * dx[h] + x.gy * dy[h]);
    }
  } else {
    const double2* w = wt + (int64_t)(g * M) * pitch + q;
    double2 sig[PTS];
#pragma unroll
    for (int h = 0; h < PTS; ++h) sig[h] = __ldg(sigma + (int64_t)(g + h) * pitch + q);
    auto weights = [&](int h, int j) { return __ldg(w + (h * M + j) * pitch); };
    if (!face_points_f64<M, PTS>(cand, weights, dx, dy, sig, incr))
      face_points_ieee<M, PTS>(cand, weights, dx, dy, sig, a0, eps, incr);
  }
#pragma unroll
  for (int h = 0; h < PTS; ++h) inc[h * threads + t] = incr[h];
  __syncthreads();
  if (qr < N) {  // variable l of R dU
    const double* r = f0 + 16 + 4 * l;
    double* out = Wg + (gbase + q * G + g) * 4 + l;
#pragma unroll
    for (int h = 0; h < PTS; ++h) {
      const double* x = inc + h * threads + (t & ~3);
      out[h * 4] = w0 + (r[0] * x[0] + r[1] * x[1] + r[2] * x[2] + r[3] * x[3]);
    }
  }
}

// ---------------------------------------------------------------- K2
// HLLC flux of one Gauss point, as hllc in kernels.cuh with the divisions and square roots of this file,
// one reciprocal fewer on the star side (k p / m = p / (S_K - S*)) and the side taken by selection
// instead of branches: about 130 FP64 instructions.  Returns false, and no flux, unless every quantity
// it takes a reciprocal or a root of is in the range of the iterations; in particular a state that
// passes has rho > 0, p > 0 and a finite energy.
__device__ __forceinline__ bool hllc_f64(const double wl[4], const double wr[4], double nx, double ny, double gam,
                                         double out[4]) {
  const double gm1 = gam - 1.0;
  const double rl = wl[0], rr = wr[0], El = wl[3], Er = wr[3];
  const double il = rcp_f64(rl), ir = rcp_f64(rr);
  const double nl = wl[1] * nx + wl[2] * ny, tl = wl[2] * nx - wl[1] * ny;  // normal and tangential momentum
  const double nr = wr[1] * nx + wr[2] * ny, tr = wr[2] * nx - wr[1] * ny;
  const double ul = nl * il, vl = tl * il, ur = nr * ir, vr = tr * ir;
  const double pl = gm1 * (El - 0.5 * (nl * ul + tl * vl)), pr = gm1 * (Er - 0.5 * (nr * ur + tr * vr));
  const double al2 = gam * pl * il, ar2 = gam * pr * ir;
  const double al = sqrt_f64(al2), ar = sqrt_f64(ar2);
  const double sl = sqrt_f64(rl), sr = sqrt_f64(rr), iw = rcp_f64(sl + sr);
  const double u = (sl * ul + sr * ur) * iw, v = (sl * vl + sr * vr) * iw;
  const double H = (sl * ((El + pl) * il) + sr * ((Er + pr) * ir)) * iw;
  const double a2 = gm1 * (H - 0.5 * (u * u + v * v)), a = sqrt_f64(a2);
  const double SL = fmin(ul - al, u - a), SR = fmax(ur + ar, u + a);
  const double ml = rl * (SL - ul), mr = rr * (SR - ur), dm = ml - mr;
  const double SS = (pr - pl + ul * ml - ur * mr) * rcp_f64(dm);
  const bool left = SL >= 0.0 || SS >= 0.0;
  const double S = left ? SL : SR, dS = S - SS, id = rcp_f64(dS);
  const double r = left ? rl : rr, mn = left ? nl : nr, mt = left ? tl : tr, E = left ? El : Er;
  const double un = left ? ul : ur, ut = left ? vl : vr, p = left ? pl : pr, ri = left ? il : ir, m = left ? ml : mr;
  const double k = m * id;  // rho of the star state
  const double Es = k * (E * ri + (SS - un) * SS) + (SS - un) * (p * id);
  const double Se = (left ? SL >= 0.0 : !(SR > 0.0)) ? 0.0 : S;  // no star term beyond the outer waves
  const double f0 = mn + Se * (k - r), f1 = mn * un + p + Se * (k * SS - mn);
  const double f2 = mn * ut + Se * (k * ut - mt), f3 = (E + p) * un + Se * (Es - E);
  out[0] = f0;
  out[1] = f1 * nx - f2 * ny;
  out[2] = f1 * ny + f2 * nx;
  out[3] = f3;
  const uint32_t h[7] = {hi_word(rl), hi_word(rr), hi_word(al2), hi_word(ar2), hi_word(a2), hi_word(dm) & 0x7fffffffu,
                         hi_word(dS) & 0x7fffffffu};
  uint32_t lo = h[0], hi = h[0];
#pragma unroll
  for (int i = 1; i < 7; ++i) {
    lo = min(lo, h[i]);
    hi = max(hi, h[i]);
  }
  return rcp_safe(lo, hi);
}

// The general form, for states that hllc_f64 declines (and to find out whether they are non-physical).
__device__ __noinline__ void hllc_ieee(const double* wl, const double* wr, double nx, double ny, double gam, double* out,
                                       bool* bad) {
  hllc<double>(wl, wr, nx, ny, gam, out, *bad);
}

// FP64 K2: thread (face, Gauss point), the two points of a face on neighbouring lanes, which add their
// fluxes and store half of the face's variables each.  Twice the threads of the FP32 kernel: the FP64
// pipe is filled on meshes half the size, and each lane's two states are 64 contiguous bytes with its
// neighbour's.  Flags and boundary states as k_face.
template <int NV, bool INFLOW>
__global__ void __launch_bounds__(256) k_face_f64(
    const double* Wg, const int32_t* __restrict__ gl, const int32_t* __restrict__ gr,
    const double* __restrict__ fnx, const double* __restrict__ fny, const double* __restrict__ flen, int64_t nF,
    double* F, Prm<double> prm, int* flag, const int32_t* __restrict__ inst, int64_t nQ, Inflow<double> inf) {
  const int64_t total = 2 * nF;
  // the loop is uniform over a warp, whose lanes exchange fluxes; lanes past the end repeat the last face
  for (int64_t t0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); t0 < total;
       t0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t t = t0 + (threadIdx.x & 31);
    const bool act = t < total;
    const int64_t f = act ? t >> 1 : nF - 1;
    const int k = (int)(t & 1);
    const int64_t il = __ldg(gl + f), ir = __ldg(gr + f);
    const double nx = __ldg(fnx + f), ny = __ldg(fny + f), hl = 0.5 * __ldg(flen + f);
    kernel_wait();
    double wl[NV], wr[NV], fk[NV];
    load_vec<double, NV>(Wg + (il + k) * NV, wl);
    if (ir >= 0) {
      load_vec<double, NV>(Wg + (ir + 1 - k) * NV, wr);
    } else if constexpr (NV == 4) {
      const int i = INFLOW && ir <= -3 && inst ? __ldg(inst + cell_of_gauss(il, nQ)) : 0;
      outer_state<double, INFLOW>(wl, ir, nx, ny, k, inf, i, wr);
    } else {
      wr[0] = wl[0];
    }
    bool bad = false;
    if constexpr (NV == 4) {
      if (!hllc_f64(wl, wr, nx, ny, prm.gas_gamma, fk)) hllc_ieee(wl, wr, nx, ny, prm.gas_gamma, fk, &bad);
    } else {
      const double an = prm.ax * nx + prm.ay * ny;
      fk[0] = an * (an >= 0.0 ? wl[0] : wr[0]);
      bad = !(fk[0] == fk[0]);
    }
    double sum[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) sum[v] = hl * (fk[v] + __shfl_xor_sync(0xffffffffu, fk[v], 1));
    if (act) {
      if constexpr (NV == 4)
        reinterpret_cast<double2*>(F + f * 4)[k] = k ? make_double2(sum[2], sum[3]) : make_double2(sum[0], sum[1]);
      else if (k == 0)
        F[f] = sum[0];
      if (bad) flag[inst ? __ldg(inst + cell_of_gauss(il, nQ)) : 0] = 1;  // every writer stores the same value
    }
  }
}

}  // namespace dev
}  // namespace weno
