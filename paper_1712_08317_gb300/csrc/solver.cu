// C ABI of the library: meshes (host), solvers (device tables, launches,
// CUDA graphs of the RK3 step, autotuning, reductions).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <memory>
#include <mutex>
#include <new>
#include <string>
#include <type_traits>
#include <vector>

#include "host_lsq.hpp"
#include "host_mesh.hpp"
#include "kernels_f64.cuh"
#include "weno3.h"

namespace weno {
int set_error(int code, const std::string& msg);
}

using weno::GroupTables;
using weno::Mesh;

namespace {

thread_local std::string g_err;

int fail(int code, const std::string& msg) {
  g_err = msg;
  return code;
}

}  // namespace

int weno::set_error(int code, const std::string& msg) { return fail(code, msg); }

namespace {

#define CK(call)                                                                                 \
  do {                                                                                           \
    cudaError_t e_ = (call);                                                                     \
    if (e_ != cudaSuccess) return fail(WENO_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

struct DeviceGuard {
  int prev = -1;
  explicit DeviceGuard(int dev) {
    if (cudaGetDevice(&prev) == cudaSuccess && prev != dev) cudaSetDevice(dev);
    else prev = -1;
  }
  ~DeviceGuard() { if (prev >= 0) cudaSetDevice(prev); }
};

struct Launch {
  int block = 256;
  int grid = 0;  // 0: one thread per work item
};

unsigned grid_of(const Launch& l, int64_t work) {
  const int64_t full = (work + l.block - 1) / l.block;
  const int64_t g = l.grid > 0 ? std::min<int64_t>(l.grid, full) : full;
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>(g, 0x7fffffff));
}

// Launch of a kernel of the chain (kernel_begin / kernel_wait): it may start before the kernel ahead of it
// in the stream has finished.
template <typename... P, typename... A>
void launch(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t st, A&&... args) {
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);  // errors: cudaGetLastError (check_launch)
}

// TMA reconstruction: TILE x 4 threads per block, one TILE-cell tile per iteration.
constexpr int kTile = weno::dev::PairTile<12, 8>::TILE;
unsigned tma_grid(const Launch& l, int64_t tiles) {
  const int64_t g = l.grid > 0 ? std::min<int64_t>(l.grid, tiles) : tiles;
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>(g, 0x7fffffff));
}

}  // namespace

struct weno_mesh_s {
  Mesh m;
  // FP64 precompute of the last solver created on this mesh (same rcond / optimize reuse it)
  std::shared_ptr<std::pair<GroupTables, GroupTables>> tables;
  double tables_rcond = -1.0;
  int tables_optimize = -1;
};

struct weno_solver_s {
  int dev = 0, nsm = 0;
  int l2_bytes = 0;
  weno_params prm{};
  int nv = 4;
  bool fp64 = true;
  size_t esz = 8;
  int64_t nQ = 0, nT = 0, N = 0, nF = 0, n_boundary = 0;
  int n_inst = 1;
  // device tables
  // FP64: SoA tables [entry][cell] (gop, dg; gam for the linear scheme, otherwise the split weights
  // wt [g][j][cell] and their sums sig [g][cell], rows of q_pitch / t_pitch cells).  FP32C: packed rows of float4 / float2
  // with the cell fastest: gop = D_j^+ entries, dg = (x_G - c0, sigma+, sigma-),
  // gam = gamma+ then gamma- rows, gam1 = (gamma+_8, gamma-_8) of triangles.
  void *q_gop = nullptr, *q_dg = nullptr, *q_gam = nullptr, *t_gop = nullptr, *t_dg = nullptr, *t_gam = nullptr;
  void *q_gam1 = nullptr, *t_gam1 = nullptr;
  void *q_pgam = nullptr, *q_pdg = nullptr, *t_pgam = nullptr, *t_pdg = nullptr;  // point-pair tables (Euler FP32C)
  void *q_wt = nullptr, *t_wt = nullptr;        // FP64 split weights: PosPair, in characteristic variables double2,
  double2 *q_sig = nullptr, *t_sig = nullptr;   // and their sums
  int64_t q_pitch = 0, t_pitch = 0;  // row pitch (cells) of the packed FP32C tables and the FP64 split weights
  bool tma = false;                   // Euler FP32C: reconstruction with TMA-staged tables
  weno::dev::TileMaps q_maps{}, t_maps{};  // point-pair tables and gradient operators (FP32C Euler)
  int* err = nullptr;                 // set by a kernel whose bounded wait timed out
  int32_t *q_slot = nullptr, *t_slot = nullptr, *q_cf = nullptr, *t_cf = nullptr;
  void *area = nullptr, *inv_area = nullptr, *inv_area_lo = nullptr;
  double* area64 = nullptr;
  int32_t *gl = nullptr, *gr = nullptr;
  weno::dev::CellFace* cell_faces = nullptr;  // FP32C Euler: faces of each cell (4 per quad, then 3 per triangle)
  void *fnx = nullptr, *fny = nullptr, *flen = nullptr;
  double *fnx64 = nullptr, *fny64 = nullptr, *flen64 = nullptr;
  int32_t* inst = nullptr;
  int64_t *chunks = nullptr, *chunk_off = nullptr;  // reduction partition: [begin, end) pairs; per-instance offsets
  int64_t n_chunks = 0;
  double* partial = nullptr;
  // scratch
  void *Wg = nullptr, *F = nullptr, *Ws = nullptr, *Wslo = nullptr;
  float2* dt_split = nullptr;  // dt_dev as (hi, lo), for the FP32C stages
  double* dt_dev = nullptr;
  double* red = nullptr;     // results of the reductions, in pinned host memory that the device writes
  double* t_dev = nullptr;   // time of each instance (advanced by every step)
  int64_t n_in = 0;          // inflow faces
  double* in_xi = nullptr;   // [n_in][2] n . x_G - c0 of their Gauss points
  double in_wa[4] = {}, in_wb[4] = {};  // prescribed conservative states
  int* flag = nullptr;
  int debug_stall = 0;  // weno_solver_debug_stall
  bool walls = false;   // the mesh has reflective wall faces (stencil values carry momentum flips)
  std::vector<void*> allocs;
  Launch k1q, k1t, k2, k3;
  bool fused = false;  // FP32C Euler: fluxes and update in one kernel (use_fused)
  cudaStream_t cap = nullptr;
  struct Graph {
    const void* U;
    const void* Ulo;
    cudaGraphExec_t exec;
  };
  std::vector<Graph> graphs;

  ~weno_solver_s() {
    DeviceGuard g(dev);
    for (auto& x : graphs) cudaGraphExecDestroy(x.exec);
    if (cap) cudaStreamDestroy(cap);
    for (void* p : allocs) cudaFree(p);
    if (red) cudaFreeHost(red);
  }
  template <typename P>
  int alloc(P** p, size_t bytes) {
    void* q = nullptr;
    if (bytes == 0) bytes = 16;
    cudaError_t e = cudaMalloc(&q, bytes);
    if (e != cudaSuccess) return fail(WENO_ENOMEM, std::string("cudaMalloc: ") + cudaGetErrorString(e));
    allocs.push_back(q);
    *p = reinterpret_cast<P*>(q);
    return WENO_OK;
  }
  void drop_graphs() {
    for (auto& x : graphs) cudaGraphExecDestroy(x.exec);
    graphs.clear();
  }
};

namespace {

using S = weno_solver_s;
static_assert(weno::dev::kDevFlipX == weno::kFlipX && weno::dev::kDevFlipY == weno::kFlipY &&
                  weno::dev::kDevSlotCell == weno::kSlotCell,
              "stencil table bit layout shared by the host tables and the kernels");

// ------------------------------------------------------------ launches
// Grid of an FP64 reconstruction over n cells of G Gauss points and M candidates: blocks of `width` (cell,
// variable) columns with a thread for every pts points of a column, and the kernel's shared memory.  The
// FP64 pipe, split between the quarters of the SMs, is the bound and has to be shared out evenly: tiles
// shrink from 32 columns to 8 until every SM has four blocks (1,600 scalar quads: 18 us with 8 columns),
// and in characteristic variables the two points of a face go to two threads below four warps for every
// quarter.
struct F64Grid {
  int width, pts;
  unsigned blocks, threads;
  size_t smem;
};
F64Grid f64_grid(const S& s, int64_t n, int nv, int M, int G, bool characteristic) {
  const int pts = !characteristic || n * nv * (G / 2) < (int64_t)4 * 4 * 32 * s.nsm ? 1 : 2;
  int width = weno::dev::kF64MaxWidth;
  while (width > 8 && n * nv < (int64_t)4 * s.nsm * width) width /= 2;
  const int tile = width / nv, threads = width * G / pts;
  const size_t doubles = characteristic ? (size_t)M * width + (size_t)(M + pts) * threads + weno::dev::kFrame * tile * (G / 2)
                                        : (size_t)6 * M * width;
  return {width, pts, (unsigned)((n + tile - 1) / tile), (unsigned)threads, doubles * sizeof(double)};
}

// Mixed meshes: one launch for both cell types, quads first, up to 16 rounds of resident tiles.  It saves a
// launch and the wait for the quads' last tiles, about 5 us; against that its triangles run at the quads'
// register count, 16 instead of 24 warps an SM and 5 % slower.  A step of 133k cells takes 138.8 us in one
// launch and 151.1 in two, of 241k cells (63 % triangles) 211 and 219, of 1.0M cells 815 and 796.
bool merge_kinds(const S& s) { return s.nQ && s.nT && s.nQ + s.nT <= (int64_t)16 * 8 * kTile * s.nsm; }

// Characteristic variables, FP32C: a set of threads for every face of a cell while the blocks, three or four
// an SM with 256 or 192 threads, are all resident at once; above, the longer chain of a thread is hidden by
// other blocks and the gathers are not repeated.  A step: 1,600 quads 30.9 -> 22.7 us, 6,400 quads 37.0 -> 30.9,
// 6,370 mixed cells (2.6 tiles an SM) 37.0 -> 30.9, 8,192 triangles (3.4 an SM) 30.9 -> 28.9; but 8,320 mixed
// cells (3.4) equal and 10,000 triangles (4.1) 35.2 -> 39.1.
bool split_faces(const S& s) {
  return (s.nQ + kTile - 1) / kTile + (s.nT + kTile - 1) / kTile <= (int64_t)3 * s.nsm;
}

// Whether the tables of the FP32C Euler reconstruction leave L2 first.  A pass streams them; where they are
// about as large as the L2, the Gauss values, fluxes and states that the kernels of a stage hand to one
// another otherwise make room for tables that will not be there either when the next pass wants them.  Up to four times the
// L2 (129 MB): a step of 96,800 triangles 80.5 -> 76.1 us, 133k mixed cells 135.8 -> 125.1, 180k triangles
// 137.6 -> 125.8, 229k mixed cells 213.7 -> 196.9, 314k quads 304 -> 302, 500k mixed cells 425 -> 420; tables well inside
// the L2 (51k triangles, 40k quads) equal; 1.0M cells 806 -> 809.
bool tables_once(const S& s) {
  const int64_t q = weno::dev::PairTile<12, 8>::STAGE / kTile, t = weno::dev::PairTile<9, 6>::STAGE / kTile;
  return q * s.nQ + t * s.nT <= (int64_t)4 * s.l2_bytes;
}

// FP32C Euler reconstruction into wg.  which as below.
template <int KINDS, bool CHAR, bool WALLS>
void launch_tma_kinds(S& s, const Launch& l, const float* u, const float* ul, float* wg, cudaStream_t st) {
  const weno::dev::TileCells q{u, ul, (const float*)s.area, s.q_slot, s.nQ, 0, 0, wg, (float)s.prm.eps,
                               (float)s.prm.gas_gamma, s.prm.linear};
  weno::dev::TileCells t = q;
  t.slot = s.t_slot;
  t.N = s.nT;
  t.first = s.nQ;
  t.gbase = 8 * s.nQ;
  const int64_t tiles = (KINDS & 1 ? (s.nQ + kTile - 1) / kTile : 0) + (KINDS & 2 ? (s.nT + kTile - 1) / kTile : 0);
  auto run = [&](auto split) {
    constexpr bool SPLIT = decltype(split)::value;
    constexpr int smem = weno::dev::K1Smem<KINDS>::bytes;
    const auto kernel = weno::dev::k_reconstruct_tma<KINDS, CHAR, WALLS, SPLIT>;
    if constexpr (smem > 48 * 1024)  // tiles of 64 cells (WENO_K1_TILE)
      cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    launch(kernel, SPLIT ? (unsigned)tiles : tma_grid(l, tiles), weno::dev::K1Threads<KINDS, SPLIT>::value, smem, st, s.q_maps,
           s.t_maps, q, t, s.err, s.debug_stall, tables_once(s));
  };
  if constexpr (CHAR) {
    if (split_faces(s)) return run(std::true_type{});
  }
  run(std::false_type{});
}
template <bool CHAR, bool WALLS>
void launch_tma(S& s, const void* U, const void* Ulo, void* wg, cudaStream_t st, int which) {
  const float *u = static_cast<const float*>(U), *ul = static_cast<const float*>(Ulo);
  float* w = static_cast<float*>(wg);
  which &= (s.nQ ? 1 : 0) | (s.nT ? 2 : 0);
  if (which == 3 && merge_kinds(s)) return launch_tma_kinds<3, CHAR, WALLS>(s, s.k1q, u, ul, w, st);
  if (which & 1) launch_tma_kinds<1, CHAR, WALLS>(s, s.k1q, u, ul, w, st);
  if (which & 2) launch_tma_kinds<2, CHAR, WALLS>(s, s.k1t, u, ul, w, st);
}

// Cell reconstruction into the Gauss-value array wg.  which: bit 0 = quad group,
// bit 1 = triangle group.
template <typename T, int NV, bool COMP, bool WALLS>
void launch_reconstruct_impl(S& s, const void* U, const void* Ulo, void* wg, cudaStream_t st, int which) {
  if constexpr (COMP && NV == 4) {
    if (s.prm.characteristic) return launch_tma<true, WALLS>(s, U, Ulo, wg, st, which);
    return launch_tma<false, WALLS>(s, U, Ulo, wg, st, which);
  } else {
    const T* u = static_cast<const T*>(U);
    const T eps = (T)s.prm.eps;
    if constexpr (!COMP && NV == 4) {
      if (s.prm.characteristic) {
        const T gg = (T)s.prm.gas_gamma;
        if (s.nQ && (which & 1)) {
          const F64Grid g = f64_grid(s, s.nQ, 4, 12, 8, true);
          const auto kernel = g.pts == 1 ? weno::dev::k_reconstruct_char_f64<12, 8, 1, WALLS>
                                         : weno::dev::k_reconstruct_char_f64<12, 8, 2, WALLS>;
          launch(kernel, g.blocks, g.threads, g.smem, st, u, s.q_slot, (const double*)s.q_gop, (const double*)s.q_dg, (const double*)s.q_gam, s.q_wt, s.q_sig,
              (const double*)s.area, s.nQ, s.q_pitch, 0, 0, (double*)wg, eps, gg, s.prm.linear, g.width);
        }
        if (s.nT && (which & 2)) {
          const F64Grid g = f64_grid(s, s.nT, 4, 9, 6, true);
          const auto kernel = g.pts == 1 ? weno::dev::k_reconstruct_char_f64<9, 6, 1, WALLS>
                                         : weno::dev::k_reconstruct_char_f64<9, 6, 2, WALLS>;
          launch(kernel, g.blocks, g.threads, g.smem, st, u, s.t_slot, (const double*)s.t_gop, (const double*)s.t_dg, (const double*)s.t_gam, s.t_wt, s.t_sig,
              (const double*)s.area, s.nT, s.t_pitch, s.nQ, 8 * s.nQ, (double*)wg, eps, gg, s.prm.linear, g.width);
        }
        return;
      }
    }
    if constexpr (COMP) {
      if (s.nQ && (which & 1))
        launch(weno::dev::k_reconstruct_f32c<NV, 12, 8>, grid_of(s.k1q, s.nQ * NV), s.k1q.block, 0, st, u, static_cast<const T*>(Ulo), s.q_slot, (const float4*)s.q_gop, (const float4*)s.q_dg, (const float4*)s.q_gam,
            (const float2*)s.q_gam1, (const float*)s.area, s.nQ, s.q_pitch, 0, 0, (float*)wg, eps, s.prm.linear);
      if (s.nT && (which & 2))
        launch(weno::dev::k_reconstruct_f32c<NV, 9, 6>, grid_of(s.k1t, s.nT * NV), s.k1t.block, 0, st, u, static_cast<const T*>(Ulo), s.t_slot, (const float4*)s.t_gop, (const float4*)s.t_dg, (const float4*)s.t_gam,
            (const float2*)s.t_gam1, (const float*)s.area, s.nT, s.t_pitch, s.nQ, 8 * s.nQ, (float*)wg, eps,
            s.prm.linear);
    } else {
      if (s.nQ && (which & 1)) {
        const F64Grid g = f64_grid(s, s.nQ, NV, 12, 8, false);
        launch(weno::dev::k_reconstruct_f64<NV, 12, 8, WALLS>, g.blocks, g.threads, g.smem, st, u, s.q_slot, (const double*)s.q_gop, (const double*)s.q_dg, (const double*)s.q_gam, s.q_wt, s.q_sig,
            (const double*)s.area, s.nQ, s.q_pitch, 0, 0, (double*)wg, eps, s.prm.linear, g.width);
      }
      if (s.nT && (which & 2)) {
        const F64Grid g = f64_grid(s, s.nT, NV, 9, 6, false);
        launch(weno::dev::k_reconstruct_f64<NV, 9, 6, WALLS>, g.blocks, g.threads, g.smem, st, u, s.t_slot, (const double*)s.t_gop, (const double*)s.t_dg, (const double*)s.t_gam, s.t_wt, s.t_sig,
            (const double*)s.area, s.nT, s.t_pitch, s.nQ, 8 * s.nQ, (double*)wg, eps, s.prm.linear, g.width);
      }
    }
  }
}

// Walls only change the stencil gathers (momentum flips of mirror images); meshes without
// walls run kernels without that code.
template <typename T, int NV, bool COMP>
void launch_reconstruct_into(S& s, const void* U, const void* Ulo, void* wg, cudaStream_t st, int which) {
  if constexpr (NV == 4) {
    if (s.walls) return launch_reconstruct_impl<T, NV, COMP, true>(s, U, Ulo, wg, st, which);
  }
  launch_reconstruct_impl<T, NV, COMP, false>(s, U, Ulo, wg, st, which);
}

template <typename T, int NV, bool COMP>
void launch_reconstruct(S& s, const void* U, const void* Ulo, cudaStream_t st, int which = 3) {
  launch_reconstruct_into<T, NV, COMP>(s, U, Ulo, s.Wg, st, which);
}

template <typename T>
weno::dev::Inflow<T> inflow_of(const S& s, double c) {
  weno::dev::Inflow<T> in{};
  for (int v = 0; v < 4; ++v) {
    in.wa[v] = (T)s.in_wa[v];
    in.wb[v] = (T)s.in_wb[v];
  }
  in.xi = s.in_xi;
  in.t = s.t_dev;
  in.dt = s.dt_dev;
  in.speed = s.prm.inflow_line[3];
  in.c = c;
  return in;
}

// Face fluxes of the Gauss values wg into fl; c places the stage in the step (time t + c dt).
template <typename T, int NV>
void launch_face(S& s, const void* wg, void* fl, double c, cudaStream_t st) {
  if (!s.nF) return;
  const weno::dev::Prm<T> p{(T)s.prm.gas_gamma, (T)s.prm.adv[0], (T)s.prm.adv[1]};
  if constexpr (std::is_same<T, double>::value) {
    // inflow faces exist for the Euler equations only
    const auto kernel = NV == 4 && s.n_in ? weno::dev::k_face_f64<NV, NV == 4> : weno::dev::k_face_f64<NV, false>;
    launch(kernel, grid_of(s.k2, 2 * s.nF), s.k2.block, 0, st, (const T*)wg, s.gl, s.gr, (const T*)s.fnx, (const T*)s.fny, (const T*)s.flen, s.nF, (T*)fl, p, s.flag,
        s.inst, s.nQ, inflow_of<T>(s, c));
  } else if constexpr (NV == 4) {
    const auto kernel = s.n_in ? weno::dev::k_face_f32<true> : weno::dev::k_face_f32<false>;
    launch(kernel, grid_of(s.k2, s.nF), s.k2.block, 0, st, (const T*)wg, s.gl, s.gr, (const T*)s.fnx, (const T*)s.fny, (const T*)s.flen, s.nF, (T*)fl, p, s.flag,
        s.inst, s.nQ, inflow_of<T>(s, c));
  } else {
    launch(weno::dev::k_face_scalar, grid_of(s.k2, s.nF), s.k2.block, 0, st, (const T*)wg, s.gl, s.gr, (const T*)s.fnx, (const T*)s.fny, (const T*)s.flen, s.nF, (T*)fl, p, s.flag,
        s.inst, s.nQ);
  }
}

template <typename T, int NV, bool COMP, int MODE>
void launch_gather_mode(S& s, const void* fl, void* U, void* Ulo, void* R, cudaStream_t st) {
  launch(weno::dev::k_gather<T, NV, COMP, MODE>, grid_of(s.k3, s.N), s.k3.block, 0, st, (const T*)fl, s.q_cf, s.t_cf, (const T*)s.inv_area, (const T*)s.inv_area_lo, s.nQ, s.nT, (T*)U, (T*)Ulo,
      (T*)s.Ws, (T*)s.Wslo, (T*)R, s.dt_dev, s.dt_split, s.inst);
}

template <typename T, int NV, bool COMP>
void launch_gather(S& s, int mode, const void* fl, void* U, void* Ulo, void* R, cudaStream_t st) {
  switch (mode) {
    case 0: launch_gather_mode<T, NV, COMP, 0>(s, fl, U, Ulo, R, st); break;
    case 1: launch_gather_mode<T, NV, COMP, 1>(s, fl, U, Ulo, R, st); break;
    case 2: launch_gather_mode<T, NV, COMP, 2>(s, fl, U, Ulo, R, st); break;
    default: launch_gather_mode<T, NV, COMP, 3>(s, fl, U, Ulo, R, st); break;
  }
}

// FP32C Euler: fluxes, gather and stage in one pass.
constexpr int kUpdateBlock = 128;
// While the pass's four lanes per cell fit the SMs at once (its 60 registers allow 1,024 threads an SM).
bool use_fused(const S& s) { return !s.fp64 && s.nv == 4 && 4 * s.N <= (int64_t)1024 * s.nsm; }

// Launch shapes of a residual's kernels as they are chosen now; grid 0: as many blocks as the work takes.  Where the
// cell types take launches of their own, cell_launch is that of the quads.
bool split_form(const S& s) { return s.tma && s.prm.characteristic && split_faces(s); }
Launch cell_launch(const S& s) {
  if (s.fp64) {
    const F64Grid g = s.nQ ? f64_grid(s, s.nQ, s.nv, 12, 8, s.prm.characteristic) : f64_grid(s, s.nT, s.nv, 9, 6, s.prm.characteristic);
    return {(int)g.threads, 0};
  }
  if (split_form(s)) return {s.nQ ? weno::dev::K1Threads<1, true>::value : weno::dev::K1Threads<2, true>::value, 0};
  const Launch& l = s.nQ ? s.k1q : s.k1t;
  return s.tma ? Launch{kTile * 4, l.grid} : l;
}
Launch face_launch(const S& s) { return s.fused ? Launch{kUpdateBlock} : s.k2; }
Launch gather_launch(const S& s) { return s.fused ? Launch{kUpdateBlock} : s.k3; }

template <int MODE>
void launch_update_mode(S& s, const void* wg, double c, void* U, void* Ulo, void* R, cudaStream_t st) {
  const auto kernel = s.n_in ? weno::dev::k_update_f32c<MODE, true> : weno::dev::k_update_f32c<MODE, false>;
  launch(kernel, grid_of(Launch{kUpdateBlock}, 4 * s.N), kUpdateBlock, 0, st, (const float*)wg, s.cell_faces, (const float*)s.inv_area, (const float*)s.inv_area_lo, s.nQ, s.N, (float*)U,
      (float*)Ulo, (float*)s.Ws, (float*)s.Wslo, (float*)R, s.dt_split, s.inst, (float)s.prm.gas_gamma, s.flag,
      inflow_of<float>(s, c));
}

// What follows the reconstruction in a stage: fluxes of the Gauss values wg (through fl where they are
// stored), gather and, for mode 1..3, the RK3 stage; mode 0 writes the residual to R.
template <typename T, int NV, bool COMP>
void launch_update(S& s, int mode, double c, const void* wg, void* fl, void* U, void* Ulo, void* R, cudaStream_t st) {
  if constexpr (COMP && NV == 4) {
    if (s.fused) {
      switch (mode) {
        case 0: launch_update_mode<0>(s, wg, c, U, Ulo, R, st); break;
        case 1: launch_update_mode<1>(s, wg, c, U, Ulo, R, st); break;
        case 2: launch_update_mode<2>(s, wg, c, U, Ulo, R, st); break;
        default: launch_update_mode<3>(s, wg, c, U, Ulo, R, st); break;
      }
      return;
    }
  }
  launch_face<T, NV>(s, wg, fl, c, st);
  launch_gather<T, NV, COMP>(s, mode, fl, U, Ulo, R, st);
}

// The passes after the reconstruction on their own (weno_pass, weno_autotune), in the kernels that launch_update
// takes: where one does both passes, it is pass 3.
template <typename T, int NV, bool COMP>
void launch_pass2(S& s, cudaStream_t st) {
  if (!s.fused) launch_face<T, NV>(s, s.Wg, s.F, 0.0, st);
}
template <typename T, int NV, bool COMP>
void launch_pass3(S& s, cudaStream_t st) {
  if (s.fused) launch_update<T, NV, COMP>(s, 0, 0.0, s.Wg, s.F, nullptr, nullptr, s.Ws, st);
  else launch_gather<T, NV, COMP>(s, 0, s.F, nullptr, nullptr, s.Ws, st);
}

template <typename T, int NV, bool COMP>
void launch_step_body(S& s, void* U, void* Ulo, cudaStream_t st) {
  // the stages of Section 4 evaluate L at t, t + dt, t + dt/2
  constexpr double kStageTime[3] = {0.0, 1.0, 0.5};
  for (int stage = 1; stage <= 3; ++stage) {
    const void* src = stage == 1 ? U : s.Ws;
    const void* srclo = stage == 1 ? Ulo : s.Wslo;
    launch_reconstruct<T, NV, COMP>(s, src, srclo, st);
    launch_update<T, NV, COMP>(s, stage, kStageTime[stage - 1], s.Wg, s.F, U, Ulo, nullptr, st);
  }
  launch(weno::dev::k_advance_time, (s.n_inst + 127) / 128, 128, 0, st, s.t_dev, s.dt_dev, s.n_inst);
}

// one call per precision / variable count
#define WENO_DISPATCH(s, FN, ...)                                  \
  do {                                                             \
    if ((s).fp64) {                                                \
      if ((s).nv == 4) FN<double, 4, false>(__VA_ARGS__);          \
      else FN<double, 1, false>(__VA_ARGS__);                      \
    } else {                                                       \
      if ((s).nv == 4) FN<float, 4, true>(__VA_ARGS__);            \
      else FN<float, 1, true>(__VA_ARGS__);                        \
    }                                                              \
  } while (0)

// Level 1 of a reduction follows whatever the stream holds; level 2 may start before it has drained.
template <typename T, int NV, bool COMP>
void launch_max_dt(S& s, const void* U, const void* Ulo, cudaStream_t st) {
  if (s.n_chunks)
    weno::dev::k_chunk_dt<T, NV, COMP><<<(unsigned)s.n_chunks, 256, 0, st>>>(
        (const T*)U, (const T*)Ulo, s.q_cf, s.t_cf, s.fnx64, s.fny64, s.flen64, s.area64, s.chunks, s.nQ, s.nT,
        s.prm.gas_gamma, s.prm.adv[0], s.prm.adv[1], s.partial);
  launch(weno::dev::k_instance_dt, s.n_inst, 256, 0, st, s.partial, s.chunk_off, s.red);
}

template <typename T, int NV, bool COMP>
void launch_sums(S& s, const void* U, const void* Ulo, cudaStream_t st) {
  if (s.n_chunks)
    weno::dev::k_chunk_sum<T, NV, COMP><<<(unsigned)s.n_chunks, 256, 0, st>>>(
        (const T*)U, (const T*)Ulo, s.area64, s.chunks, s.partial);
  launch(weno::dev::k_instance_sum<NV>, s.n_inst, 256, 0, st, s.partial, s.chunk_off, s.red);
}

int check_launch() {
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail(WENO_ECUDA, std::string("kernel launch: ") + cudaGetErrorString(e));
  return WENO_OK;
}

template <typename D>
int upload(S& s, D** dst, const std::vector<D>& src, cudaStream_t st) {
  int r = s.alloc(dst, src.size() * sizeof(D));
  if (r) return r;
  if (!src.empty()) CK(cudaMemcpyAsync(*dst, src.data(), src.size() * sizeof(D), cudaMemcpyHostToDevice, st));
  return WENO_OK;
}

// Upload a double table in the solver's precision.
int upload_real(S& s, void** dst, const std::vector<double>& src, cudaStream_t st) {
  if (s.fp64) {
    double* d;
    int r = upload(s, &d, src, st);
    *dst = d;
    return r;
  }
  std::vector<float> f(src.size());
  for (size_t i = 0; i < src.size(); ++i) f[i] = (float)src[i];
  float* d;
  int r = upload(s, &d, f, st);
  if (r) return r;
  CK(cudaStreamSynchronize(st));  // f goes out of scope
  *dst = d;
  return WENO_OK;
}

// FP32C tables, rows of P >= N cells (padding zero, every row on a 256-byte boundary):
//   gop [j][q]        float4 D_j^+ entries
//   dg  [g][q]        float4 (x_G - c0, sigma+, sigma-)
//   gam [g][k][q]     float4 rows: gamma+_{4k..4k+3} for k < M/4, then gamma- rows
//   gam1 [g][q]       float2 (gamma+_8, gamma-_8) of triangles
// The splitting of Section 3.4 depends on the geometry only; it is evaluated
// here in FP64: gt+ = (gamma + theta|gamma|)/2, gt- = gt+ - gamma,
// sigma+- = sum gt+-, gamma+- = gt+- / sigma+-.  rows = false uploads gop only.
int upload_packed(S& s, const GroupTables& T, int64_t P, double theta, void** gop, void** dg, void** gam,
                  void** gam1, cudaStream_t st, bool rows = true) {
  const int64_t N = T.N;
  const int M = T.M, G = T.G, M4 = M / 4;
  std::vector<float> a((size_t)M * 4 * P, 0.f), b((size_t)G * 4 * P, 0.f), c((size_t)G * 2 * M4 * 4 * P, 0.f), e;
  if (M % 4) e.assign((size_t)G * 2 * P, 0.f);
  for (int j = 0; j < M; ++j)
    for (int64_t q = 0; q < N; ++q)
      for (int k = 0; k < 4; ++k) a[((size_t)j * P + q) * 4 + k] = (float)T.gop[((size_t)j * 4 + k) * N + q];
  std::vector<double> gp(M), gn(M);
  for (int g = 0; g < G; ++g) {
    for (int64_t q = 0; q < N; ++q) {
      double sp = 0.0, sm = 0.0;
      for (int j = 0; j < M; ++j) {
        const double x = T.gam[((size_t)g * M + j) * N + q];
        gp[j] = 0.5 * (x + theta * std::fabs(x));
        gn[j] = gp[j] - x;
        sp += gp[j];
        sm += gn[j];
      }
      float* d = &b[((size_t)g * P + q) * 4];
      d[0] = (float)T.dg[((size_t)g * 2 + 0) * N + q];
      d[1] = (float)T.dg[((size_t)g * 2 + 1) * N + q];
      d[2] = (float)sp;
      d[3] = (float)sm;
      for (int j = 0; j < 4 * M4; ++j) {
        c[(((size_t)g * 2 * M4 + j / 4) * P + q) * 4 + j % 4] = (float)(gp[j] / sp);
        c[(((size_t)g * 2 * M4 + M4 + j / 4) * P + q) * 4 + j % 4] = (float)(gn[j] / sm);
      }
      if (M % 4) {
        e[((size_t)g * P + q) * 2] = (float)(gp[M - 1] / sp);
        e[((size_t)g * P + q) * 2 + 1] = (float)(gn[M - 1] / sm);
      }
    }
  }
  float *pa, *pb = nullptr, *pc = nullptr, *pe = nullptr;
  int r;
  if ((r = upload(s, &pa, a, st))) return r;
  if (rows && (r = upload(s, &pb, b, st))) return r;
  if (rows && (r = upload(s, &pc, c, st))) return r;
  if (rows && M % 4 && (r = upload(s, &pe, e, st))) return r;
  CK(cudaStreamSynchronize(st));  // the host vectors go out of scope
  *gop = pa;
  *dg = pb;
  *gam = pc;
  *gam1 = pe;
  return WENO_OK;
}

// Point-pair tables of the Euler FP32C reconstruction (k_reconstruct_tma), rows of P >= N cells
// of float4, the G Gauss points of a cell taken as G/2 pairs (points 2k, 2k+1 of face k):
//   gam [k][j][q]   (gamma+_j(2k), gamma+_j(2k+1), gamma-_j(2k), gamma-_j(2k+1))
//   dg  [2k][q]     (dx(2k), dx(2k+1), dy(2k), dy(2k+1)), (dx, dy) = x_G - c0
//   dg  [2k+1][q]   (sigma+(2k), sigma+(2k+1), sigma-(2k), sigma-(2k+1))
// with the splitting of Section 3.4 evaluated in FP64 as in upload_packed.
int upload_pairs(S& s, const GroupTables& T, int64_t P, double theta, void** gam, void** dg, cudaStream_t st) {
  const int64_t N = T.N;
  const int M = T.M, G = T.G;
  std::vector<float> a((size_t)(G / 2) * M * 4 * P, 0.f), b((size_t)G * 4 * P, 0.f);
  std::vector<double> gp(M), gn(M);
  for (int g = 0; g < G; ++g) {
    const int k = g / 2, h = g % 2;
    for (int64_t q = 0; q < N; ++q) {
      double sp = 0.0, sm = 0.0;
      for (int j = 0; j < M; ++j) {
        const double x = T.gam[((size_t)g * M + j) * N + q];
        gp[j] = 0.5 * (x + theta * std::fabs(x));
        gn[j] = gp[j] - x;
        sp += gp[j];
        sm += gn[j];
      }
      for (int j = 0; j < M; ++j) {
        float* r = &a[(((size_t)k * M + j) * P + q) * 4];
        r[h] = (float)(gp[j] / sp);
        r[2 + h] = (float)(gn[j] / sm);
      }
      float* d0 = &b[((size_t)(2 * k) * P + q) * 4];
      float* d1 = &b[((size_t)(2 * k + 1) * P + q) * 4];
      d0[h] = (float)T.dg[((size_t)g * 2 + 0) * N + q];
      d0[2 + h] = (float)T.dg[((size_t)g * 2 + 1) * N + q];
      d1[h] = (float)sp;
      d1[2 + h] = (float)sm;
    }
  }
  float *pa, *pb;
  int r;
  if ((r = upload(s, &pa, a, st))) return r;
  if ((r = upload(s, &pb, b, st))) return r;
  CK(cudaStreamSynchronize(st));  // the host vectors go out of scope
  *gam = pa;
  *dg = pb;
  return WENO_OK;
}

// FP64 tables of the linear weights: gam itself for the linear scheme, otherwise the split weights,
// formed on the device from a temporary copy of gam.
template <int M>
int upload_split(S& s, const GroupTables& T, int64_t pitch, void** gam, void** wt, double2** sig, cudaStream_t st) {
  if (s.prm.linear) return upload_real(s, gam, T.gam, st);
  int r;
  if ((r = s.alloc(wt, sizeof(double2) * (size_t)T.G * M * pitch))) return r;
  if ((r = s.alloc(sig, sizeof(double2) * (size_t)T.G * pitch))) return r;
  if (!T.N) return WENO_OK;
  double* tmp = nullptr;
  cudaError_t e = cudaMalloc(&tmp, T.gam.size() * sizeof(double));
  if (e != cudaSuccess) return fail(WENO_ENOMEM, std::string("cudaMalloc: ") + cudaGetErrorString(e));
  e = cudaMemcpyAsync(tmp, T.gam.data(), T.gam.size() * sizeof(double), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) {
    const unsigned blocks = (unsigned)((T.N * T.G + 127) / 128);
    if (s.prm.characteristic)
      weno::dev::k_split_weights<M><<<blocks, 128, 0, st>>>(tmp, T.N, T.G, s.prm.theta, pitch, (double2*)*wt, *sig);
    else
      weno::dev::k_split_weights<M><<<blocks, 128, 0, st>>>(tmp, T.N, T.G, s.prm.theta, pitch, (weno::dev::PosPair*)*wt, *sig);
    e = cudaGetLastError();
  }
  const cudaError_t es = cudaStreamSynchronize(st);
  cudaFree(tmp);
  if (e == cudaSuccess) e = es;
  if (e != cudaSuccess) return fail(WENO_ECUDA, std::string("split weights: ") + cudaGetErrorString(e));
  return WENO_OK;
}

using EncodeTiled = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                 const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// 2D float tensor map: `inner` floats per row, `rows` rows `pitch_bytes` apart, box of
// box_inner x box_rows; out-of-range elements of the last tile are filled with zeros.
int make_map_2d(EncodeTiled enc, CUtensorMap* map, void* base, uint64_t inner, uint64_t rows, uint64_t pitch_bytes,
                uint32_t box_inner, uint32_t box_rows) {
  const cuuint64_t dims[2] = {inner, rows};
  const cuuint64_t strides[1] = {pitch_bytes};
  const cuuint32_t box[2] = {box_inner, box_rows};
  const cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, base, dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(WENO_ECUDA, "cuTensorMapEncodeTiled failed with code " + std::to_string((int)r));
  return WENO_OK;
}

// Tensor maps of the TMA reconstruction (Euler FP32C).
int setup_tma(S& s) {
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult q;
  cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q);
  if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || !fn) return fail(WENO_ECUDA, "cuTensorMapEncodeTiled unavailable");
  EncodeTiled enc = reinterpret_cast<EncodeTiled>(fn);
  // point-pair tables: gamma+- (G/2) * M float4 rows, offsets and sigma+- G float4 rows; D_j^+ M rows
  auto maps = [&](weno::dev::TileMaps& t, void* gam, void* dg, void* gop, int64_t pitch, uint32_t M, uint32_t G) -> int {
    int r;
    if ((r = make_map_2d(enc, &t.gam, gam, 4 * pitch, G / 2 * M, 16 * pitch, 4 * kTile, G / 2 * M))) return r;
    if ((r = make_map_2d(enc, &t.dg, dg, 4 * pitch, G, 16 * pitch, 4 * kTile, G))) return r;
    return make_map_2d(enc, &t.gop, gop, 4 * pitch, M, 16 * pitch, 4 * kTile, M);
  };
  int r;
  if (s.nQ && (r = maps(s.q_maps, s.q_pgam, s.q_pdg, s.q_gop, s.q_pitch, 12, 8))) return r;
  if (s.nT && (r = maps(s.t_maps, s.t_pgam, s.t_pdg, s.t_gop, s.t_pitch, 9, 6))) return r;
  s.tma = true;
  return WENO_OK;
}

int run_step(S& s, void* U, void* Ulo, const double* dts, double dt, cudaStream_t st);

}  // namespace

// ====================================================================== C ABI
extern "C" {

const char* weno_last_error(void) { return g_err.c_str(); }

void weno_params_default(weno_params* p) {
  if (!p) return;
  std::memset(p, 0, sizeof(*p));
  p->eqn = WENO_EQN_EULER;
  p->precision = WENO_FP64;
  p->gas_gamma = 1.4;
  p->adv[0] = 1.0;
  p->adv[1] = 1.0;
  p->eps = 1e-3;
  p->theta = 3.0;
  p->rcond = 1e-12;
  p->optimize = 1;
  p->linear = 0;
  p->n_threads = 0;
}

int weno_mesh_create(const double* node_xy, int64_t n_nodes, const int64_t* cell_ptr, const int64_t* cell_nodes,
                     int64_t n_cells, const weno_mesh_opts* opts, weno_mesh_t* out) {
  if (!node_xy || !cell_ptr || !cell_nodes || !opts || !out) return fail(WENO_EINVAL, "null argument");
  if (opts->bc != WENO_BC_PERIODIC && opts->bc != WENO_BC_OUTFLOW) return fail(WENO_EINVAL, "unknown boundary kind");
  *out = nullptr;
  try {
    auto m = std::make_unique<weno_mesh_s>();
    std::string err;
    int r = weno::build_mesh(node_xy, n_nodes, cell_ptr, cell_nodes, n_cells, opts->bc, opts->origin, opts->extent,
                             opts->walls, opts->wall_from, opts->inflow, m->m, err);
    if (r) return fail(r, err);
    *out = m.release();
  } catch (const std::bad_alloc&) {
    return fail(WENO_ENOMEM, "host allocation failed while building the mesh");
  }
  return WENO_OK;
}

int weno_mesh_concat(const weno_mesh_t* meshes, int32_t n, weno_mesh_t* out) {
  if (!meshes || !out || n <= 0) return fail(WENO_EINVAL, "bad arguments to weno_mesh_concat");
  *out = nullptr;
  try {
    std::vector<const Mesh*> v(n);
    for (int i = 0; i < n; ++i) {
      if (!meshes[i]) return fail(WENO_EINVAL, "null mesh");
      v[i] = &meshes[i]->m;
    }
    auto m = std::make_unique<weno_mesh_s>();
    std::string err;
    int r = weno::concat_meshes(v.data(), n, m->m, err);
    if (r) return fail(r, err);
    *out = m.release();
  } catch (const std::bad_alloc&) {
    return fail(WENO_ENOMEM, "host allocation failed while joining meshes");
  }
  return WENO_OK;
}

int weno_mesh_get_info(weno_mesh_t mesh, weno_mesh_info* info) {
  if (!mesh || !info) return fail(WENO_EINVAL, "null argument");
  const Mesh& m = mesh->m;
  info->n_cells = m.n();
  info->n_quads = m.nQ;
  info->n_tris = m.nT;
  info->n_faces = m.nF;
  info->n_boundary = m.n_boundary;
  info->n_instances = m.n_inst;
  info->n_inflow = (int32_t)std::count(m.fin.begin(), m.fin.end(), (int8_t)1);
  return WENO_OK;
}

int weno_mesh_cell_permutation(weno_mesh_t mesh, int64_t* perm) {
  if (!mesh || !perm) return fail(WENO_EINVAL, "null argument");
  std::copy(mesh->m.perm.begin(), mesh->m.perm.end(), perm);
  return WENO_OK;
}

int weno_mesh_cell_instance(weno_mesh_t mesh, int32_t* instance) {
  if (!mesh || !instance) return fail(WENO_EINVAL, "null argument");
  std::copy(mesh->m.inst.begin(), mesh->m.inst.end(), instance);
  return WENO_OK;
}

int weno_mesh_weight_stats(weno_mesh_t mesh, const weno_params* params, double* max_raw, double* max_opt) {
  if (!mesh || !max_raw || !max_opt) return fail(WENO_EINVAL, "null argument");
  weno_params p;
  if (params) p = *params;
  else weno_params_default(&p);
  weno::LsqParams lp;
  lp.rcond = p.rcond > 0 ? p.rcond : 1e-12;
  lp.optimize = p.optimize != 0;
  lp.n_threads = p.n_threads;
  try {
    GroupTables tq, tt;
    std::string err;
    int r = weno::precompute_tables(mesh->m, lp, tq, tt, err);
    if (r) return fail(r, err);
    for (int64_t i = 0; i < tq.N; ++i) { max_raw[i] = tq.max_raw[i]; max_opt[i] = tq.max_opt[i]; }
    for (int64_t i = 0; i < tt.N; ++i) { max_raw[tq.N + i] = tt.max_raw[i]; max_opt[tq.N + i] = tt.max_opt[i]; }
  } catch (const std::bad_alloc&) {
    return fail(WENO_ENOMEM, "host allocation failed in the precompute");
  }
  return WENO_OK;
}

int weno_mesh_cell_tables(weno_mesh_t mesh, const weno_params* params, int64_t cell, int32_t* slot_cells,
                          double* grad_op, double* gauss_offset, double* gamma, int32_t* mg) {
  if (!mesh || !slot_cells || !grad_op || !gauss_offset || !gamma || !mg) return fail(WENO_EINVAL, "null argument");
  const Mesh& m = mesh->m;
  if (cell < 0 || cell >= m.n()) return fail(WENO_EINVAL, "cell out of range");
  weno_params p;
  if (params) p = *params;
  else weno_params_default(&p);
  const double rcond = p.rcond > 0 ? p.rcond : 1e-12;
  if (!mesh->tables || mesh->tables_rcond != rcond || mesh->tables_optimize != (p.optimize != 0)) {
    try {
      mesh->tables.reset();
      auto tab = std::make_shared<std::pair<GroupTables, GroupTables>>();
      weno::LsqParams lp;
      lp.rcond = rcond;
      lp.optimize = p.optimize != 0;
      lp.n_threads = p.n_threads;
      std::string err;
      int r = weno::precompute_tables(m, lp, tab->first, tab->second, err);
      if (r) return fail(r, err);
      mesh->tables = tab;
      mesh->tables_rcond = rcond;
      mesh->tables_optimize = p.optimize != 0;
    } catch (const std::bad_alloc&) {
      return fail(WENO_ENOMEM, "host allocation failed in the precompute");
    }
  }
  const bool quad = cell < m.nQ;
  const GroupTables& T = quad ? mesh->tables->first : mesh->tables->second;
  const int64_t q = quad ? cell : cell - m.nQ;
  const int64_t N = T.N;
  mg[0] = T.M;
  mg[1] = T.G;
  for (int j = 0; j < T.M; ++j) {
    slot_cells[j] = T.slot[(size_t)j * N + q] & weno::kSlotCell;
    for (int e = 0; e < 4; ++e) grad_op[j * 4 + e] = T.gop[(size_t)(j * 4 + e) * N + q];
  }
  for (int g = 0; g < T.G; ++g) {
    gauss_offset[2 * g] = T.dg[(size_t)(g * 2) * N + q];
    gauss_offset[2 * g + 1] = T.dg[(size_t)(g * 2 + 1) * N + q];
    for (int j = 0; j < T.M; ++j) gamma[g * T.M + j] = T.gam[(size_t)(g * T.M + j) * N + q];
  }
  return WENO_OK;
}

void weno_mesh_destroy(weno_mesh_t mesh) { delete mesh; }

int weno_solver_create(weno_mesh_t mesh, const weno_params* params, void* cuda_stream, weno_solver_t* out) {
  if (!mesh || !params || !out) return fail(WENO_EINVAL, "null argument");
  *out = nullptr;
  const weno_params& p = *params;
  if (p.eqn != WENO_EQN_SCALAR && p.eqn != WENO_EQN_EULER) return fail(WENO_EINVAL, "unknown equation");
  if (p.precision != WENO_FP64 && p.precision != WENO_FP32C) return fail(WENO_EINVAL, "unknown precision");
  // theta > 1 keeps sigma- = sum (theta |gamma| - gamma) / 2 > 0 (Section 3.4); at theta = 1 a Gauss
  // point whose linear weights are all >= 0 has sigma- = 0 and gamma- = 0 / 0
  if (!(p.eps > 0) || !(p.theta > 1) || (p.eqn == WENO_EQN_EULER && !(p.gas_gamma > 1)))
    return fail(WENO_EINVAL, "parameters out of range (eps > 0, theta > 1, gamma > 1)");
  // FP32 weights: alpha = gamma / (beta~ + eps)^2 <= 1 / eps^2 stays far inside the FP32 range
  if (p.precision == WENO_FP32C && !(p.eps >= 1e-15))
    return fail(WENO_EINVAL, "FP32C solvers need eps >= 1e-15 (FP32 range of the nonlinear weights); use FP64");
  if (p.characteristic && p.eqn != WENO_EQN_EULER)
    return fail(WENO_EINVAL, "characteristic variables are defined for the Euler equations only");
  const bool walls = std::any_of(mesh->m.fwall.begin(), mesh->m.fwall.end(), [](int8_t w) { return w >= 0; });
  if (walls && p.eqn != WENO_EQN_EULER) return fail(WENO_EINVAL, "reflective walls are defined for the Euler equations only");
  const int64_t n_in = std::count(mesh->m.fin.begin(), mesh->m.fin.end(), (int8_t)1);
  if (n_in && p.eqn != WENO_EQN_EULER) return fail(WENO_EINVAL, "inflow faces are defined for the Euler equations only");
  if (n_in && !(p.inflow_a[0] > 0 && p.inflow_a[3] > 0 && p.inflow_b[0] > 0 && p.inflow_b[3] > 0 &&
                std::isfinite(p.inflow_a[1] + p.inflow_a[2] + p.inflow_b[1] + p.inflow_b[2]) &&
                std::isfinite(p.inflow_line[0] + p.inflow_line[1] + p.inflow_line[2] + p.inflow_line[3])))
    return fail(WENO_EINVAL, "inflow faces need both prescribed states with rho > 0, p > 0 and a finite line");
  const Mesh& m = mesh->m;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  std::unique_ptr<S> s;
  try {
    s.reset(new S());
  } catch (const std::bad_alloc&) {
    return fail(WENO_ENOMEM, "host allocation failed");
  }
  CK(cudaGetDevice(&s->dev));
  CK(cudaDeviceGetAttribute(&s->nsm, cudaDevAttrMultiProcessorCount, s->dev));
  CK(cudaDeviceGetAttribute(&s->l2_bytes, cudaDevAttrL2CacheSize, s->dev));
  s->prm = p;
  s->walls = walls;
  s->n_in = n_in;
  if (!(s->prm.rcond > 0)) s->prm.rcond = 1e-12;
  s->nv = p.eqn == WENO_EQN_EULER ? 4 : 1;
  s->fp64 = p.precision == WENO_FP64;
  s->esz = s->fp64 ? 8 : 4;
  s->nQ = m.nQ;
  s->nT = m.nT;
  s->N = m.n();
  s->nF = m.nF;
  s->n_boundary = m.n_boundary;
  s->n_inst = m.n_inst;
  // precompute on the host (FP64), shared by solvers of the same mesh and weight options
  if (!mesh->tables || mesh->tables_rcond != s->prm.rcond || mesh->tables_optimize != (p.optimize != 0)) {
    try {
      mesh->tables.reset();
      auto tab = std::make_shared<std::pair<GroupTables, GroupTables>>();
      weno::LsqParams lp;
      lp.rcond = s->prm.rcond;
      lp.optimize = p.optimize != 0;
      lp.n_threads = p.n_threads;
      std::string err;
      int r = weno::precompute_tables(m, lp, tab->first, tab->second, err);
      if (r) return fail(r, err);
      mesh->tables = tab;
      mesh->tables_rcond = s->prm.rcond;
      mesh->tables_optimize = p.optimize != 0;
    } catch (const std::bad_alloc&) {
      return fail(WENO_ENOMEM, "host allocation failed in the precompute");
    }
  }
  const GroupTables& tq = mesh->tables->first;
  const GroupTables& tt = mesh->tables->second;
  S& d = *s;
  int r;
  if ((r = upload(d, &d.q_slot, tq.slot, st))) return r;
  if ((r = upload(d, &d.t_slot, tt.slot, st))) return r;
  if (d.fp64) {
    if ((r = upload_real(d, &d.q_gop, tq.gop, st))) return r;
    if ((r = upload_real(d, &d.q_dg, tq.dg, st))) return r;
    if ((r = upload_real(d, &d.t_gop, tt.gop, st))) return r;
    if ((r = upload_real(d, &d.t_dg, tt.dg, st))) return r;
    d.q_pitch = (d.nQ + 7) / 8 * 8;
    d.t_pitch = (d.nT + 7) / 8 * 8;
    if ((r = upload_split<12>(d, tq, d.q_pitch, &d.q_gam, &d.q_wt, &d.q_sig, st))) return r;
    if ((r = upload_split<9>(d, tt, d.t_pitch, &d.t_gam, &d.t_wt, &d.t_sig, st))) return r;
    d.k2.block = 128;  // a warp for each quarter of an SM: the FP64 pipe is split four ways
  } else {
    d.q_pitch = (d.nQ + 63) / 64 * 64;
    d.t_pitch = (d.nT + 63) / 64 * 64;
    // the split-weight rows of upload_packed serve the scalar kernel; both Euler kernels
    // (component-wise and characteristic) read the point-pair tables
    const bool rows = d.nv != 4;
    if ((r = upload_packed(d, tq, d.q_pitch, p.theta, &d.q_gop, &d.q_dg, &d.q_gam, &d.q_gam1, st, rows))) return r;
    if ((r = upload_packed(d, tt, d.t_pitch, p.theta, &d.t_gop, &d.t_dg, &d.t_gam, &d.t_gam1, st, rows))) return r;
    if (d.nv == 4) {
      if ((r = upload_pairs(d, tq, d.q_pitch, p.theta, &d.q_pgam, &d.q_pdg, st))) return r;
      if ((r = upload_pairs(d, tt, d.t_pitch, p.theta, &d.t_pgam, &d.t_pdg, st))) return r;
    }
  }
  {
    std::vector<double> inv(d.N);
    for (int64_t c = 0; c < d.N; ++c) inv[c] = 1.0 / m.area[c];
    if ((r = upload_real(d, &d.area, m.area, st))) return r;
    if ((r = upload_real(d, &d.inv_area, inv, st))) return r;
    // FP32C: the rounding remainder of 1/|Omega| (double-float reciprocal)
    std::vector<double> inv_lo(d.N, 0.0);
    if (!d.fp64)
      for (int64_t c = 0; c < d.N; ++c) inv_lo[c] = inv[c] - (double)(float)inv[c];
    if ((r = upload_real(d, &d.inv_area_lo, inv_lo, st))) return r;
    if ((r = upload(d, &d.area64, m.area, st))) return r;
    CK(cudaStreamSynchronize(st));
  }
  {
    // cell -> face lists with orientation (f: cell is L, ~f: cell is R)
    std::vector<int32_t> cq((size_t)4 * d.nQ), ct((size_t)3 * d.nT);
    for (int64_t c = 0; c < d.N; ++c) {
      const int nf = m.nvert[c];
      for (int k = 0; k < nf; ++k) {
        const int32_t f = m.cell_face[c * 4 + k];
        const bool left = m.fL[f] == (int32_t)c && m.fkL[f] == k;
        const int32_t e = left ? f : ~f;
        if (c < d.nQ) cq[(size_t)k * d.nQ + c] = e;
        else ct[(size_t)k * d.nT + (c - d.nQ)] = e;
      }
    }
    if ((r = upload(d, &d.q_cf, cq, st))) return r;
    if ((r = upload(d, &d.t_cf, ct, st))) return r;
    std::vector<int32_t> gl(d.nF), gr(d.nF);
    auto gbase = [&](int64_t c) -> int64_t { return c < d.nQ ? 8 * c : 8 * d.nQ + 6 * (c - d.nQ); };
    for (int64_t f = 0; f < d.nF; ++f) {
      gl[f] = (int32_t)(gbase(m.fL[f]) + 2 * m.fkL[f]);
      gr[f] = m.fR[f] >= 0 ? (int32_t)(gbase(m.fR[f]) + 2 * m.fkR[f]) : (m.fwall[f] >= 0 ? -2 : -1);
    }
    // inflow faces: gr = -3 - q, and n . x_G - c0 of their two Gauss points (edge k of the
    // L cell: point 0 near node k, point 1 near node k + 1, Eq. 5)
    std::vector<double> xi;
    const double ga = (3.0 + std::sqrt(3.0)) / 6.0, gb = (3.0 - std::sqrt(3.0)) / 6.0;
    const double* ln = p.inflow_line;
    for (int64_t f = 0; f < d.nF; ++f) {
      if (!m.fin[f]) continue;
      gr[f] = (int32_t)(-3 - (int64_t)xi.size() / 2);
      const int64_t c = m.fL[f];
      const int k = m.fkL[f], k1 = (k + 1) % m.nvert[c];
      const double* v = &m.verts[(size_t)c * 8];
      for (int q = 0; q < 2; ++q) {
        const double wa = q == 0 ? ga : gb, wb = q == 0 ? gb : ga;
        const double x = wa * v[2 * k] + wb * v[2 * k1], y = wa * v[2 * k + 1] + wb * v[2 * k1 + 1];
        xi.push_back(ln[0] * x + ln[1] * y - ln[2]);
      }
    }
    if (d.n_in) {
      if ((r = upload(d, &d.in_xi, xi, st))) return r;
      auto cons = [&](const double* q, double* w) {
        w[0] = q[0];
        w[1] = q[0] * q[1];
        w[2] = q[0] * q[2];
        w[3] = q[3] / (p.gas_gamma - 1.0) + 0.5 * q[0] * (q[1] * q[1] + q[2] * q[2]);
      };
      cons(p.inflow_a, d.in_wa);
      cons(p.inflow_b, d.in_wb);
    }
    std::vector<weno::dev::CellFace> faces;
    d.fused = use_fused(d);
    if (d.fused) {
      faces.resize((size_t)4 * d.nQ + (size_t)3 * d.nT);
      for (int64_t f = 0; f < d.nF; ++f) {
        const float nx = (float)m.fnx[f], ny = (float)m.fny[f], len = (float)m.flen[f];
        auto at = [&](int64_t c, int k) { return c < d.nQ ? 4 * c + k : 4 * d.nQ + 3 * (c - d.nQ) + k; };
        faces[at(m.fL[f], m.fkL[f])] = {gr[f] >= 0 ? gr[f] + 1 : gr[f], nx, ny, len};
        if (gr[f] >= 0) faces[at(m.fR[f], m.fkR[f])] = {gl[f] + 1, nx, ny, -len};
      }
      if ((r = upload(d, &d.cell_faces, faces, st))) return r;
    }
    if ((r = upload(d, &d.gl, gl, st))) return r;
    if ((r = upload(d, &d.gr, gr, st))) return r;
    if ((r = upload_real(d, &d.fnx, m.fnx, st))) return r;
    if ((r = upload_real(d, &d.fny, m.fny, st))) return r;
    if ((r = upload_real(d, &d.flen, m.flen, st))) return r;
    if ((r = upload(d, &d.fnx64, m.fnx, st))) return r;
    if ((r = upload(d, &d.fny64, m.fny, st))) return r;
    if ((r = upload(d, &d.flen64, m.flen, st))) return r;
    // instance ranges (quads, triangles) and per-cell instance ids
    std::vector<int64_t> ranges((size_t)4 * d.n_inst, 0);
    for (int i = 0; i < d.n_inst; ++i) { ranges[4 * i] = ranges[4 * i + 1] = -1; ranges[4 * i + 2] = ranges[4 * i + 3] = -1; }
    for (int64_t c = 0; c < d.N; ++c) {
      const int i = m.inst[c];
      const int part = c < d.nQ ? 0 : 2;
      if (ranges[4 * i + part] < 0) ranges[4 * i + part] = c;
      ranges[4 * i + part + 1] = c + 1;
    }
    for (auto& x : ranges) if (x < 0) x = 0;
    // fixed partition of each instance's quad and triangle ranges into chunks, a block each (deterministic
    // reductions): 256 cells, one a thread, up to about eight blocks an SM, then multiples of 256 so that
    // the second level, one block an instance, stays short
    const int64_t chunk = 256 * ((d.N + 256 * 8 * d.nsm - 1) / (256 * 8 * d.nsm));
    std::vector<int64_t> chunks, chunk_off(1, 0);
    for (int i = 0; i < d.n_inst; ++i) {
      for (int part = 0; part < 2; ++part)
        for (int64_t c = ranges[4 * i + 2 * part]; c < ranges[4 * i + 2 * part + 1]; c += chunk) {
          chunks.push_back(c);
          chunks.push_back(std::min(c + chunk, ranges[4 * i + 2 * part + 1]));
        }
      chunk_off.push_back((int64_t)chunks.size() / 2);
    }
    d.n_chunks = (int64_t)chunks.size() / 2;
    if ((r = upload(d, &d.chunks, chunks, st))) return r;
    if ((r = upload(d, &d.chunk_off, chunk_off, st))) return r;
    if ((r = d.alloc(&d.partial, sizeof(double) * std::max<int64_t>(1, d.n_chunks) * d.nv))) return r;
    if (d.n_inst > 1) {
      if ((r = upload(d, &d.inst, m.inst, st))) return r;
    }
    CK(cudaStreamSynchronize(st));
  }
  // scratch
  const int64_t ngauss = 8 * d.nQ + 6 * d.nT;
  if ((r = d.alloc(&d.Wg, (size_t)ngauss * d.nv * d.esz))) return r;
  if ((r = d.alloc(&d.F, (size_t)d.nF * d.nv * d.esz))) return r;
  if ((r = d.alloc(&d.Ws, (size_t)d.N * d.nv * d.esz))) return r;
  if (!d.fp64 && (r = d.alloc(&d.Wslo, (size_t)d.N * d.nv * d.esz))) return r;
  if ((r = d.alloc(&d.dt_dev, sizeof(double) * d.n_inst))) return r;
  if ((r = d.alloc(&d.dt_split, sizeof(float2) * d.n_inst))) return r;
  if ((r = d.alloc(&d.t_dev, sizeof(double) * d.n_inst))) return r;
  CK(cudaMemsetAsync(d.t_dev, 0, sizeof(double) * d.n_inst, st));
  CK(cudaMemsetAsync(d.dt_dev, 0, sizeof(double) * d.n_inst, st));
  CK(cudaHostAlloc((void**)&d.red, sizeof(double) * d.n_inst * d.nv, cudaHostAllocPortable | cudaHostAllocMapped));
  if ((r = d.alloc(&d.flag, sizeof(int) * d.n_inst))) return r;
  CK(cudaMemsetAsync(d.flag, 0, sizeof(int) * d.n_inst, st));
  if ((r = d.alloc(&d.err, sizeof(int)))) return r;
  CK(cudaMemsetAsync(d.err, 0, sizeof(int), st));
  if (!d.fp64 && d.nv == 4 && (r = setup_tma(d))) return r;
  CK(cudaStreamCreateWithFlags(&d.cap, cudaStreamNonBlocking));
  CK(cudaStreamSynchronize(st));
  *out = s.release();
  return WENO_OK;
}

int weno_solver_get_info(weno_solver_t s, weno_mesh_info* info) {
  if (!s || !info) return fail(WENO_EINVAL, "null argument");
  info->n_cells = s->N;
  info->n_quads = s->nQ;
  info->n_tris = s->nT;
  info->n_faces = s->nF;
  info->n_boundary = s->n_boundary;
  info->n_instances = s->n_inst;
  info->n_inflow = (int32_t)s->n_in;
  return WENO_OK;
}

int weno_residual(weno_solver_t s, const void* U, const void* U_lo, void* R, void* cuda_stream) {
  if (!s || !U || !R || (!s->fp64 && !U_lo)) return fail(WENO_EINVAL, "null argument");
  DeviceGuard g(s->dev);
  cudaStream_t st = (cudaStream_t)cuda_stream;
  WENO_DISPATCH(*s, launch_reconstruct, *s, U, U_lo, st);
  WENO_DISPATCH(*s, launch_update, *s, 0, 0.0, s->Wg, s->F, const_cast<void*>(U), const_cast<void*>(U_lo), R, st);
  return check_launch();
}

int weno_pass(weno_solver_t s, int32_t pass, const void* U, const void* U_lo, void* cuda_stream) {
  if (!s || (pass == 1 && (!U || (!s->fp64 && !U_lo)))) return fail(WENO_EINVAL, "null argument");
  if (pass < 1 || pass > 3) return fail(WENO_EINVAL, "pass must be 1, 2 or 3");
  DeviceGuard g(s->dev);
  cudaStream_t st = (cudaStream_t)cuda_stream;
  if (pass == 1) WENO_DISPATCH(*s, launch_reconstruct, *s, U, U_lo, st);
  else if (pass == 2) WENO_DISPATCH(*s, launch_pass2, *s, st);
  else WENO_DISPATCH(*s, launch_pass3, *s, st);
  return check_launch();
}

int weno_step_instances(weno_solver_t s, void* U, void* U_lo, const double* dt_dev, void* cuda_stream) {
  if (!s || !U || !dt_dev || (!s->fp64 && !U_lo)) return fail(WENO_EINVAL, "null argument");
  DeviceGuard g(s->dev);
  return run_step(*s, U, U_lo, dt_dev, 0.0, (cudaStream_t)cuda_stream);
}

int weno_set_time(weno_solver_t s, double t, void* cuda_stream) {
  if (!s || !std::isfinite(t)) return fail(WENO_EINVAL, "null solver or non-finite time");
  DeviceGuard g(s->dev);
  weno::dev::k_fill<<<(s->n_inst + 127) / 128, 128, 0, (cudaStream_t)cuda_stream>>>(s->t_dev, t, s->n_inst);
  CK(cudaGetLastError());
  return WENO_OK;
}

int weno_get_time(weno_solver_t s, double* t_out, void* cuda_stream) {
  if (!s || !t_out) return fail(WENO_EINVAL, "null argument");
  DeviceGuard g(s->dev);
  cudaStream_t st = (cudaStream_t)cuda_stream;
  CK(cudaMemcpyAsync(t_out, s->t_dev, sizeof(double) * s->n_inst, cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  return WENO_OK;
}

int weno_step(weno_solver_t s, void* U, void* U_lo, double dt, void* cuda_stream) {
  if (!s || !U || (!s->fp64 && !U_lo)) return fail(WENO_EINVAL, "null argument");
  if (!(dt >= 0)) return fail(WENO_EINVAL, "dt must be >= 0");
  DeviceGuard g(s->dev);
  cudaStream_t st = (cudaStream_t)cuda_stream;
  return run_step(*s, U, U_lo, nullptr, dt, st);
}

int weno_max_dt(weno_solver_t s, const void* U, const void* U_lo, double cfl, double* dt_out, void* cuda_stream) {
  if (!s || !U || !dt_out || (!s->fp64 && !U_lo)) return fail(WENO_EINVAL, "null argument");
  DeviceGuard g(s->dev);
  cudaStream_t st = (cudaStream_t)cuda_stream;
  WENO_DISPATCH(*s, launch_max_dt, *s, U, U_lo, st);
  int r = check_launch();
  if (r) return r;
  CK(cudaStreamSynchronize(st));
  for (int i = 0; i < s->n_inst; ++i) dt_out[i] = cfl * s->red[i];
  return WENO_OK;
}

int weno_conservation(weno_solver_t s, const void* U, const void* U_lo, double* sums, void* cuda_stream) {
  if (!s || !U || !sums || (!s->fp64 && !U_lo)) return fail(WENO_EINVAL, "null argument");
  DeviceGuard g(s->dev);
  cudaStream_t st = (cudaStream_t)cuda_stream;
  WENO_DISPATCH(*s, launch_sums, *s, U, U_lo, st);
  int r = check_launch();
  if (r) return r;
  CK(cudaStreamSynchronize(st));
  std::memcpy(sums, s->red, sizeof(double) * s->n_inst * s->nv);
  return WENO_OK;
}

int weno_check(weno_solver_t s, void* cuda_stream) {
  if (!s) return fail(WENO_EINVAL, "null argument");
  DeviceGuard g(s->dev);
  cudaStream_t st = (cudaStream_t)cuda_stream;
  std::vector<int> h(s->n_inst, 0);
  int t = 0;
  CK(cudaMemcpyAsync(h.data(), s->flag, sizeof(int) * s->n_inst, cudaMemcpyDeviceToHost, st));
  CK(cudaMemcpyAsync(&t, s->err, sizeof(int), cudaMemcpyDeviceToHost, st));
  CK(cudaMemsetAsync(s->flag, 0, sizeof(int) * s->n_inst, st));
  CK(cudaMemsetAsync(s->err, 0, sizeof(int), st));
  CK(cudaStreamSynchronize(st));
  if (t) return fail(WENO_ETIMEOUT, "a bounded wait for a tensor-memory copy gave up; results of that launch are invalid");
  int bad = 0;
  for (int i = 0; i < s->n_inst; ++i) bad += h[i] != 0;
  if (bad)
    return fail(WENO_ENONPHYS, "non-physical state (rho <= 0, p <= 0 or non-finite) at a Gauss point in " +
                                   std::to_string(bad) + " of " + std::to_string(s->n_inst) + " instance(s)");
  return WENO_OK;
}

int weno_check_instances(weno_solver_t s, int32_t* flags, void* cuda_stream) {
  if (!s || !flags) return fail(WENO_EINVAL, "null argument");
  DeviceGuard g(s->dev);
  cudaStream_t st = (cudaStream_t)cuda_stream;
  int t = 0;
  CK(cudaMemcpyAsync(flags, s->flag, sizeof(int) * s->n_inst, cudaMemcpyDeviceToHost, st));
  CK(cudaMemcpyAsync(&t, s->err, sizeof(int), cudaMemcpyDeviceToHost, st));
  CK(cudaMemsetAsync(s->flag, 0, sizeof(int) * s->n_inst, st));
  CK(cudaMemsetAsync(s->err, 0, sizeof(int), st));
  CK(cudaStreamSynchronize(st));
  if (t) return fail(WENO_ETIMEOUT, "a bounded wait for a tensor-memory copy gave up; results of that launch are invalid");
  return WENO_OK;
}

int weno_solver_launch_config(weno_solver_t s, int32_t* cfg) {
  if (!s || !cfg) return fail(WENO_EINVAL, "null argument");
  const Launch l[3] = {cell_launch(*s), face_launch(*s), gather_launch(*s)};
  for (int i = 0; i < 3; ++i) {
    cfg[2 * i] = l[i].block;
    cfg[2 * i + 1] = l[i].grid;
  }
  return WENO_OK;
}

int weno_solver_debug_stall(weno_solver_t s, int32_t on) {
  if (!s) return fail(WENO_EINVAL, "null argument");
  if (!s->tma) return fail(WENO_EINVAL, "this solver's kernels have no bounded waits (FP32C Euler only)");
  s->debug_stall = on != 0;
  s->drop_graphs();
  return WENO_OK;
}

int weno_autotune(weno_solver_t s, const void* U, const void* U_lo, void* cuda_stream) {
  if (!s || !U || (!s->fp64 && !U_lo)) return fail(WENO_EINVAL, "null argument");
  DeviceGuard g(s->dev);
  cudaStream_t st = (cudaStream_t)cuda_stream;
  cudaEvent_t e0, e1;
  CK(cudaEventCreate(&e0));
  CK(cudaEventCreate(&e1));
  const int blocks[3] = {64, 128, 256};
  // grid candidates: one item per thread, or 1, 2, 4 resident waves of a persistent grid
  const int waves[4] = {0, 1, 2, 4};
  std::vector<Launch> generic, tma;
  for (int b : blocks)
    for (int w : waves) generic.push_back(Launch{b, w == 0 ? 0 : w * s->nsm * std::max(1, 2048 / b)});
  // TMA reconstruction: TILE x 4 threads; 1-4 blocks of 256 threads per SM (persistent), or one block per tile
  for (int w : {0, 1, 2, 3, 4}) tma.push_back(Launch{kTile * 4, w * s->nsm * (64 / kTile)});
  auto tune = [&](Launch& L, auto run, const std::vector<Launch>& cands) -> int {
    float best = 1e30f;
    Launch bestL = L;
    for (const Launch& c : cands) {
      {
        L = c;
        run();
        float tmin = 1e30f;
        for (int rep = 0; rep < 3; ++rep) {
          cudaEventRecord(e0, st);
          run();
          cudaEventRecord(e1, st);
          cudaEventSynchronize(e1);
          float ms = 0.f;
          cudaEventElapsedTime(&ms, e0, e1);
          tmin = std::min(tmin, ms);
        }
        if (cudaGetLastError() != cudaSuccess) continue;  // configuration not launchable
        if (tmin < best) { best = tmin; bestL = c; }
      }
    }
    L = bestL;
    return WENO_OK;
  };
  S& d = *s;
  const std::vector<Launch>& k1c = d.tma ? tma : generic;
  // What is tuned is what a residual launches: the blocks of the FP64 reconstruction and of the characteristic one
  // with a set of threads for every face follow from the mesh; both cell types in one launch take k1q; fluxes and
  // gather in one kernel have a lane for every face.  The passes after the reconstruction work on the Gauss values
  // and fluxes of U.
  WENO_DISPATCH(d, launch_reconstruct, d, U, U_lo, st);
  WENO_DISPATCH(d, launch_pass2, d, st);
  if (!d.fp64 && !split_form(d)) {
    const bool merged = d.tma && merge_kinds(d);
    const int first = merged ? 3 : 1;
    if (d.nQ) tune(d.k1q, [&] { WENO_DISPATCH(d, launch_reconstruct, d, U, U_lo, st, first); }, k1c);
    if (d.nT && !merged) tune(d.k1t, [&] { WENO_DISPATCH(d, launch_reconstruct, d, U, U_lo, st, 2); }, k1c);
  }
  if (!d.fused) {
    tune(d.k2, [&] { WENO_DISPATCH(d, launch_pass2, d, st); }, generic);
    tune(d.k3, [&] { WENO_DISPATCH(d, launch_pass3, d, st); }, generic);
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  CK(cudaStreamSynchronize(st));
  CK(cudaGetLastError());
  d.drop_graphs();
  return WENO_OK;
}

void weno_solver_destroy(weno_solver_t s) { delete s; }

}  // extern "C"

namespace {

int capture_step(S& s, void* U, void* Ulo) {
  cudaGraph_t graph = nullptr;
  CK(cudaStreamBeginCapture(s.cap, cudaStreamCaptureModeThreadLocal));
  WENO_DISPATCH(s, launch_step_body, s, U, Ulo, s.cap);
  cudaError_t le = cudaGetLastError();
  cudaError_t ce = cudaStreamEndCapture(s.cap, &graph);
  if (le != cudaSuccess) {
    if (graph) cudaGraphDestroy(graph);
    return fail(WENO_ECUDA, std::string("kernel launch in capture: ") + cudaGetErrorString(le));
  }
  if (ce != cudaSuccess) return fail(WENO_ECUDA, std::string("cudaStreamEndCapture: ") + cudaGetErrorString(ce));
  cudaGraphExec_t exec = nullptr;
  cudaError_t ie = cudaGraphInstantiate(&exec, graph, 0);
  cudaGraphDestroy(graph);
  if (ie != cudaSuccess) return fail(WENO_ECUDA, std::string("cudaGraphInstantiate: ") + cudaGetErrorString(ie));
  if (s.graphs.size() >= 8) {
    cudaGraphExecDestroy(s.graphs.front().exec);
    s.graphs.erase(s.graphs.begin());
  }
  s.graphs.push_back({U, Ulo, exec});
  return WENO_OK;
}

// Whether k_set_dt may read p itself: doubles in the memory of the solver's device.  A copy also reaches another
// device's memory and starts at any byte.
bool readable_here(const S& s, const double* p) {
  cudaPointerAttributes a{};
  if (reinterpret_cast<uintptr_t>(p) % alignof(double) || cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();  // an error here is the copy's to report
    return false;
  }
  return a.type == cudaMemoryTypeDevice && a.device == s.dev;
}

// One step with the time steps dts[instance] (device), or dt for every instance.
int run_step(S& s, void* U, void* Ulo, const double* dts, double dt, cudaStream_t st) {
  if (dts && !readable_here(s, dts)) {
    CK(cudaMemcpyAsync(s.dt_dev, dts, sizeof(double) * s.n_inst, cudaMemcpyDeviceToDevice, st));
    dts = s.dt_dev;
  }
  weno::dev::k_set_dt<<<(s.n_inst + 127) / 128, 128, 0, st>>>(s.dt_dev, s.dt_split, dts, dt, s.n_inst);
  int r = check_launch();
  if (r) return r;
  cudaGraphExec_t exec = nullptr;
  for (auto& x : s.graphs)
    if (x.U == U && x.Ulo == Ulo) exec = x.exec;
  if (!exec) {
    if ((r = capture_step(s, U, Ulo))) return r;
    exec = s.graphs.back().exec;
  }
  CK(cudaGraphLaunch(exec, st));
  return WENO_OK;
}

}  // namespace

// ===========================================================================
// Residual whose scratch lives in a fixed array compiled into the library.
//
// For callers that may not allocate device memory once they are running:
// code that works inside a fixed device-memory budget handed out at start-up
// (for example when another component's memory pool owns the rest of the
// GPU), or whose per-step loop is not allowed to make allocation calls.
// weno_residual keeps its Gauss-point values and face fluxes in buffers the
// solver allocated; weno_residual_static puts them in g_static_scratch
// instead and allocates nothing.
namespace {

constexpr size_t kStaticScratchBytes = size_t(16) << 20;  // 16 MiB, held by every GPU that loads the library
constexpr int kMaxStaticDevices = 64;

__device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

std::mutex g_static_mu;
void* g_static_base[kMaxStaticDevices] = {};

// Device address of g_static_scratch on the current device (looked up once
// per device; the host-side symbol itself is not a device address).
int static_scratch_base(int dev, void** base) {
  if (dev < 0 || dev >= kMaxStaticDevices) return fail(WENO_EINVAL, "device index out of range for the static scratch");
  std::lock_guard<std::mutex> lock(g_static_mu);
  if (!g_static_base[dev]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_static_scratch);
    if (e != cudaSuccess || !p)
      return fail(WENO_ECUDA, std::string("cudaGetSymbolAddress(g_static_scratch): ") + cudaGetErrorString(e));
    g_static_base[dev] = p;
  }
  *base = g_static_base[dev];
  return WENO_OK;
}

template <typename T, int NV, bool COMP>
void launch_residual_static(S& s, const void* U, const void* Ulo, void* R, void* wg, void* fl, cudaStream_t st) {
  launch_reconstruct_into<T, NV, COMP>(s, U, Ulo, wg, st, 3);
  launch_update<T, NV, COMP>(s, 0, 0.0, wg, fl, nullptr, nullptr, R, st);
}

}  // namespace

extern "C" int weno_residual_static(weno_solver_t s, const void* U, const void* U_lo, void* R, void* cuda_stream) {
  if (!s || !U || !R || (!s->fp64 && !U_lo)) return fail(WENO_EINVAL, "null argument");
  // Gauss-point values first, face fluxes after them on a 256-byte boundary; after those FP32C Euler solvers
  // count, but do not use, a byte per 16-cell tile and a bit per cell: the limit the header states, which
  // keeps refusing what it refused
  const size_t wg_bytes = (size_t)(8 * s->nQ + 6 * s->nT) * s->nv * s->esz;
  const size_t f_off = (wg_bytes + 255) / 256 * 256;
  const size_t r_off = (f_off + (size_t)s->nF * s->nv * s->esz + 255) / 256 * 256;
  auto reserve = [](int64_t n) -> size_t {
    const int64_t tiles = (n + 15) / 16;
    return (size_t)((tiles + 15) / 16 * 16 + (2 * tiles + 15) / 16 * 16);
  };
  const size_t need = r_off + (!s->fp64 && s->nv == 4 ? reserve(s->nQ) + reserve(s->nT) : 0);
  if (need > kStaticScratchBytes)
    return fail(WENO_EINVAL, "mesh too large for weno_residual_static: needs " + std::to_string(need) +
                                 " bytes of scratch, the fixed array holds " + std::to_string(kStaticScratchBytes));
  DeviceGuard g(s->dev);
  void* base = nullptr;
  int r = static_scratch_base(s->dev, &base);
  if (r) return r;
  unsigned char* b = static_cast<unsigned char*>(base);
  WENO_DISPATCH(*s, launch_residual_static, *s, U, U_lo, R, b, b + f_off, (cudaStream_t)cuda_stream);
  return check_launch();
}
