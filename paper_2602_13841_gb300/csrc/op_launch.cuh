// Launch helpers for the operator kernels (included by the per-precision translation units).
#pragma once
#include <type_traits>
#include "level.hpp"
#include "operator.cuh"
#include "operator_cells.cuh"
#include "counters.hpp"

namespace stmg {

template <typename T>
LevelArgs<T> level_args(const Level& lv, const Problem& pb, double t0) {
  LevelArgs<T> a{};
  a.verts = std::is_same<T, double>::value ? (const T*)lv.verts64 : (const T*)lv.verts32;
  a.n = lv.n; a.N1 = lv.N1;
  a.nnodes = lv.nnodes; a.Nv = lv.Nv; a.Np = lv.Np;
  a.nu = (T)pb.nu; a.gamma1 = (T)pb.gamma1; a.gamma2 = (T)pb.gamma2;
  a.hscale = (T)lv.hscale;
  a.bconv = pb.bconv; a.problem = pb.problem;
  a.t0 = (T)t0; a.tau = (T)pb.tau;
  a.ftab = pb.ftab; a.gtab = pb.gtab;
  return a;
}

// Cells per block of the cell kernels: the count whose threads fill whole warps best (the FP64 pipe
// is paid for by the warp), the largest among equals; fewer on meshes that would not give every SM
// two blocks.
inline int cells_per_block(int threads_per_cell, int max_threads, int64_t cells) {
  int best = 1;
  double eff = 0.0;
  for (int c = 1; c * threads_per_cell <= max_threads; ++c) {
    const int t = c * threads_per_cell;
    const double e = (double)t / ((t + 31) / 32 * 32);
    if (e >= eff) { eff = e; best = c; }
  }
  const int64_t spread = (cells + 303) / 304;
  return spread < best ? (int)spread : best;
}

// The level's cell buffer for `batch` columns: columns per pass and cell planes per launch -- whole
// columns while they fit, else one column at a time in chunks of planes.
template <typename T, int D, int N>
static bool plan_cellbuf(const Level& lv, int batch, CellBuf<T>& cb, int64_t& cols, int& step) {
  const int kp1 = lv.k + 1;
  const int64_t cplane = D == 2 ? lv.n : (int64_t)lv.n * lv.n;
  cb.s = (T*)lv.cellbuf;
  cb.plane = cplane * Shape<D, N>::Q;
  const int64_t cap = (int64_t)(lv.cellbuf_bytes / sizeof(T)), per = (int64_t)kp1 * D * cb.plane;
  const bool whole = per * lv.n <= cap;
  cb.P = whole ? lv.n : (int)(cap / per);
  if (!cb.s || (!whole && cb.P < 2)) return false;
  cb.comp = cb.plane * cb.P;
  cb.col = cb.comp * kp1 * D;
  cols = whole ? cap / cb.col : 1;
  if (cols > batch) cols = batch;
  if (cols > 32768) cols = 32768;
  step = whole ? lv.n : cb.P - 1;
  return true;
}

// Whether an operator's two launches are chained, by the blocks of its cell kernel.  Blocks placed while the
// previous grid still holds room spread unevenly over the SMs, which costs a grid of about one wave more
// than the gap it saves; grids of up to a block or two per SM and those of many waves gain (2D, in a graph,
// chained / plain: FP32 Q2/P1 DG(0) 32^2 7.1 / 7.7 us, 192^2 11.4 / 10.1; Q3/P2 DG(0) 128^2 11.6 / 10.3; Q3/P2
// DG(2) 96^2 13.9 / 12.7, 256^2 50.6 / 51.0; FP64 Q2/P1 DG(1) 8^2 26.2 / 26.7, 64^2 39.2 / 36.1; Q3/P2 DG(2) 32^2
// 49.0 / 39.7, 256^2 865 / 866).  3D FP64: few long waves, 16^3 Q3/P2 DG(2) residual 745 / 727 us.  The lines are
// where these measurements put them: no one property of the grids (blocks, waves, time of a block) explains
// them all.  2D FP32 calls of one time node are always chained, with a late release: by blocks / so, Q2/P1
// DG(0) 64^2 8.3 / 7.6 us, 128^2 8.9 / 7.9, 192^2 10.9 / 9.9, 256^2 15.8 / 14.9, 512^2 41.0 / 40.7; Q3/P2 DG(0) 128^2
// 11.1 / 10.2 (three time nodes do worse so: 256^2 Q3/P2 DG(2) 51.2 / 54.7).
template <typename T, int D>
static bool chained_cells(int64_t blocks, int kp1) {
  constexpr int64_t sms = 152;
  if (chain_late<T, D>(kp1)) return true;
  if (sizeof(T) == 8) return D == 2 && blocks <= sms;
  return blocks <= 2 * sms || blocks >= 20 * sms;
}

// Node sums of the cell planes z0 .. z1 - 1 (see k_node_sum).
template <typename T, int D, int N>
static void launch_node_sum(const Level& lv, const CellBuf<T>& cb, const T* src, T* y, T alpha, int64_t ys, int z0,
                            int z1, int columns, cudaStream_t s, bool chained = true) {
  const int g0 = z0 * (N - 1), g1 = z1 == lv.n ? lv.N1 : z1 * (N - 1);
  const int64_t nodes = (int64_t)(g1 - g0) * (D == 2 ? (int64_t)lv.N1 : (int64_t)lv.N1 * lv.N1);
  const int64_t blocks = (nodes + 127) / 128;
  auto kern = lv.k == 0 ? k_node_sum<T, D, N, 1> : lv.k == 1 ? k_node_sum<T, D, N, 2> : k_node_sum<T, D, N, 3>;
  launch_if_chained(chained, kern, dim3((unsigned)(blocks < 152 * 64 ? blocks : 152 * 64), columns), 128, 0, s,
                 cb, src, y, alpha, lv.n, lv.N1, lv.nnodes, lv.Nv, ys, g0, nodes);
  note_launch();
}

// One operator call in two launches per chunk (cells, node sums): whole columns while they fit the
// level's cell buffer, else one column at a time in chunks of cell planes.
template <typename T, int D, int N, int MODE>
static cudaError_t launch_dn(const Level& lv, const Problem& pb, double t0, const T* x,
                             const T* state, const T* vprev, T* y, cudaStream_t stream,
                             int batch, int64_t xs, int64_t ys, int64_t ss, const T* nub, const T* rhs) {
  constexpr int TPG = D == 2 ? N : N * N;             // threads per (cell, time node)
  constexpr bool F64 = sizeof(T) == 8;
  // threads per block and blocks per SM, as measured: 2D FP32 at 256^2 Q3/P2 DG(2) 128 x 7 53.3 us,
  // 192 x 5 54.5, 192 x 4 57.4, 256 x 3 57.7, 192 x 3 64.0; 2D FP64 there 128 x 4 879 us, 96 x 4 882, 192 x 2
  // 893, 256 x 1 981; 3D FP32 at 37^3 Q3/P2 DG(1) 128 x 4 284 us, 256 x 2 291, 128 x 5 297, 192 x 2 307; 3D
  // FP64 at 64^3 Q2/P1 DG(2) 192 x 2 12.6 ms, 128 x 3 14.0 (more lanes idle)
  constexpr int BT = D == 2 ? 128 : (N == 5 ? 256 : (F64 ? 192 : 128));
  constexpr int MINB = D == 2 ? (F64 ? 4 : 7) : (N == 5 ? (F64 ? 1 : 2) : (F64 ? 2 : 4));
  const int kp1 = lv.k + 1;
  const Tab<T> tb = make_tab<T>(lv.tabs, pb.tau);
  const T* geo = nullptr;
  const T* fgeo = nullptr;
  if constexpr (D == 2 && F64) { geo = lv.geo64; fgeo = lv.fgeo64; }
  const int64_t cplane = D == 2 ? lv.n : (int64_t)lv.n * lv.n;   // cells per plane of the last axis
  CellBuf<T> cb{};
  int64_t cols;
  int step;
  if (!plan_cellbuf<T, D, N>(lv, batch, cb, cols, step)) return cudaErrorInvalidValue;
  auto kern = [] {
    if constexpr (D == 2) return k_cells2d<T, N, MODE, BT, MINB>; else return k_cells3d<T, N, MODE, BT, MINB>;
  }();
  for (int64_t b0 = 0; b0 < batch; b0 += cols) {
    const int nb = (int)(batch - b0 < cols ? batch - b0 : cols);
    OpArgs<T> A{level_args<T>(lv, pb, t0), x + b0 * xs, state ? state + b0 * ss : nullptr, vprev, y + b0 * ys,
                xs, ys, geo, fgeo, ss, nub ? nub + b0 : nullptr};
    const T* rb = rhs ? rhs + b0 * ys : nullptr;
    for (int z0 = 0; z0 < lv.n; z0 += step) {
      const int z1 = z0 + step < lv.n ? z0 + step : lv.n;
      const int64_t c0 = z0 * cplane, c1 = z1 * cplane;
      const int cpb = cells_per_block(TPG * kp1, BT, (c1 - c0) * nb);
      const size_t smem = D == 2 ? cells2d_smem<T, N>(cpb, kp1) : cells3d_smem<T, N, MODE>(cpb, kp1);
      if (smem > 48 * 1024) {
        cudaError_t e = allow_smem(kern, smem);
        if (e != cudaSuccess) return e;
      }
      const int threads = (cpb * kp1 * TPG + 31) / 32 * 32;
      const int64_t blocks = (c1 - c0 + cpb - 1) / cpb;
      const bool chained = chained_cells<T, D>(blocks * nb, kp1);
      launch_if_chained(chained, kern, dim3((unsigned)blocks, nb), threads, smem, stream, A, tb,
                     cb, c0, c1, cpb, rb);
      note_launch();
      launch_node_sum<T, D, N>(lv, cb, rb, A.y, rhs ? (T)-1 : (T)1, ys, z0, z1, nb, stream, chained);
    }
  }
  return cudaGetLastError();
}

template <typename T, int MODE>
static cudaError_t launch_any(const Level& lv, const Problem& pb, double t0, const T* x,
                              const T* state, const T* vprev, T* y, cudaStream_t s,
                              int batch, int64_t xs, int64_t ys, int64_t ss = 0, const T* nub = nullptr,
                              const T* rhs = nullptr) {
  const int N = lv.r + 2;
#define STMG_LAUNCH(DD, NN) return launch_dn<T, DD, NN, MODE>(lv, pb, t0, x, state, vprev, y, s, batch, xs, ys, ss, nub, rhs)
  if (lv.d == 2) {
    if (N == 3) STMG_LAUNCH(2, 3);
    if (N == 4) STMG_LAUNCH(2, 4);
    if (N == 5) STMG_LAUNCH(2, 5);
  } else {
    if (N == 3) STMG_LAUNCH(3, 3);
    if (N == 4) STMG_LAUNCH(3, 4);
    if (N == 5) STMG_LAUNCH(3, 5);
  }
#undef STMG_LAUNCH
  return cudaErrorInvalidValue;
}

}  // namespace stmg
