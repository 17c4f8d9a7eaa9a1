// Host-side description of one level of the hp space-time hierarchy and the operator launchers.
#pragma once
#include <cuda_runtime.h>

#include <string>
#include <vector>

#include "common.cuh"
#include "refdata.hpp"

namespace stmg {

struct Level {
  int d = 2, n = 0, r = 1, k = 0;
  int N1 = 0, npc = 0;
  int64_t nnodes = 0, Nv = 0, Np = 0, Nst = 0;
  LevelTables tabs{};
  double* verts64 = nullptr;          // device, (n+1)^d * d
  float* verts32 = nullptr;
  ColorInfo colors[8]{};
  int ncolors = 0;
  double hscale = 0;                  // Nitsche length factor (see LevelArgs)
  int64_t chunk_cells = 262144;       // cells per chunk of the smoother build's element scratch
  int smoother = 0;                   // 0: surrogate patches (Sec. 4.3); 1: diagonal space-time Vanka
  double* geo64 = nullptr;            // 2D: geometry tables of the FP64 operator (see OpArgs::geo, fgeo)
  double* fgeo64 = nullptr;
  void* cellbuf = nullptr;            // cell-wise results of the operator kernels (CellBuf), one buffer
  size_t cellbuf_bytes = 0;           // for all levels of a handle, on the handle's stream only
};

struct Problem {
  double nu, tau, gamma1, gamma2;
  int bconv, problem;
  // STMG_USER: f at the volume Gauss points and g at the boundary-face Gauss points of the
  // finest level for the current slab (device tables filled from the host callbacks; see
  // LevelArgs::ftab / gtab for the layout)
  const double* ftab = nullptr;
  const double* gtab = nullptr;
};

template <typename T>
LevelArgs<T> level_args(const Level& lv, const Problem& pb, double t0);

enum OpMode { OP_JAC = 0, OP_RES = 1, OP_MASS = 2 };

// y = operator(x): J(state) x (OP_JAC), R(x; vprev) (OP_RES, FP64 only) or the slab mass
// diag(w_a M_h, w_a M_p) x (OP_MASS).  With batch > 1, column b reads x + b*xs and writes
// y + b*ys (the state is shared).  y is zeroed first.  Enqueued on `stream`.
template <typename T>
cudaError_t launch_operator(const Level& lv, const Problem& pb, int mode, double t0, const T* x,
                            const T* state, const T* vprev, T* y, cudaStream_t stream,
                            int batch = 1, int64_t xs = 0, int64_t ys = 0);

// y = rhs - J(state) x on a level (rhs null: y = J(state) x), the residual of a multigrid sweep.
// `columns` independent residuals at strides n_st (own rhs, x, state, y; per-column viscosity
// nub[column] on the device, or null for pb.nu).
template <typename T>
cudaError_t launch_level_residual(const Level& lv, const Problem& pb, const T* rhs, const T* x, const T* state, T* y,
                                  cudaStream_t stream, int columns = 1, const T* nub = nullptr);

// Bytes of the cell buffer that the operator calls of a level use at most: one column of cell-wise FP64
// results, capped at 1 GiB (larger meshes run in chunks of cell planes; two planes at least), and
// at least 16 MiB, so that the batched applies of small levels share launches.  A group's hierarchy takes its
// level residuals and sweeps for all slots at once: `slots` columns of es-byte results, each capped alike
// (1 to 2 % of a slot's patch inverses).
inline size_t cellbuf_need(int d, int n, int r, int k, int slots = 1, int es = 8) {
  double plane = 8.0 * (k + 1) * d, cells = 1;
  for (int l = 0; l < d; ++l) plane *= r + 2;
  for (int l = 0; l + 1 < d; ++l) cells *= n;
  plane *= cells;
  const double cap = plane * 2 > 1073741824.0 ? plane * 2 : 1073741824.0;
  double b = plane * n;
  const double batch = slots * (b * es / 8.0 < cap ? b * es / 8.0 : cap);
  if (b > cap) b = cap;
  if (b < batch) b = batch;
  return (size_t)(b < 16777216.0 ? 16777216.0 : b);
}

cudaError_t launch_initial_condition(const Level& lv, const Problem& pb, double* V0, cudaStream_t s);

// Fill lv.geo64 and lv.fgeo64 (allocated by the caller: cells x 5 x (r+2)^2 and 4 n x 6 x (r+2) entries) of
// a 2D level.
cudaError_t build_geometry(const Level& lv, const Problem& pb, cudaStream_t s);

}  // namespace stmg
