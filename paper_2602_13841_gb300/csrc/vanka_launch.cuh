// Vanka launch templates shared by the per-dimension translation units (vanka_d2_*.cu,
// vanka_d3_*.cu) and the dispatch in vanka.cu: shared-memory budgets, the build of one level and
// the launches of one sweep, per element type T, dimension D and N = r + 2.
#pragma once
#include <type_traits>

#include "mg.hpp"
#include "op_launch.cuh"
#include "vanka.cuh"
#include "vanka_patch.cuh"
#include "vanka_stream.cuh"
#include "vanka_diag.cuh"
#include "vanka_exact.cuh"
#include "vec.cuh"
#include "counters.hpp"

namespace stmg {

template <int D, int N>
static constexpr size_t elem_smem(size_t es) { return es * elem_table_entries<D, N>(); }

// Surrogate patches whose whole elimination runs in registers (k_patch_small).
static bool patch_small(const Level& lv, size_t es) { return lv.d == 2 && !(es == 8 && lv.r == 3); }

static size_t elem_smem_any(const Level& lv, size_t es) {
  int N = lv.r + 2;
  if (lv.d == 2) return N == 3 ? elem_smem<2, 3>(es) : N == 4 ? elem_smem<2, 4>(es) : elem_smem<2, 5>(es);
  return N == 3 ? elem_smem<3, 3>(es) : N == 4 ? elem_smem<3, 4>(es) : elem_smem<3, 5>(es);
}

// The patch matrix of a cell stays on the chip (else a global workspace slot per block).
static bool patch_onchip(const Level& lv, size_t es) {
  size_t nl = 1;
  for (int l = 0; l < lv.d; ++l) nl *= (lv.r + 2);
  return patch_small(lv, es) || patch_matrix_onchip((int)vanka_spatial_size(lv), (int)nl, es);
}

// Shared memory of k_patch_diag: inverse temporal blocks, Schur complement, pivots, column.
static size_t patch_diag_smem(const Level& lv, size_t es) {
  const size_t mv = vanka_spatial_size(lv) - lv.npc, kp1 = lv.k + 1, ns = kp1 * lv.npc;
  return es * (mv * kp1 * kp1 + ns * ns + 2 * ns + 2) + sizeof(int) * (ns + 1);
}

// The per-cell tables of the element-matrix kernel fit shared memory (else k_elem_global).
static bool elem_onchip(const Level& lv, size_t es) { return elem_smem_any(lv, es) <= 227 * 1024; }

static size_t elem_table_any(const Level& lv) {
  int N = lv.r + 2;
  if (lv.d == 2) return N == 3 ? elem_table_entries<2, 3>() : N == 4 ? elem_table_entries<2, 4>() : elem_table_entries<2, 5>();
  return N == 3 ? elem_table_entries<3, 3>() : N == 4 ? elem_table_entries<3, 4>() : elem_table_entries<3, 5>();
}


// Block slots of the global build workspace and their size in entries.
constexpr int kWorkSlots = 152 * 2;
static size_t work_slot(const Level& lv, size_t es) {
  return patch_matrix_bytes((int)vanka_spatial_size(lv), es) / es;
}

// v* = sum_a phi_a(t*) V^a
template <typename T>
__global__ void k_midpoint(const T* __restrict__ U, T* __restrict__ vs, int64_t Nv, int kp1, Tab<T> tb) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < Nv; i += (int64_t)gridDim.x * blockDim.x) {
    T acc = 0;
    for (int a = 0; a < kp1; ++a) acc += tb.phi_mid[a] * U[a * Nv + i];
    vs[i] = acc;
  }
}

template <typename T, int D, int N>
static cudaError_t build_dn(const Level& lv, const Problem& pb, const T* U, T* vstar, T* EA, T* EB, T* EM,
                            T* inv, void* invh, float* scale, int* status, T* work, cudaStream_t s) {
  Tab<T> tb = make_tab<T>(lv.tabs, pb.tau);
  int64_t ncells = lv.Np / lv.npc;
  int64_t g = (lv.Nv + 255) / 256; if (g > 152 * 8) g = 152 * 8;
  k_midpoint<T><<<(int)g, 256, 0, s>>>(U, vstar, lv.Nv, lv.k + 1, tb);
  const bool diag = lv.smoother == 1;
  // where the patch matrix and the element tables live follows from (T, D, N) alone
  constexpr int MS = patch_rows<D, N>(), NLOC = Shape<D, N>::Q;
  constexpr bool SMALL = D == 2 && !(sizeof(T) == 8 && N == 5);
  constexpr bool MATRIX_ONCHIP = SMALL || patch_matrix_onchip(MS, NLOC, sizeof(T));
  constexpr bool eon = elem_smem<D, N>(sizeof(T)) <= 227 * 1024;
  const bool onchip = diag || MATRIX_ONCHIP;
  if ((!onchip || !eon) && !work) return cudaErrorInvalidValue;
  VankaArgs<T> V{level_args<T>(lv, pb, 0.0), vstar, EA, EB, EM, 0, inv, (__half*)invh, scale, status,
                 onchip ? nullptr : work, onchip ? 0 : (int64_t)work_slot(lv, sizeof(T))};
  size_t es = elem_smem<D, N>(sizeof(T));
  cudaError_t e = cudaSuccess;
  if constexpr (eon) {
    e = allow_smem(k_elem<T, D, N>, es);
    if (e != cudaSuccess) return e;
  }
  size_t ps = 0;
  if (lv.smoother == 2) {
    if (!eon) return cudaErrorNotSupported;
    const int ms = (int)vanka_spatial_size(lv), mv = ms - lv.npc;
    ps = patch_exact_smem((lv.k + 1) * ms, mv, mv / D, sizeof(T));
    e = allow_smem(k_patch_exact<T, D, N>, ps);
    if (e != cudaSuccess) return e;
  } else if (diag) {
    ps = patch_diag_smem(lv, sizeof(T));
    e = allow_smem(k_patch_diag<T, D, N>, ps);
    if (e != cudaSuccess) return e;
  } else if constexpr (!SMALL) {
    ps = (patch_panel_smem(MS, NLOC, sizeof(T)) + 15) & ~(size_t)15;
    if (MATRIX_ONCHIP) ps += patch_matrix_bytes(MS, sizeof(T));
    e = allow_smem(k_patch_blocked<T, D, N, MATRIX_ONCHIP>, ps);
    if (e != cudaSuccess) return e;
  }
  const TEig<T> te = make_teig<T>(lv.tabs, pb.tau);
  // chunks of whole cell planes (the last coordinate): the element matrices of the chunk and of
  // one plane on either side (the patches' neighbours) fit the scratch of vanka_elem_cells cells
  const int64_t plane = ncells / lv.n;
  int64_t planes = (int64_t)vanka_elem_cells(lv) >= ncells ? lv.n : (int64_t)vanka_elem_cells(lv) / plane - 2;
  if (planes < 1 || planes > lv.n) planes = lv.n;
  for (int64_t z0 = 0; z0 < lv.n; z0 += planes) {
    const int64_t z1 = z0 + planes < lv.n ? z0 + planes : lv.n;
    const int64_t e0 = (z0 > 0 ? z0 - 1 : 0) * plane, e1 = (z1 < lv.n ? z1 + 1 : lv.n) * plane;
    const int64_t p0 = z0 * plane, p1 = z1 * plane;
    V.ebase = e0;
    if (lv.smoother == 2) {
      // exact patches: velocity element blocks at every time node's own state (the level state,
      // velocity part V^a at U + a N_v)
      const int64_t stride = (int64_t)vanka_elem_cells(lv) * (int64_t)vanka_elem_size(lv, 0);
      for (int a = 0; a <= lv.k; ++a) {
        VankaArgs<T> Va = V;
        Va.vstar = U + (int64_t)a * lv.Nv;
        Va.EA = EA + a * stride;
        if constexpr (eon)
          k_elem<T, D, N><<<(unsigned)(e1 - e0), elem_threads<D, N>(), es, s>>>(Va, tb, e0, e1);
      }
      k_patch_exact<T, D, N><<<(unsigned)(p1 - p0), 256, ps, s>>>(V, tb, stride, p0, p1);
      note_launch(lv.k + 2);
      continue;
    }
    if constexpr (eon) {
      k_elem<T, D, N><<<(unsigned)(e1 - e0), elem_threads<D, N>(), es, s>>>(V, tb, e0, e1);
    } else {
      // tables in global memory: one slot per block (the slots precede any patch workspace use,
      // which follows on the same stream)
      VankaArgs<T> Ve = V;
      Ve.work = work;
      const int64_t grid = e1 - e0 < kWorkSlots ? e1 - e0 : kWorkSlots;
      k_elem_global<T, D, N><<<(unsigned)grid, 256, 0, s>>>(Ve, tb, e0, e1);
    }
    if (diag) {
      k_patch_diag<T, D, N><<<(unsigned)(p1 - p0), 128, ps, s>>>(V, tb, p0, p1);
    } else if constexpr (SMALL) {
      k_patch_small<T, D, N><<<(unsigned)((p1 - p0 + kSmallCells - 1) / kSmallCells), kSmallCells * small_team<D, N>(), 0, s>>>(
          V, te, lv.k + 1, p0, p1);
    } else {
      const int64_t grid = MATRIX_ONCHIP || p1 - p0 < kWorkSlots ? p1 - p0 : kWorkSlots;
      k_patch_blocked<T, D, N, MATRIX_ONCHIP><<<(unsigned)grid, blocked_threads<D, N>(), ps, s>>>(V, te, lv.k + 1, p0, p1);
    }
    note_launch(2);
  }
  note_launch(1);
  return cudaGetLastError();
}

// d <- d + omega W y over all cells of a level by the streamed inverses (first: d = 0 on entry).
template <typename T, typename SI, int D, int N>
static cudaError_t apply_stream(const Level& lv, const Problem& pb, const SI* inv, const float* scale, const T* res,
                                T* d, double omega, double omega_p, int* wstat, unsigned extra_tx, cudaStream_t s,
                                int slots, SlotStrides zs, bool first) {
  using Sh = StreamShape<T, SI, D, N>;
  if ((int)vanka_spatial_size(lv) != Sh::MS) return cudaErrorInvalidValue;
  const int kp1 = lv.k + 1;
  CellBuf<T> cb{};
  int64_t cols;
  int step;
  if (!plan_cellbuf<T, D, N>(lv, slots, cb, cols, step)) return cudaErrorInvalidValue;
  const int64_t cplane = D == 2 ? lv.n : (int64_t)lv.n * lv.n;
  // inverses beyond half of the 129 MB L2 are streamed past it
  const int64_t bytes = cplane * lv.n * (int64_t)kp1 * Sh::MS * Sh::ST * (int64_t)sizeof(SI);
  const int stream = bytes * slots > (int64_t)64 << 20;
  const LevelArgs<T> L = level_args<T>(lv, pb, 0.0);
  const TEig<T> te = make_teig<T>(lv.tabs, pb.tau);
  // the kernel's blocks: one real (k = 0), one complex pair (k = 1), one of each (k = 2)
  const int pairs = te.cplx[0] + (te.nblk > 1 ? te.cplx[1] : 0);
  if (te.nblk != (kp1 + 1) / 2 || pairs != kp1 / 2) return cudaErrorNotSupported;
  auto kern = kp1 == 1 ? k_vanka_stream<T, SI, D, N, 1> : kp1 == 2 ? k_vanka_stream<T, SI, D, N, 2> : k_vanka_stream<T, SI, D, N, 3>;
  if (extra_tx) {                                     // a sweep that times out leaves d as it was: the hook alone
    cudaError_t e = first ? cudaMemsetAsync(d, 0, (size_t)slots * zs.vec * sizeof(T), s) : cudaSuccess;
    if (e != cudaSuccess) return e;
    k_wait_hook<<<1, 1, 0, s>>>(wstat, extra_tx);
    note_launch();
    return cudaGetLastError();
  }
  for (int b0 = 0; b0 < slots; b0 += (int)cols) {
    const int nb = slots - b0 < (int)cols ? slots - b0 : (int)cols;
    const T* rb = res + b0 * zs.vec;
    T* db = d + b0 * zs.vec;
    for (int z0 = 0; z0 < lv.n; z0 += step) {
      const int z1 = z0 + step < lv.n ? z0 + step : lv.n;
      launch_chained(kern, dim3((unsigned)((z1 - z0) * cplane), nb), Sh::THREADS, 0, s,
                     L, inv + b0 * zs.inv, scale ? scale + b0 * zs.scale : nullptr, rb, db, (T)omega_p, te, cb, z0 * cplane, zs, first,
          stream);
      note_launch();
      launch_node_sum<T, D, N>(lv, cb, first ? nullptr : db, db, (T)omega, zs.vec, z0, z1, nb, s);
    }
  }
  return cudaGetLastError();
}

template <typename T, int D, int N>
static cudaError_t apply_dn(const Level& lv, const Problem& pb, const T* inv, const void* invh, const float* scale,
                            const T* res, T* d, double omega, double omega_p, int* wstat, unsigned extra_tx,
                            cudaStream_t s, int slots, bool first) {
  const int64_t cells = lv.Np / lv.npc;
  const SlotStrides zs{cells * (int64_t)vanka_inv_entries(lv, invh ? 2 : (int)sizeof(T)), cells * (lv.k + 1),
                       lv.Nst};
  if (lv.smoother == 0)
    return invh ? apply_stream<T, __half, D, N>(lv, pb, (const __half*)invh, scale, res, d, omega, omega_p, wstat,
                                                extra_tx, s, slots, zs, first)
                : apply_stream<T, T, D, N>(lv, pb, inv, nullptr, res, d, omega, omega_p, wstat, extra_tx, s, slots, zs,
                                           first);
  if (first) {
    cudaError_t e = cudaMemsetAsync(d, 0, (size_t)slots * lv.Nst * sizeof(T), s);
    if (e != cudaSuccess) return e;
  }
  // the other smoothers scatter in place, colour by colour
  for (int c = 0; c < lv.ncolors; ++c) {
    const ColorInfo& ci = lv.colors[c];
    if (ci.count == 0) continue;
    if (lv.smoother == 2) {
      const int ms = (int)vanka_spatial_size(lv), mst = (lv.k + 1) * ms;
      const size_t smem = apply_exact_smem(mst, ms, sizeof(T));
      cudaError_t e = allow_smem(k_vanka_apply_exact<T, D, N>, smem);
      if (e != cudaSuccess) return e;
      k_vanka_apply_exact<T, D, N><<<dim3((unsigned)ci.count, slots), ((mst + 31) / 32) * 32, smem, s>>>(
          level_args<T>(lv, pb, 0.0), inv, res, d, (T)omega, (T)omega_p, lv.k + 1, lv.npc, ci, wstat, extra_tx, zs);
    } else {
      // diagonal space-time Vanka: one warp per cell, up to four cells per block
      constexpr int NL = Shape<D, N>::Q;
      const size_t slot = diag_slot_bytes(D * NL, lv.npc, lv.k + 1, sizeof(T));
      int cpb = 4;
      while (cpb > 1 && (size_t)cpb * slot > 200 * 1024) --cpb;
      const size_t smem = (size_t)cpb * slot;
      cudaError_t e = allow_smem(k_vanka_apply_diag<T, D, N>, smem);
      if (e != cudaSuccess) return e;
      k_vanka_apply_diag<T, D, N><<<dim3((unsigned)((ci.count + cpb - 1) / cpb), slots), 32 * cpb, smem, s>>>(
          level_args<T>(lv, pb, 0.0), inv, res, d, (T)omega, (T)omega_p, make_tab<T>(lv.tabs, pb.tau), ci, cpb, zs);
    }
    note_launch();
  }
  return cudaGetLastError();
}


// Dispatch on N for one (T, D), instantiated in the per-dimension translation units.
template <typename T, int D>
cudaError_t vanka_build_dim(const Level& lv, const Problem& pb, const T* U, T* vstar, T* EA, T* EB, T* EM,
                            T* inv, void* invh, float* scale, int* status, T* work, cudaStream_t s) {
  const int N = lv.r + 2;
  if (N == 3) return build_dn<T, D, 3>(lv, pb, U, vstar, EA, EB, EM, inv, invh, scale, status, work, s);
  if (N == 4) return build_dn<T, D, 4>(lv, pb, U, vstar, EA, EB, EM, inv, invh, scale, status, work, s);
  if (N == 5) return build_dn<T, D, 5>(lv, pb, U, vstar, EA, EB, EM, inv, invh, scale, status, work, s);
  return cudaErrorNotSupported;
}

template <typename T, int D>
cudaError_t vanka_apply_dim(const Level& lv, const Problem& pb, const T* inv, const void* invh, const float* scale,
                            const T* res, T* d, double omega, double omega_p, int* wstat, cudaStream_t s,
                            unsigned extra_tx, int slots, bool first) {
  const int N = lv.r + 2;
  if (N == 3) return apply_dn<T, D, 3>(lv, pb, inv, invh, scale, res, d, omega, omega_p, wstat, extra_tx, s, slots, first);
  if (N == 4) return apply_dn<T, D, 4>(lv, pb, inv, invh, scale, res, d, omega, omega_p, wstat, extra_tx, s, slots, first);
  if (N == 5) return apply_dn<T, D, 5>(lv, pb, inv, invh, scale, res, d, omega, omega_p, wstat, extra_tx, s, slots, first);
  return cudaErrorNotSupported;
}

}  // namespace stmg
