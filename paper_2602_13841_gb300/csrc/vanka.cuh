// Inexact space-time Vanka smoother (Sec. 4.3, Eq. LVS, vanka0, DefTildeHn, DefVnAst).
//
// Build (per level, at the level state U):
//   1. v* = sum_a phi_a(t*) V^a at the slab midpoint (one spatial field);
//   2. k_elem: per cell K the spatial element matrices at v*:
//        A_K = nu A + H'(v*) + N^c'(v*) + N^{b,r}   (velocity x velocity, boundary faces included)
//        B_K = B + G^p                                (pressure x velocity)
//        M_K                                          (scalar velocity mass)
//   3. k_patch_small / k_patch_blocked: the patch matrix is the global submatrix on the DoFs of K (all velocity and
//      pressure DoFs of K at all k+1 time nodes), so the velocity blocks sum the element
//      matrices of every neighbour cell sharing both DoFs:
//        S~_K = [ K^tau (x) M_patch + M^tau (x) A_patch ,  M^tau (x) B_K^T ]
//               [ M^tau (x) B_K                         ,  0               ]
//      M^tau = diag(w_a).  S~_K is inverted through its time diagonalisation, one spatial system per
//      eigenvalue, by Gauss-Jordan elimination with partial pivoting (vanka_patch.cuh); the inverse is
//      stored column-major per cell.
// Sweep (additive, damped): d <- d + omega sum_K R_K^T S~_K^{-1} R_K (rhs - J d); the cells' corrections
// are added per node in a fixed order (vanka_stream.cuh; the other smoothers: cells in 2^d colours), so
// that the scatter is race free and deterministic.
#pragma once
#include <cuda_fp16.h>

#include "operator.cuh"

namespace stmg {

template <typename T>
struct VankaArgs {
  LevelArgs<T> L;
  const T* vstar;       // midpoint velocity field (Nv)
  T* EA;                // [cells][mv][mv]   element matrices of the cells ebase, ebase+1, ...
  T* EB;                // [cells][npc][mv]  (the build runs in chunks of cell planes that share
  T* EM;                // [cells][nl][nl]    one scratch; cell c is stored at c - ebase)
  int64_t ebase;
  // Patch inverse of a cell, time-diagonalised: one spatial inverse T_e^{-1} (size m_s = mv +
  // npc) per eigen-block e, column-major with stride inv_stride(m_s, element size); a complex block
  // stores (re, im) pairs.  k+1 units of m_s x stride reals per cell, storage in T, or
  T* inv;
  __half* invh;         // the same scaled to [-1, 1] in FP16 with one FP32 factor per block
  float* scale;         // [cells][nblk]
  int* status;          // set to 1 on a zero pivot
  T* work;              // global workspace of k_patch_blocked (null for on-chip patches) ...
  int64_t wslot;        // ... entries per block slot
};

// Column stride of a stored patch inverse: the smallest st >= m for which one m x st block of
// `es`-byte entries is a whole number of 16-byte units, so that every block and every cell's blob
// starts 16-byte aligned (the bulk copy's requirement) with the least padding (FP32, m = 38: 38).
__host__ __device__ constexpr inline int inv_stride(int m, int es) {
  int st = m;
  while (((long long)m * st * es) % 16 != 0) ++st;
  return st;
}

// Rows of the spatial Vanka patch of Q_{N-1} / P_{N-2}^disc: D N^D velocity DoFs and C(r+D, D)
// pressure modes (r = N - 2), known at compile time so that the row products unroll.
template <int D, int N>
__host__ __device__ constexpr int patch_rows() {
  return D * Shape<D, N>::Q + (D == 2 ? (N - 1) * N / 2 : (N - 1) * N * (N + 1) / 6);
}

// max |x| over the block (all threads receive it)
template <typename T>
__device__ inline T block_absmax(T v) {
  __shared__ T wmax[32];
  for (int off = 16; off > 0; off >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, off));
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) wmax[w] = v;
  __syncthreads();
  if (w == 0) {
    v = (lane < (int)((blockDim.x + 31) >> 5)) ? wmax[lane] : (T)0;
    for (int off = 16; off > 0; off >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, off));
    if (lane == 0) wmax[0] = v;
  }
  __syncthreads();
  v = wmax[0];
  __syncthreads();
  return v;
}

template <int D>
__device__ inline void cell_coords(int64_t cell, int n, int* cc) {
  for (int l = 0; l < D; ++l) { cc[l] = (int)(cell % n); cell /= n; }
}

template <int D, int N>
__device__ inline void node_multi(int i, int* im) {
  im[0] = i % N; im[1] = (i / N) % N; im[2] = (D == 3) ? i / (N * N) : 0;
}

// ---------------------------------------------------------------------------- element matrices
// Element matrices of one cell, computed by the whole block.  `sm` holds the per-cell tables
// (shared memory, or for cells whose tables exceed it a per-block slot of global memory).
template <typename T, int D, int N>
__device__ void elem_cell(const VankaArgs<T>& V, const Tab<T>& tb, int64_t cell, T* sm) {
  constexpr int Q = Shape<D, N>::Q;
  constexpr int NL = Q;                  // local nodes per component (N = n_q)
  constexpr int NF = Shape<D, N>::NF;
  constexpr int MV = D * NL;
  T* s_gphi = sm;                        // [Q][NL][D] physical basis gradients
  T* s_phi = s_gphi + Q * NL * D;        // [Q][NL]
  T* s_jxw = s_phi + Q * NL;             // [Q]
  T* s_v = s_jxw + Q;                    // [Q][D] v* at quadrature points
  T* s_vn = s_v + Q * D;                 // [D][NL] v* nodal
  T* s_f = s_vn + D * NL;                // per face: [NF] jxw, [NF][D] n, [NF] y, [NF][D] v, [NF][NL] phi, [NF][NL] dn
  constexpr int NP = patch_rows<D, N>() - MV;
  constexpr int FSZ = NF * (2 + 2 * D) + 2 * NF * NL + NF * NP;   // ... and [NF][NP] pressure modes
  T* s_misc = s_f + D * FSZ;             // [8]: volume, area
  T(*corner)[3] = reinterpret_cast<T(*)[3]>(s_misc + 8);
  T* s_psi = s_misc + 8 + 24;            // [Q][NP] pressure modes
  __shared__ int s_faces[6];
  __shared__ int s_nf;

  const LevelArgs<T>& L = V.L;
  int cc[3] = {0, 0, 0};
  cell_coords<D>(cell, L.n, cc);
  const int tid = threadIdx.x, nt = blockDim.x;
  if (tid < (1 << D) * D) {
    int c = tid / D, i = tid % D;
    int64_t v = 0, s = 1;
    for (int l = 0; l < D; ++l) { v += (int64_t)(cc[l] + ((c >> l) & 1)) * s; s *= (L.n + 1); }
    corner[c][i] = L.verts[v * D + i];
  }
  for (int e = tid; e < D * NL; e += nt) {
    int c = e / NL, i = e % NL;
    s_vn[e] = V.vstar[c * L.nnodes + global_node<D>(L.N1, cc, N - 1, i, N)];
  }
  if (tid == 0) {
    int nf = 0;
    for (int ax = 0; ax < D; ++ax) {
      if (cc[ax] == 0) s_faces[nf++] = ax * 2 + 0;
      if (cc[ax] == L.n - 1) s_faces[nf++] = ax * 2 + 1;
    }
    s_nf = nf;
  }
  __syncthreads();
  // volume quadrature data
  for (int q = tid; q < Q; q += nt) {
    int tq[3]; node_multi<D, N>(q, tq);
    T xh[3], J[3][3], G[3][3], x[3];
    for (int l = 0; l < D; ++l) xh[l] = tb.qx[tq[l]];
    map_jacobian<T, D>(corner, xh, J, x);
    T det = invert<T, D>(J, G);
    T w = det;
    for (int l = 0; l < D; ++l) w *= tb.qw[tq[l]];
    s_jxw[q] = w;
    for (int m = 0; m < NP; ++m) {
      T psi = tb.P1[tq[0]][tb.modes[m][0]] * tb.P1[tq[1]][tb.modes[m][1]];
      if (D == 3) psi *= tb.P1[tq[2]][tb.modes[m][2]];
      s_psi[q * NP + m] = psi;
    }
    for (int j = 0; j < NL; ++j) {
      int jm[3]; node_multi<D, N>(j, jm);
      T val = 1, gr[3] = {1, 1, 1};
      for (int l = 0; l < D; ++l) {
        val *= tb.B[tq[l]][jm[l]];
        for (int m = 0; m < D; ++m) gr[m] *= (m == l) ? tb.D[tq[l]][jm[l]] : tb.B[tq[l]][jm[l]];
      }
      s_phi[q * NL + j] = val;
      for (int l = 0; l < D; ++l) {
        T acc = 0;
        for (int m = 0; m < D; ++m) acc += G[m][l] * gr[m];
        s_gphi[(q * NL + j) * D + l] = acc;
      }
    }
  }
  __syncthreads();
  for (int e = tid; e < Q * D; e += nt) {
    int q = e / D, c = e % D;
    T acc = 0;
    for (int j = 0; j < NL; ++j) acc += s_phi[q * NL + j] * s_vn[c * NL + j];
    s_v[e] = acc;
  }
  if (tid == 0) { T v = 0; for (int q = 0; q < Q; ++q) v += s_jxw[q]; s_misc[0] = v; }
  __syncthreads();
  // boundary face data (one buffer per boundary face of this cell)
  const int nfaces = s_nf;
  for (int f = 0; f < nfaces; ++f) {
    const int axis = s_faces[f] / 2, side = s_faces[f] % 2;
    T* F = s_f + f * FSZ;
    T* f_jxw = F; T* f_n = F + NF; T* f_y = f_n + NF * D; T* f_v = f_y + NF; T* f_phi = f_v + NF * D;
    T* f_dn = f_phi + NF * NL;
    for (int p = tid; p < NF; p += nt) {
      int pq[2] = {p % N, p / N};
      int qq[3] = {0, 0, 0};
      { int ti = 0; for (int l = 0; l < D; ++l) if (l != axis) qq[l] = pq[ti++]; }
      T xh[3], J[3][3], G[3][3], x[3];
      for (int l = 0; l < D; ++l) xh[l] = (l == axis) ? (T)side : tb.qx[qq[l]];
      map_jacobian<T, D>(corner, xh, J, x);
      T det = invert<T, D>(J, G);
      const T nh = side ? (T)1 : (T)-1;
      T cof[3], len2 = 0;
      for (int i = 0; i < D; ++i) { cof[i] = det * G[axis][i] * nh; len2 += cof[i] * cof[i]; }
      T dS = sqrt(len2), w = dS;
      for (int l = 0; l < D; ++l) if (l != axis) w *= tb.qw[qq[l]];
      f_jxw[p] = w;
      T nrm[3];
      for (int i = 0; i < D; ++i) { nrm[i] = cof[i] / dS; f_n[p * D + i] = nrm[i]; }
      T ghat[3];
      for (int m = 0; m < D; ++m) { T acc = 0; for (int l = 0; l < D; ++l) acc += G[m][l] * nrm[l]; ghat[m] = acc; }
      T vv[3] = {0, 0, 0};
      for (int j = 0; j < NL; ++j) {
        T wv, wg[3];
        face_weights<T, D, N>(tb, axis, side, pq, j, wv, wg);
        T dn = 0;
        for (int m = 0; m < D; ++m) dn += ghat[m] * wg[m];
        f_phi[p * NL + j] = wv;
        f_dn[p * NL + j] = dn;
        for (int c = 0; c < D; ++c) vv[c] += wv * s_vn[c * NL + j];
      }
      T y = 0;
      for (int c = 0; c < D; ++c) { f_v[p * D + c] = vv[c]; y += vv[c] * nrm[c]; }
      f_y[p] = y;
      for (int m = 0; m < NP; ++m) f_dn[NF * NL + p * NP + m] = face_psi<T, D, N>(tb, axis, side, pq, m);
    }
    __syncthreads();
    if (tid == 0) { T a = 0; for (int p = 0; p < NF; ++p) a += f_jxw[p]; s_misc[1 + f] = a; }
    __syncthreads();
  }
  // velocity block: entry (c, i ; e, j) = row (test c, i), column (trial e, j).  A thread computes a
  // tile of TI test nodes x TJ trial nodes for all components: with g_ce = sum_q w v_c phi_j d_e phi_i
  // the convection part is -(g_ce + delta_ce sum_l g_ll), so per Gauss point and node pair the whole
  // D x D block costs D^2 + D + 1 multiply-adds on values shared by the tile (3D Q3/P2, 4096 cells:
  // 9.6 -> 1.2 ms against one matrix entry at a time).
  constexpr int TI = D == 3 ? 2 : 1, TJ = 4;
  constexpr int NTI = (NL + TI - 1) / TI, NTJ = (NL + TJ - 1) / TJ;
  T* EA = V.EA + (cell - V.ebase) * (int64_t)MV * MV;
  T* EM = V.EM + (cell - V.ebase) * (int64_t)NL * NL;
  for (int tile = tid; tile < NTI * NTJ; tile += nt) {
    const int i0 = tile / NTJ * TI, j0 = (tile - tile / NTJ * NTJ) * TJ;
    int in[TI], jn[TJ];                               // nodes past the end repeat the last one and are not stored
#pragma unroll
    for (int x = 0; x < TI; ++x) in[x] = i0 + x < NL ? i0 + x : NL - 1;
#pragma unroll
    for (int y = 0; y < TJ; ++y) jn[y] = j0 + y < NL ? j0 + y : NL - 1;
    T g[TI][TJ][D][D], sm_[TI][TJ], mass[TI][TJ];     // sm_: the part common to the diagonal blocks
#pragma unroll
    for (int x = 0; x < TI; ++x)
#pragma unroll
      for (int y = 0; y < TJ; ++y) {
        sm_[x][y] = 0;
        mass[x][y] = 0;
#pragma unroll
        for (int c = 0; c < D; ++c)
#pragma unroll
          for (int e = 0; e < D; ++e) g[x][y][c][e] = 0;
      }
#pragma unroll 1
    for (int q = 0; q < Q; ++q) {
      const T w = s_jxw[q];
      T wv[D], gi[TI][D], pi[TI];
#pragma unroll
      for (int c = 0; c < D; ++c) wv[c] = w * s_v[q * D + c];
#pragma unroll
      for (int x = 0; x < TI; ++x) {
        pi[x] = w * s_phi[q * NL + in[x]];
#pragma unroll
        for (int e = 0; e < D; ++e) gi[x][e] = s_gphi[(q * NL + in[x]) * D + e];
      }
#pragma unroll
      for (int y = 0; y < TJ; ++y) {
        const T pj = s_phi[q * NL + jn[y]];
        T wg[D], yc[D];
#pragma unroll
        for (int e = 0; e < D; ++e) wg[e] = w * s_gphi[(q * NL + jn[y]) * D + e];
#pragma unroll
        for (int c = 0; c < D; ++c) yc[c] = wv[c] * pj;
#pragma unroll
        for (int x = 0; x < TI; ++x) {
          mass[x][y] += pi[x] * pj;
#pragma unroll
          for (int e = 0; e < D; ++e) {
            sm_[x][y] += gi[x][e] * wg[e];
#pragma unroll
            for (int c = 0; c < D; ++c) g[x][y][c][e] += gi[x][e] * yc[c];
          }
        }
      }
    }
#pragma unroll
    for (int x = 0; x < TI; ++x)
#pragma unroll
      for (int y = 0; y < TJ; ++y) {
        T tr = 0;
#pragma unroll
        for (int c = 0; c < D; ++c) tr += g[x][y][c][c];
        sm_[x][y] = L.nu * sm_[x][y] - tr;
#pragma unroll
        for (int c = 0; c < D; ++c)
#pragma unroll
          for (int e = 0; e < D; ++e) g[x][y][c][e] = -g[x][y][c][e];
      }
    for (int f = 0; f < nfaces; ++f) {
      const T* F = s_f + f * FSZ;
      const T* f_jxw = F; const T* f_n = F + NF; const T* f_y = f_n + NF * D; const T* f_v = f_y + NF;
      const T* f_phi = f_v + NF * D; const T* f_dn = f_phi + NF * NL;
      const T h = s_misc[0] / s_misc[1 + f] * L.hscale;
      const T p1 = L.nu * L.gamma1 / h, p2 = L.gamma2 / h;
#pragma unroll 1
      for (int p = 0; p < NF; ++p) {
        const T w = f_jxw[p], yn = f_y[p];
        const T ypos = (T)0.5 * (fabs(yn) + yn), yneg = (T)0.5 * (fabs(yn) - yn);
        const T sgn = (yn > 0) ? (T)1 : ((yn < 0) ? (T)-1 : (T)0);
        const T sc = w * (p1 + (L.bconv ? ypos - 2 * yneg : (T)0)), wn = w * L.nu;
        T K[D][D];
#pragma unroll
        for (int c = 0; c < D; ++c)
#pragma unroll
          for (int e = 0; e < D; ++e)
            K[c][e] = w * f_n[p * D + e] *
                      (p2 * f_n[p * D + c] + (L.bconv ? (T)0.5 * ((T)3 - sgn) * f_v[p * D + c] : (T)0));
#pragma unroll
        for (int x = 0; x < TI; ++x) {
          const T pi = f_phi[p * NL + in[x]], di = f_dn[p * NL + in[x]];
#pragma unroll
          for (int y = 0; y < TJ; ++y) {
            const T pj = f_phi[p * NL + jn[y]], dj = f_dn[p * NL + jn[y]];
            const T pp = pi * pj;
            sm_[x][y] += sc * pp - wn * (dj * pi + pj * di);
#pragma unroll
            for (int c = 0; c < D; ++c)
#pragma unroll
              for (int e = 0; e < D; ++e) g[x][y][c][e] += K[c][e] * pp;
          }
        }
      }
    }
#pragma unroll
    for (int x = 0; x < TI; ++x)
#pragma unroll
      for (int c = 0; c < D; ++c)
#pragma unroll
        for (int e = 0; e < D; ++e)
#pragma unroll
          for (int y = 0; y < TJ; ++y)
            if (i0 + x < NL && j0 + y < NL)
              EA[(int64_t)(c * NL + i0 + x) * MV + e * NL + j0 + y] = g[x][y][c][e] + (c == e ? sm_[x][y] : (T)0);
#pragma unroll
    for (int x = 0; x < TI; ++x)
#pragma unroll
      for (int y = 0; y < TJ; ++y)
        if (i0 + x < NL && j0 + y < NL) EM[(i0 + x) * NL + j0 + y] = mass[x][y];
  }
  // pressure x velocity block B_K[m][(e, j)]: a thread per column, all modes
  constexpr int NPC = patch_rows<D, N>() - MV;
  T* EB = V.EB + (cell - V.ebase) * (int64_t)NPC * MV;
  for (int col = tid; col < MV; col += nt) {
    const int e = col / NL, j = col - e * NL;
    T acc[NPC];
#pragma unroll
    for (int m = 0; m < NPC; ++m) acc[m] = 0;
#pragma unroll 1
    for (int q = 0; q < Q; ++q) {
      const T w = s_jxw[q] * s_gphi[(q * NL + j) * D + e];
#pragma unroll
      for (int m = 0; m < NPC; ++m) acc[m] -= s_psi[q * NPC + m] * w;
    }
    for (int f = 0; f < nfaces; ++f) {
      const T* F = s_f + f * FSZ;
      const T* f_jxw = F; const T* f_n = F + NF; const T* f_phi = f_n + NF * D + NF + NF * D;
      const T* f_psi = f_phi + 2 * NF * NL;
#pragma unroll 1
      for (int p = 0; p < NF; ++p) {
        const T w = f_jxw[p] * f_n[p * D + e] * f_phi[p * NL + j];
#pragma unroll
        for (int m = 0; m < NPC; ++m) acc[m] += f_psi[p * NPC + m] * w;
      }
    }
#pragma unroll
    for (int m = 0; m < NPC; ++m) EB[m * MV + col] = acc[m];
  }
}

// Entries of the per-cell tables of elem_cell.
template <int D, int N>
__host__ __device__ constexpr size_t elem_table_entries() {
  constexpr size_t Q = Shape<D, N>::Q, NF = Shape<D, N>::NF, NP = patch_rows<D, N>() - D * Q;
  return Q * Q * D + Q * Q + Q + Q * D + D * Q + D * (NF * (2 + 2 * D) + 2 * NF * Q + NF * NP) + 8 + 24 + Q * NP;
}
// Threads of a block of element matrices: about one node tile each.
template <int D, int N> __host__ __device__ constexpr int elem_threads() { return D == 2 ? 64 : (N == 3 ? 128 : 256); }

template <typename T, int D, int N>
__global__ void k_elem(VankaArgs<T> V, Tab<T> tb, int64_t c0, int64_t c1) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int64_t cell = c0 + blockIdx.x;
  if (cell >= c1) return;
  elem_cell<T, D, N>(V, tb, cell, reinterpret_cast<T*>(smem_raw));
}

// Cells whose tables exceed shared memory (3D Q4/P3): the tables live in a per-block slot of the
// global workspace V.work (elem_table_entries entries per slot); blocks stride over the cells.
template <typename T, int D, int N>
__global__ void k_elem_global(VankaArgs<T> V, Tab<T> tb, int64_t c0, int64_t c1) {
  T* sm = V.work + (int64_t)blockIdx.x * (int64_t)elem_table_entries<D, N>();
  for (int64_t cell = c0 + blockIdx.x; cell < c1; cell += gridDim.x) {
    elem_cell<T, D, N>(V, tb, cell, sm);
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------- Gauss-Jordan
constexpr int kGjBatch = 8;                        // rows loaded ahead in an elimination pass
// In-place inverse of the m x m row-major matrix S (leading dimension ld) with partial (row)
// pivoting; column interchanges undo the row interchanges at the end.  All threads of the
// block take part; returns false (block-uniformly) on a zero pivot.
template <typename T>
__device__ bool gauss_jordan(T* S, int m, int ld, int* piv_row, T* colbuf) {
  const int tid = threadIdx.x, nt = blockDim.x;
  __shared__ int s_piv;
  __shared__ bool s_ok;
  if (tid == 0) s_ok = true;
  for (int p = 0; p < m; ++p) {
    if (tid < 32) {
      T best = -1; int bi = p;
      for (int i = p + tid; i < m; i += 32) {
        T a = fabs(S[i * ld + p]);
        if (a > best) { best = a; bi = i; }
      }
      for (int off = 16; off > 0; off >>= 1) {
        T ob = __shfl_down_sync(0xffffffffu, best, off);
        int oi = __shfl_down_sync(0xffffffffu, bi, off);
        if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
      }
      if (tid == 0) { s_piv = bi; piv_row[p] = bi; if (!(best > 0)) s_ok = false; }
    }
    __syncthreads();
    if (!s_ok) return false;
    const int r = s_piv;
    if (r != p)
      for (int j = tid; j < m; j += nt) { T t = S[p * ld + j]; S[p * ld + j] = S[r * ld + j]; S[r * ld + j] = t; }
    __syncthreads();
    const T pinv = (T)1 / S[p * ld + p];
    __syncthreads();
    for (int j = tid; j < m; j += nt) S[p * ld + j] = (j == p) ? pinv : S[p * ld + j] * pinv;
    for (int i = tid; i < m; i += nt) {
      colbuf[i] = (i == p) ? (T)0 : S[i * ld + p];
    }
    __syncthreads();
    for (int i = tid; i < m; i += nt) if (i != p) S[i * ld + p] = 0;
    __syncthreads();
    // elimination: thread owns column j and every `rs`-th row (no division in the loop); rows
    // in batches of kGjBatch loads before their stores, so that a matrix in global memory is
    // not updated one dependent round trip at a time
    if (nt >= m) {
      const int rs = nt / m;
      if (tid < rs * m) {
        const int j = tid % m, chunk = tid / m;
        const T prow = S[p * ld + j];
        for (int i0 = chunk; i0 < m; i0 += kGjBatch * rs) {
          T v[kGjBatch];
#pragma unroll
          for (int u = 0; u < kGjBatch; ++u) {
            const int i = i0 + u * rs;
            v[u] = i < m ? S[i * ld + j] : (T)0;
          }
#pragma unroll
          for (int u = 0; u < kGjBatch; ++u) {
            const int i = i0 + u * rs;
            if (i < m && i != p) S[i * ld + j] = v[u] - colbuf[i] * prow;
          }
        }
      }
    } else {
      for (int j = tid; j < m; j += nt) {
        const T prow = S[p * ld + j];
        for (int i = 0; i < m; ++i)
          if (i != p) S[i * ld + j] -= colbuf[i] * prow;
      }
    }
    __syncthreads();
  }
  for (int p = m - 1; p >= 0; --p) {
    const int r = piv_row[p];
    if (r != p)
      for (int i = tid; i < m; i += nt) { T t = S[i * ld + p]; S[i * ld + p] = S[i * ld + r]; S[i * ld + r] = t; }
    __syncthreads();
  }
  return true;
}

// ---------------------------------------------------------------------------- patch build
// The cells K' around the cell at cc (offsets o in {-1, 0, 1}^D) that contain both nodes i and j
// of the cell (multi-indices im, jm within it), visited in the order of the offset code
// nb = (o0 + 1) + 3 (o1 + 1) + 9 (o2 + 1): f(nc, ii, jj) gets K''s linear index and the two nodes'
// local indices in K'.  Per dimension at most two offsets qualify (0, and -1 or +1 when both
// nodes lie on that side), so a patch entry visits 1 to 2^D cells instead of testing 3^D.
template <int D, int N, typename F>
__device__ __forceinline__ void for_shared_cells(const int* cc, int n, const int* im, const int* jm, F&& f) {
  int off[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
  int cnt[3] = {1, 1, 1};
  for (int l = 0; l < D; ++l) {
    cnt[l] = 0;
    for (int o = -1; o <= 1; ++o) {
      const int x = cc[l] + o, a = im[l] - o * (N - 1), b = jm[l] - o * (N - 1);
      if (x >= 0 && x < n && a >= 0 && a < N && b >= 0 && b < N) off[l][cnt[l]++] = o;
    }
  }
  for (int u2 = 0; u2 < cnt[2]; ++u2)
    for (int u1 = 0; u1 < cnt[1]; ++u1)
      for (int u0 = 0; u0 < cnt[0]; ++u0) {
        const int o[3] = {off[0][u0], off[1][u1], off[2][u2]};
        int64_t nc = 0, s = 1;
        int ii = 0, jj = 0, si = 1;
        for (int l = 0; l < D; ++l) {
          nc += (int64_t)(cc[l] + o[l]) * s;
          s *= n;
          ii += (im[l] - o[l] * (N - 1)) * si;
          jj += (jm[l] - o[l] * (N - 1)) * si;
          si *= N;
        }
        f(nc, ii, jj);
      }
}

// ---------------------------------------------------------------------------- bulk copies
// Bulk asynchronous copies into shared memory with completion on an mbarrier, and its bounded wait (the
// sweep with exact patches stages its inverses this way; the surrogate's sweep is in vanka_stream.cuh).
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t phase) {
  uint32_t ok;
  asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
               : "=r"(ok) : "r"(bar), "r"(phase) : "memory");
  return ok != 0;
}
__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Bounded wait for phase `phase` of the mbarrier: gives up after `limit_ns` of wall time (and in
// any case after 2^26 rounds).
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t bar, uint32_t phase, uint64_t limit_ns) {
  const uint64_t t0 = global_ns();
  for (int it = 0; it < (1 << 26); ++it) {
    if (mbar_try_wait(bar, phase)) return true;
    if ((it & 63) == 63 && global_ns() - t0 > limit_ns) return false;
  }
  return false;
}
constexpr int kBulkChunk = 32768;                // bytes per bulk copy instruction
constexpr uint64_t kWaitLimit = 1000000000ull;   // 1 s before the wait is declared failed

// Slot strides of a batched sweep (blockIdx.y = slot): inverse entries, FP16 scales, vector entries.
struct SlotStrides { int64_t inv, scale, vec; };

}  // namespace stmg
