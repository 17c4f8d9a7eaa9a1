// Patch inverses of the surrogate Vanka smoother: assembly of the spatial systems T_lam and their
// inversion by Gauss-Jordan exchange steps without row interchanges.
//
// Spatial patch ordering: velocity (c, i) -> c*NL + i, then pressure mode m -> MV + m.  The
// surrogate patch matrix of Eq. vanka0 is, time node by time node,
//   S~ = [ K^tau (x) M + W (x) A ,  W (x) B^T ;  W (x) B , 0 ],   W = diag(w_a),
// with the cell's assembled velocity mass M (per component), velocity block A (viscous,
// convection at v*, Nitsche) and divergence block B.  With W^{-1} K^tau = Q diag(lam) Q^{-1}
// it is similar to the block diagonal of T_lam = [lam M + A, B^T; B, 0]: one spatial inverse
// per eigenvalue instead of one inverse of the whole space-time patch (Sec. 4.3).
//
// Exchange form.  y = A x; step p trades x_p for y_(r_p), r_p the row of the largest entry of column p
// among the rows not yet used (partial pivoting).  After all steps the working matrix M holds
// A^{-1}[p][r_q] = M[r_p][q], so nothing is ever swapped: the permutation is applied when the inverse
// is written out.  A thread of the row team owns row i of a panel of PB columns in registers; one
// step is one pivot search (one warp-wide maximum over keys of magnitude bits and row index), the
// pivot row passed on through shared memory, and one update of the registers, which also rotates
// them by one place, so that the current column is always register 0 and the step loop is rolled.
//
// Small patches (2D, at most 64 rows): the panel is the whole matrix and the patch never leaves the
// registers of its one or two warps (k_patch_small).  Larger patches: panels of PB columns; the
// panel's exchange matrix W (m x PB) and the old pivot rows R (PB x m) are kept in shared memory and
// the other columns take C_i <- [i not a pivot row] C_i + W_i R in register tiles, one pass over the
// matrix per panel instead of one per column; the matrix itself is in shared memory where it fits
// (3D Q2/P1), else in an L2-resident workspace slot per block (k_patch_blocked).
#pragma once
#include "vanka.cuh"

namespace stmg {

// Scalars of the elimination: T, or pairs (re, im).
template <typename T, bool C> struct PNum;
template <typename T> struct PNum<T, false> {
  using V = T;
  __device__ static V make(T re, T) { return re; }
  __device__ static T mag(V a) { return fabs(a); }
  __device__ static V inv(V a) { return (T)1 / a; }
  __device__ static V neg(V a) { return -a; }
  __device__ static V mul(V a, V b) { return a * b; }
  __device__ static V add(V a, V b) { return a + b; }
  __device__ static V fma(V acc, V a, V b) { return acc + a * b; }
  __device__ static V fms(V acc, V a, V b) { return acc - a * b; }
  __device__ static T re(V a) { return a; }
  __device__ static T im(V) { return (T)0; }
};
template <typename T> struct alignas(2 * sizeof(T)) PCx { T x, y; };
template <typename T> struct PNum<T, true> {
  using V = PCx<T>;
  __device__ static V make(T re, T im) { return {re, im}; }
  __device__ static T mag(V a) { return a.x * a.x + a.y * a.y; }
  __device__ static V inv(V a) { const T d = (T)1 / (a.x * a.x + a.y * a.y); return {a.x * d, -a.y * d}; }
  __device__ static V neg(V a) { return {-a.x, -a.y}; }
  __device__ static V add(V a, V b) { return {a.x + b.x, a.y + b.y}; }
  __device__ static V mul(V a, V b) { return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x}; }
  __device__ static V fma(V c, V a, V b) { return {c.x + a.x * b.x - a.y * b.y, c.y + a.x * b.y + a.y * b.x}; }
  __device__ static V fms(V c, V a, V b) { return {c.x - a.x * b.x + a.y * b.y, c.y - a.x * b.y - a.y * b.x}; }
  __device__ static T re(V a) { return a.x; }
  __device__ static T im(V a) { return a.y; }
};

// Search key of a candidate pivot: the leading bits of its magnitude, then the row (lower rows win).
// Zero for magnitudes that are not positive (zeros, NaN).  The nine low bits are the row's, so that a pivot may
// miss the largest candidate by a factor of 1 - 2^-14 in FP32 (of the squared magnitude for complex entries)
// and 1 - 2^-11 in FP64.  Searching by whole magnitudes takes another exchange of bits per step: the errors of
// rebuilt sweeps against 64 bits were the same to three digits, the rebuild 1 to 5 % slower.
__device__ __forceinline__ unsigned pivot_key(float a, int row) {
  return a > 0 ? ((__float_as_uint(a) & ~511u) | (unsigned)(511 - row)) : 0u;
}
__device__ __forceinline__ unsigned pivot_key(double a, int row) {
  return a > 0 ? (((unsigned)__double2hiint(a) & ~511u) | (unsigned)(511 - row)) : 0u;
}

__device__ __forceinline__ void team_sync(int id, int n) {
  if (n == 32) __syncwarp();
  else asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// Shared line of a row team: the pivot row in whole 16-byte chunks, search keys of two steps.
template <typename T, int PB>
struct alignas(16) TeamLine {
  T prow[2 * ((PB + 3) & ~3)];
  unsigned keys[2][16];
};

// nb exchange steps (columns p0, p0 + 1, ...) on the PB columns held in w, by the n threads (whole
// warps, barrier `id`) of a row team; thread `row` owns row `row` < 511 (valid: it exists).  pos: the
// step that used this row, or -1.  piv[p]: pivot rows.  On return w[k] holds column (k + nb) mod PB of
// the panel.  False (team-uniformly) on a zero pivot.
// The dependent chain of a step is search, reciprocal, pivot row, update: the next step's column is
// updated first and its search goes ahead of the other columns' multiply-adds.
template <typename T, bool C, int PB>
__device__ __forceinline__ bool exchange_panel(typename PNum<T, C>::V (&w)[PB], int row, bool valid, int& pos, int p0,
                                               int nb, TeamLine<T, PB>& sh, int* piv, int id, const int n) {
  using O = PNum<T, C>;
  using V = typename O::V;
  constexpr int VW = 16 / sizeof(V), NC = (PB + VW - 1) / VW;
  struct alignas(16) Chunk { V v[VW]; };
  Chunk* prow = reinterpret_cast<Chunk*>(sh.prow);
  const int warps = n >> 5, wid = row >> 5, lane = row & 31;
  unsigned best = __reduce_max_sync(0xffffffffu, valid && pos < 0 ? pivot_key(O::mag(w[0]), row) : 0u);
  if (warps > 1 && lane == 0) sh.keys[0][wid] = best;
#pragma unroll 1
  for (int s = 0; s < nb; ++s) {
    if (warps > 1) {
      team_sync(id, n);
      best = __reduce_max_sync(0xffffffffu, lane < warps ? sh.keys[s & 1][lane] : 0u);
    }
    if (best == 0u) return false;
    const int r = 511 - (int)(best & 511u);
    if (row == r) {
      pos = p0 + s;
      piv[p0 + s] = r;
      w[0] = O::inv(w[0]);                            // the reciprocal in the pivot's place
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        Chunk q;
#pragma unroll
        for (int x = 0; x < VW; ++x) q.v[x] = c * VW + x < PB ? w[c * VW + x < PB ? c * VW + x : 0] : V{};
        prow[c] = q;
      }
    }
    team_sync(id, n);
    // the pivot row's own update, row <- row / pivot, as 0 - (-1 / pivot) row
    if (row == r)
#pragma unroll
      for (int k = 1; k < PB; ++k) w[k] = V{};
    const Chunk q0 = prow[0];
    const V iv = q0.v[0];
    const V f = row == r ? O::neg(iv) : O::mul(w[0], iv);
    V p1;
    if constexpr (VW > 1) p1 = q0.v[1]; else p1 = prow[1].v[0];
    w[0] = O::fms(w[1], f, p1);
    best = __reduce_max_sync(0xffffffffu, valid && pos < 0 ? pivot_key(O::mag(w[0]), row) : 0u);
    if (warps > 1 && lane == 0) sh.keys[(s + 1) & 1][wid] = best;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const Chunk q = c == 0 ? q0 : prow[c];
#pragma unroll
      for (int x = 0; x < VW; ++x)
        if (c * VW + x >= 2 && c * VW + x < PB) w[c * VW + x - 1] = O::fms(w[c * VW + x], f, q.v[x]);
    }
    w[PB - 1] = O::neg(f);
    if (warps == 1) __syncwarp();                     // prow is rewritten in the next step
  }
  return true;
}

// Which sides of the cell a node lies on: bit 2 l + s, s = 0 low, 1 high side along axis l.
template <int D, int N>
__host__ __device__ constexpr int node_sides(int j) {
  int c = 0, s = 1;
  for (int l = 0; l < D; ++l) {
    const int x = (j / s) % N;
    if (x == 0) c |= 1 << (2 * l);
    if (x == N - 1) c |= 2 << (2 * l);
    s *= N;
  }
  return c;
}

// Assembly of patch entries: two nodes share the neighbours across the sides they both lie on (and
// combinations of them); a neighbour's element matrix holds the pair at a fixed offset from its
// place in the cell's own matrix.  rowlen: entries per matrix row, entries: per cell.
template <int D, int N>
struct SideSteps {
  int64_t d[2 * D];
  int exist;                                          // sides with a neighbour cell
  __device__ SideSteps(const int* cc, int n, int rowlen, int64_t entries) {
    exist = 0;
    int64_t cs = 1;
    int ns = 1;
#pragma unroll
    for (int l = 0; l < D; ++l) {
      const int64_t shift = (int64_t)(N - 1) * ns * (rowlen + 1);
      d[2 * l] = -cs * entries + shift;
      d[2 * l + 1] = cs * entries - shift;
      if (cc[l] > 0) exist |= 1 << (2 * l);
      if (cc[l] < n - 1) exist |= 2 << (2 * l);
      cs *= n;
      ns *= N;
    }
  }
  // sum over the cells that share both nodes, `code` their common sides (existing neighbours only)
  template <typename T>
  __device__ __forceinline__ T sum(const T* e, int code) const {
    // predicated loads, so that the loads of several entries overlap
    int64_t s[D];
    bool h[D];
#pragma unroll
    for (int l = 0; l < D; ++l) {
      const int b = (code >> (2 * l)) & 3;
      h[l] = b != 0;
      s[l] = (b & 2) ? d[2 * l + 1] : d[2 * l];
    }
    T v[1 << D];
#pragma unroll
    for (int m = 0; m < (1 << D); ++m) {
      bool on = true;
      int64_t o = 0;
#pragma unroll
      for (int l = 0; l < D; ++l)
        if ((m >> l) & 1) { on = on && h[l]; o += s[l]; }
      v[m] = on ? e[o] : (T)0;
    }
    T acc = v[0];
#pragma unroll
    for (int m = 1; m < (1 << D); ++m) acc += v[m];
    return acc;
  }
};

// ---------------------------------------------------------------------------- small patches (2D)
template <int D, int N> __host__ __device__ constexpr int small_team() { return (patch_rows<D, N>() + 31) / 32 * 32; }
constexpr int kSmallCells = 4;                        // cells per block

template <typename T, int D, int N>
struct alignas(16) SmallShared {
  TeamLine<T, patch_rows<D, N>()> line;
  T mx[2];
  int piv[patch_rows<D, N>()];
};

template <typename T, int D, int N, bool C>
__device__ __forceinline__ bool patch_small_block(const VankaArgs<T>& V, const TEig<T>& te, int e, int64_t cell,
                                                  const int* cc, int i, int id, int kp1, SmallShared<T, D, N>& sh) {
  using O = PNum<T, C>;
  using E = typename O::V;
  constexpr int NL = Shape<D, N>::Q, MV = D * NL, MS = patch_rows<D, N>(), NPC = MS - MV, TEAM = small_team<D, N>();
  const LevelArgs<T>& L = V.L;
  const T lr = te.lre[e], li = te.lim[e];
  E w[MS];
  // row i of T_lam = [lam M + A, B^T; B, 0]
  if (i < MV) {
    const SideSteps<D, N> sa(cc, L.n, MV, (int64_t)MV * MV), sm(cc, L.n, NL, (int64_t)NL * NL);
    const int c = i / NL, ni = i - c * NL, side = node_sides<D, N>(ni) & sa.exist;
    const T* EA = V.EA + (cell - V.ebase) * (int64_t)MV * MV + (int64_t)i * MV;
    const T* EM = V.EM + (cell - V.ebase) * (int64_t)NL * NL + ni * NL;
    const T* EB = V.EB + (cell - V.ebase) * (int64_t)NPC * MV + i;
#pragma unroll
    for (int j = 0; j < NL; ++j) {
      const int code = side & node_sides<D, N>(j);
      const T m = sm.sum(EM + j, code);
#pragma unroll
      for (int b = 0; b < D; ++b) {
        T a = sa.sum(EA + b * NL + j, code);
        if (b == c) a += lr * m;
        w[b * NL + j] = O::make(a, b == c ? li * m : (T)0);
      }
    }
#pragma unroll
    for (int m = 0; m < NPC; ++m) w[MV + m] = O::make(EB[m * MV], (T)0);
  } else {
    const T* EB = V.EB + (cell - V.ebase) * (int64_t)NPC * MV + (i < MS ? i - MV : 0) * MV;
#pragma unroll
    for (int j = 0; j < MV; ++j) w[j] = O::make(i < MS ? EB[j] : (T)0, (T)0);
#pragma unroll
    for (int m = 0; m < NPC; ++m) w[MV + m] = O::make((T)0, (T)0);
  }
  int pos = -1;
  if (!exchange_panel<T, C, MS>(w, i, i < MS, pos, 0, MS, sh.line, sh.piv, id, TEAM)) {
    if (i == 0) *V.status = 1;
    return false;
  }
  // column piv[q] of the inverse, entry pos (see inv_stride for the layout)
  constexpr int W = C ? 2 : 1;
  const int st = inv_stride(MS, V.invh ? 2 : (int)sizeof(T));
  const int64_t base = (cell * kp1 + te.off[e]) * (int64_t)MS * st;
  const int at = i < MS ? pos : i;                    // threads MS .. st - 1 write the zero padding
  if (V.invh) {
    T mx = 0;
    if (i < MS)
#pragma unroll
      for (int q = 0; q < MS; ++q) mx = fmax(mx, fmax(fabs(O::re(w[q])), fabs(O::im(w[q]))));
    for (int off = 16; off > 0; off >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    if (TEAM > 32) {
      if ((i & 31) == 0) sh.mx[i >> 5] = mx;
      team_sync(id, TEAM);
      mx = fmax(sh.mx[0], sh.mx[1]);
    }
    // the scale is held in FP32: divide by exactly the value the apply multiplies by
    const float sc = mx > 0 ? (float)mx : 1.f;
    const T isc = (T)1 / (T)sc;
    if (i == 0) V.scale[cell * te.nblk + e] = sc;
    __half* inv = V.invh + base;
    if (at < st)
#pragma unroll
      for (int q = 0; q < MS; ++q) {
        const int64_t o = W * (int64_t)(sh.piv[q] * st + at);
        inv[o] = __float2half_rn(i < MS ? (float)(O::re(w[q]) * isc) : 0.f);
        if (C) inv[o + 1] = __float2half_rn(i < MS ? (float)(O::im(w[q]) * isc) : 0.f);
      }
  } else if (at < st) {
    E* inv = reinterpret_cast<E*>(V.inv + base);
#pragma unroll
    for (int q = 0; q < MS; ++q) inv[sh.piv[q] * st + at] = i < MS ? w[q] : O::make((T)0, (T)0);
  }
  team_sync(id, TEAM);                                // piv is rewritten by the next block
  return true;
}

// Teams of one or two warps, kSmallCells cells per block; bound by the dependent exchange steps
// (about 150 multiply-adds of a 38-row complex step between two barriers), which the resident teams
// hide in part.  2D 128^2 Q3/P2 DG(2), 16384 cells: 0.87 ms (shared-memory elimination with five block
// barriers per step: 3.1 ms together with the element matrices, now 0.09 ms).
template <typename T, int D, int N>
__global__ void __launch_bounds__(kSmallCells * small_team<D, N>())
k_patch_small(VankaArgs<T> V, const __grid_constant__ TEig<T> te, int kp1, int64_t c0, int64_t c1) {
  constexpr int TEAM = small_team<D, N>();
  __shared__ __align__(16) SmallShared<T, D, N> sh[kSmallCells];
  const int g = threadIdx.x / TEAM, i = threadIdx.x - g * TEAM;
  const int64_t cell = c0 + (int64_t)blockIdx.x * kSmallCells + g;
  if (cell >= c1) return;                             // whole teams; only team barriers below
  int cc[3] = {0, 0, 0};
  cell_coords<D>(cell, V.L.n, cc);
#pragma unroll 1
  for (int e = 0; e < te.nblk; ++e) {
    const bool ok = te.cplx[e] ? patch_small_block<T, D, N, true>(V, te, e, cell, cc, i, 1 + g, kp1, sh[g])
                               : patch_small_block<T, D, N, false>(V, te, e, cell, cc, i, 1 + g, kp1, sh[g]);
    if (!ok) return;
  }
}

// ---------------------------------------------------------------------------- large patches
// Panel width: 64 registers of a row either way.
template <typename T> __host__ __device__ constexpr int panel_cols() { return sizeof(T) == 4 ? 32 : 16; }
__host__ __device__ constexpr int patch_ld(int m) { return (m + 7) & ~7; }   // whole 16-byte chunks per row
// Shared memory of the panel (W, R, pivot row, tables) and of the matrix, complex entries of 2 es bytes.
__host__ __device__ constexpr size_t patch_panel_smem(int m, int nl, size_t es) {
  const size_t pb = es == 4 ? 32 : 16;
  return 2 * es * (2 * pb * patch_ld(m)) + (2 * es * pb + 128) + sizeof(int) * (2 * (size_t)patch_ld(m) + nl) + 64;
}
__host__ __device__ constexpr size_t patch_matrix_bytes(int m, size_t es) { return 2 * es * (size_t)m * patch_ld(m); }
__host__ __device__ constexpr bool patch_matrix_onchip(int m, int nl, size_t es) {
  return patch_panel_smem(m, nl, es) + patch_matrix_bytes(m, es) <= 227 * 1024;
}

template <typename T, int D, int N, bool C>
__device__ __forceinline__ bool patch_blocked_block(const VankaArgs<T>& V, const TEig<T>& te, int e, int64_t cell,
                                                    const int* cc, int kp1, void* Sv, unsigned char* sm) {
  using O = PNum<T, C>;
  using E = typename O::V;
  constexpr int NL = Shape<D, N>::Q, MV = D * NL, MS = patch_rows<D, N>(), NPC = MS - MV;
  constexpr int PB = panel_cols<T>(), LD = patch_ld(MS), VW = 16 / sizeof(E);
  struct alignas(16) Chunk { E v[VW]; };
  const LevelArgs<T>& L = V.L;
  E* S = reinterpret_cast<E*>(Sv);                    // [MS][LD]
  E* Wm = reinterpret_cast<E*>(sm);                   // [PB][LD]: W by columns
  E* Rm = Wm + PB * LD;                               // [PB][LD]: old pivot rows
  TeamLine<T, PB>& line = *reinterpret_cast<TeamLine<T, PB>*>(sm + 2 * sizeof(T) * 2 * PB * LD);
  static_assert(sizeof(TeamLine<T, PB>) == 2 * sizeof(T) * PB + 128, "patch_panel_smem");
  int* piv = reinterpret_cast<int*>(&line + 1);
  int* panel_of = piv + LD;                           // panel in which a row became a pivot row, or -1
  int* sides = panel_of + LD;                         // node_sides of every node, existing neighbours only
  int* flag = sides + NL;
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, wid = tid >> 5, nw = nt >> 5;
  const T lr = te.lre[e], li = te.lim[e];
  // ---- assembly, a warp per row
  const SideSteps<D, N> sa(cc, L.n, MV, (int64_t)MV * MV), smm(cc, L.n, NL, (int64_t)NL * NL);
  for (int j = tid; j < NL; j += nt) sides[j] = node_sides<D, N>(j) & sa.exist;
  for (int j = tid; j < LD; j += nt) panel_of[j] = -1;
  if (tid == 0) *flag = 0;
  __syncthreads();
  const T* EA0 = V.EA + (cell - V.ebase) * (int64_t)MV * MV;
  const T* EM0 = V.EM + (cell - V.ebase) * (int64_t)NL * NL;
  const T* EB0 = V.EB + (cell - V.ebase) * (int64_t)NPC * MV;
  for (int row = wid; row < MS; row += nw) {
    const int c = row / NL, ni = row - c * NL;
#pragma unroll
    for (int x = 0; x < (LD + 31) / 32; ++x) {
      const int col = lane + 32 * x;
      if (col >= LD) break;
      T re = 0, im = 0;
      if (row < MV && col < MV) {
        const int b = col / NL, j = col - b * NL, code = sides[ni] & sides[j];
        re = sa.sum(EA0 + (int64_t)row * MV + col, code);
        if (b == c) {
          const T m = smm.sum(EM0 + ni * NL + j, code);
          re += lr * m;
          im = li * m;
        }
      } else if (row < MV && col < MS) {
        re = EB0[(int64_t)(col - MV) * MV + row];
      } else if (row >= MV && col < MV) {
        re = EB0[(int64_t)(row - MV) * MV + col];
      }
      S[row * LD + col] = O::make(re, im);
    }
  }
  __syncthreads();
  // ---- panels
  constexpr int team = (MS + 31) / 32 * 32;           // row team: the first warps of the block
  int pos = -1;
#pragma unroll 1
  for (int p0 = 0, ip = 0; p0 < MS; p0 += PB, ++ip) {
    const int nb = MS - p0 < PB ? MS - p0 : PB;
    if (tid < team) {
      E w[PB];
      const bool valid = tid < MS;
      const Chunk* src = reinterpret_cast<const Chunk*>(S + (valid ? tid : 0) * LD + p0);
#pragma unroll
      for (int k = 0; k < PB; k += VW) {
        const bool in = p0 + k < LD;                  // chunks past the row end are zero columns
        const Chunk q = in ? src[k / VW] : Chunk{};
#pragma unroll
        for (int x = 0; x < VW; ++x) w[k + x] = valid && k + x < nb ? q.v[x] : O::make((T)0, (T)0);
      }
      const int was = pos;
      if (!exchange_panel<T, C, PB>(w, tid, valid, pos, p0, nb, line, piv, 1, team)) {
        if (tid == 0) *flag = 1;
      } else {
        if (pos != was) panel_of[tid] = ip;
        int q = nb;                                   // w[k] is column (k + nb) mod PB
#pragma unroll
        for (int k = 0; k < PB; ++k) {
          if (q >= PB) q -= PB;
          if (tid < LD) Wm[q * LD + tid] = w[k];
          ++q;
        }
      }
    }
    __syncthreads();
    if (*flag) {
      if (tid == 0) *V.status = 1;
      return false;
    }
#pragma unroll 4
    for (int t = tid; t < nb * (LD / VW); t += nt) {
      const int q = t / (LD / VW), x = t - q * (LD / VW);
      reinterpret_cast<Chunk*>(Rm + q * LD)[x] = reinterpret_cast<const Chunk*>(S + piv[p0 + q] * LD)[x];
    }
    __syncthreads();
    // update: tiles of 4 rows and two chunks (half a row apart), lanes along the row.  The panel's products are
    // summed from zero and added to the entry once: summed onto the entry, each of them is rounded at its
    // size.  The entries are loaded four products before the end, so that the last ones hide the latency (3D 16^3
    // Q3/P2 DG(1) FP32 rebuild: loaded first 19.3 ms, last 21.9, so 19.15; FP64 8^3 55.2 -> 56.5, the additions).
    // Error of a rebuilt level's sweep against 64 bits, onto the entry -> from zero: that case 5.0e-7 -> 4.4e-7, FP32
    // 4^3 5.8e-7 -> 3.2e-7, FP64 8^3 Q2/P1 7.9e-16 -> 6.2e-16 (one column at a time: 4.5e-7, 4.5e-7, 7.5e-16).
    constexpr int TC = LD / (2 * VW), TR = (MS + 3) / 4;
    for (int t = tid; t < TR * TC; t += nt) {
      const int i0 = t / TC * 4, l = t - t / TC * TC;
      const int j0 = l * VW, j1 = LD / 2 + l * VW;
      E acc[4][2][VW];
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int x = 0; x < VW; ++x) { acc[r][0][x] = E{}; acc[r][1][x] = E{}; }
      const auto product = [&](int q) {
        E wv[4];
        if constexpr (VW <= 4) {
#pragma unroll
          for (int r = 0; r < 4; r += VW) {
            const Chunk a = *reinterpret_cast<const Chunk*>(Wm + q * LD + i0 + r);
#pragma unroll
            for (int x = 0; x < VW; ++x) wv[r + x] = a.v[x];
          }
        }
        const Chunk a = *reinterpret_cast<const Chunk*>(Rm + q * LD + j0);
        const Chunk b = *reinterpret_cast<const Chunk*>(Rm + q * LD + j1);
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int x = 0; x < VW; ++x) {
            acc[r][0][x] = O::fma(acc[r][0][x], wv[r], a.v[x]);
            acc[r][1][x] = O::fma(acc[r][1][x], wv[r], b.v[x]);
          }
      };
      const int q1 = nb > 4 ? nb - 4 : 0;             // the entries are on their way during the last four
#pragma unroll 4
      for (int q = 0; q < q1; ++q) product(q);
      Chunk old[4][2];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int i = i0 + r;
        const bool keep = i < MS && panel_of[i] != ip;
        old[r][0] = keep ? *reinterpret_cast<const Chunk*>(S + i * LD + j0) : Chunk{};
        old[r][1] = keep ? *reinterpret_cast<const Chunk*>(S + i * LD + j1) : Chunk{};
      }
#pragma unroll 4
      for (int q = q1; q < nb; ++q) product(q);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int i = i0 + r;
        if (i >= MS) break;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int j = h ? j1 : j0;
          Chunk o;
          if (j >= p0 && j < p0 + PB) {               // the panel's own columns (chunks never straddle it)
#pragma unroll
            for (int x = 0; x < VW; ++x) o.v[x] = Wm[(j - p0 + x) * LD + i];
          } else {
#pragma unroll
            for (int x = 0; x < VW; ++x) o.v[x] = O::add(old[r][h].v[x], acc[r][h][x]);
          }
          *reinterpret_cast<Chunk*>(S + i * LD + j) = o;
        }
      }
    }
    __syncthreads();
  }
  // ---- write out: inv[j = piv[q]][i] = M[piv[i]][q], PB rows i at a time through shared memory
  const int st = inv_stride(MS, V.invh ? 2 : (int)sizeof(T));
  constexpr int W = C ? 2 : 1;
  const int64_t base = (cell * kp1 + te.off[e]) * (int64_t)MS * st;
  T isc = 1;
  if (V.invh) {
    T mx = 0;
    for (int t = tid; t < MS * LD; t += nt) {
      const int col = t % LD;
      if (col < MS) mx = fmax(mx, fmax(fabs(O::re(S[t])), fabs(O::im(S[t]))));
    }
    mx = block_absmax<T>(mx);
    const float sc = mx > 0 ? (float)mx : 1.f;
    isc = (T)1 / (T)sc;
    if (tid == 0) V.scale[cell * te.nblk + e] = sc;
  }
  E* Tt = Wm;                                         // [PB][LD + 1] <= the two panel buffers
  for (int i0 = 0; i0 < st; i0 += PB) {
    for (int r = wid; r < PB && i0 + r < MS; r += nw) {
      const E* src = S + piv[i0 + r] * LD;
#pragma unroll
      for (int x = 0; x < (MS + 31) / 32; ++x)
        if (lane + 32 * x < MS) Tt[r * (LD + 1) + lane + 32 * x] = src[lane + 32 * x];
    }
    __syncthreads();
#pragma unroll 4
    for (int t = tid; t < PB * MS; t += nt) {
      const int q = t / PB, r = t - q * PB, i = i0 + r;
      if (i < st) {
        const E v = i < MS ? Tt[r * (LD + 1) + q] : O::make((T)0, (T)0);
        const int64_t o = (int64_t)piv[q] * st + i;
        if (V.invh) {
          __half* inv = V.invh + base + W * o;
          inv[0] = __float2half_rn((float)(O::re(v) * isc));
          if (C) inv[1] = __float2half_rn((float)(O::im(v) * isc));
        } else {
          reinterpret_cast<E*>(V.inv + base)[o] = v;
        }
      }
    }
    __syncthreads();
  }
  return true;
}

// Rows of the largest patch that a 256-thread row team covers; larger ones take 512 threads.
template <int D, int N> __host__ __device__ constexpr int blocked_threads() { return patch_rows<D, N>() <= 256 ? 256 : 512; }

// Two blocks per SM (one block's panel steps overlap the other's update); blocks stride over the
// cells, so that a workspace slot per block is enough.  Bound by instruction issue: 1.7 M warp
// instructions for a complex m = 202 patch, 1.0 M of them the multiply-adds of the inversion.
// 3D 16^3 Q3/P2 DG(1), 4096 cells (m = 202, complex): 10.7 ms, against 78.5 ms column by column with
// the matrix in global memory; its three Q2/P1 levels (m = 85): 1.8 ms against 5.3 ms.
template <typename T, int D, int N, bool ONCHIP>
__global__ void __launch_bounds__(blocked_threads<D, N>(), blocked_threads<D, N>() == 256 ? 2 : 1)
k_patch_blocked(VankaArgs<T> V, const __grid_constant__ TEig<T> te, int kp1, int64_t c0, int64_t c1) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int MS = patch_rows<D, N>();
  void* S = ONCHIP ? (void*)(smem_raw + ((patch_panel_smem(MS, Shape<D, N>::Q, sizeof(T)) + 15) & ~(size_t)15))
                   : (void*)(V.work + (int64_t)blockIdx.x * V.wslot);
  for (int64_t cell = c0 + blockIdx.x; cell < c1; cell += gridDim.x) {
    int cc[3] = {0, 0, 0};
    cell_coords<D>(cell, V.L.n, cc);
#pragma unroll 1
    for (int e = 0; e < te.nblk; ++e) {
      const bool ok = te.cplx[e] ? patch_blocked_block<T, D, N, true>(V, te, e, cell, cc, kp1, S, smem_raw)
                                 : patch_blocked_block<T, D, N, false>(V, te, e, cell, cc, kp1, S, smem_raw);
      if (!ok) return;
    }
  }
}

}  // namespace stmg
