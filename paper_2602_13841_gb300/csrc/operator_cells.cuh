// Matrix-free slab operator kernels: Jacobian apply y = J_n(U) x, residual R_n(U; V_prev) and slab
// mass, in two launches: every cell's contribution to its own nodes (k_cells2d / k_cells3d), then
// one sum per node over the cells that share it (k_node_sum).
//
// Sec. 4.4 ("matrix-free application of the slab Jacobian"): for every temporal basis index a
// the state-dependent spatial operator is evaluated cell-wise by sum factorisation, and the
// temporal matrices mix the results densely:
//   Y_v^i = sum_a K_ia M_h V^a + w_i [nu A_h + H'(V^i) + N^c'(V^i) + N^{b,r}] V^i + w_i (B+G^p)^T P^i
//   Y_p^i = w_i (B + G^p) V^i
// The mixing is done at the quadrature points (values sum_b K_ib JxW v^b).  The residual uses
// the same data path with the nonlinear terms (Eq. InAlgNS): convective flux -v (x) v, body force
// w_i f(t_i), the jump term -phi_i(t_{n-1}^+) M_h v_{n-1} and the Nitsche data g.
//
// Layout.  A group of N^(D-1) threads serves one (cell, time node); all time nodes of a cell sit in
// one block, so the increments at the Gauss points and the cell's geometry are computed once and
// shared.  A thread owns a whole line of N points: a 1D pass (interpolation with B, collocation
// derivative Dc, their transposes) is N^2 multiply-adds on registers with table entries at
// compile-time indices, and between two passes the line's direction changes through shared
// memory (one write and one read per point, against N reads per point when a thread owns a point).
// Boundary cells add their Nitsche / boundary-convection faces in the same block, the group's
// threads then being the N^(D-1) face points.
//
// Scatter.  The nodal results go to a cell-wise buffer (CellBuf) laid out as lines along x, and
// k_node_sum adds the up to 2^D contributions of a node in a fixed order: deterministic, no
// atomics, no colouring, so one launch covers the whole mesh (small meshes: 2 launches in place of
// 2^D or, in 3D, 2^(D+1); and rhs - J x needs no pass of its own).  The buffer holds a ring of cell
// planes (slot = plane mod P), so meshes beyond its size run in chunks of planes, each chunk
// finding the previous chunk's last plane still in place.
//
// What bounds it: FP64 the FP64 pipe (2 multiply-adds per clock and SM; 83 % busy in the 3D 24^3 Q2/P1 DG(2)
// apply, 86 % in the 16^3 Q3/P2 DG(2) residual), FP32 shared-memory wavefronts (a third of them bank conflicts
// in 2D Q3/P2) and instruction issue.  A 3D boundary cell costs about three interior ones (FP64 residual, Q3/P2
// DG(2), per cell: 16^3 181 ns, 24^3 149, 40^3 135).  Measured against the colour-by-colour kernels this
// replaces (a zero fill, then a volume and a face launch per colour with one thread per point):
//   3D 64^3 Q2/P1 DG(2) FP64 apply 20.14 -> 12.64 ms    3D 37^3 Q3/P2 DG(1) FP32 apply 940 -> 279 us
//   3D 16^3 Q3/P2 DG(2) residual    3.00 -> 0.73 ms     2D 256^2 Q3/P2 DG(2) FP64 apply 1086 -> 870 us
//   2D 8^2 Q2/P1 DG(1) FP64 apply    133 -> 27 us
// and, 2D FP32, against one kernel with a thread per cell on a tile of 16 x 8 cells in shared memory:
//   256^2 Q3/P2 DG(2) 104 -> 51 us, Q2/P1 DG(1) 28.6 -> 22.7 us; 32^2 59 -> 8.8 us and 14.5 -> 8.0 us
//   (Q2/P1 DG(0) is the exception: 8.1 -> 7.6 us at 64^2, 8.5 -> 7.9 at 128^2, 13.8 -> 12.8 at 224^2 and level
//   from 320^2 on, but 8.4 -> 8.9 at 160^2, 9.05 -> 9.9 at 192^2 and 14.3 -> 14.9 at 256^2)
#pragma once
#include <type_traits>

#include "chain.cuh"
#include "common.cuh"

namespace stmg {

// 2D FP32 calls of one time node release their successor late (see chain.cuh): their grids are short, so that
// both the gap to the next launch and the blocks that an early successor displaces count.
template <typename T, int D> __host__ __device__ constexpr bool chain_late(int kp1) { return D == 2 && sizeof(T) == 4 && kp1 == 1; }

enum { MJ = 0, MR = 1, MM = 2 };   // Jacobian apply, residual, mass (w_a M_h, w_a M_p)

template <typename T>
struct OpArgs {
  LevelArgs<T> L;
  const T* x;        // operand (J: increment; R: the iterate U)
  const T* state;    // J: the Newton state U (velocity part read); R: unused
  const T* vprev;    // R: V_{n-1}
  T* y;              // output
  int64_t xs, ys;    // batch strides (blockIdx.y selects the column of a batched apply)
  const T* geo;      // 2D FP64: per cell [5][Q] inverse Jacobian G[0][0], G[0][1], G[1][0], G[1][1] and
                     // JxW at the quadrature points (precomputed at set-up)
  const T* fgeo;     // 2D FP64: per boundary face (axis, side, position) [6][N] G n (2), n (2), JxW_f, 1 / h
  int64_t ss;        // batch stride of the state (0: one state shared by the batch)
  const T* nub;      // per-batch-column viscosity (device, blockIdx.y), or null: L.nu
};

// Viscosity of the batch column of this block.
template <typename T>
__device__ __forceinline__ T column_nu(const OpArgs<T>& A) { return A.nub ? A.nub[blockIdx.y] : A.L.nu; }

// Cell-wise results: entry (component ac = a D + c, cell plane z, [cy, k,] j, cx, i) at
//   column * col + ac * comp + (z mod P) * plane + line * (n N) + cx N + i,
// line = cy N + j within a plane of the last axis (3D: (cy N + k) N + j; 2D: j).
template <typename T>
struct CellBuf {
  T* s;
  int P;                 // cell planes held
  int64_t plane, comp, col;
};

template <int D, int N> __host__ __device__ constexpr int npress() {
  return D == 2 ? N * (N - 1) / 2 : (N - 1) * N * (N + 1) / 6;
}
// Pressure mode m of P_{N-2}: degree along axis l (total degree, then ascending degree of the last
// coordinate, of the one before it).
template <int D> constexpr int mode_deg(int m, int l) {
  int s = 0, cnt = 0;
  while (m >= cnt + (D == 2 ? s + 1 : (s + 1) * (s + 2) / 2)) { cnt += D == 2 ? s + 1 : (s + 1) * (s + 2) / 2; ++s; }
  int y = m - cnt, z = 0;
  if (D == 3)
    while (y >= s - z + 1) { y -= s - z + 1; ++z; }
  return l == 0 ? s - y - z : (l == 1 ? y : z);
}
template <int D, int M> struct Mode {
  static constexpr int x = mode_deg<D>(M, 0), y = mode_deg<D>(M, 1), z = mode_deg<D>(M, 2);
  __device__ static constexpr int deg(int l) { return l == 0 ? x : (l == 1 ? y : z); }
};

// f(integral_constant<int, 0>), ..., f(integral_constant<int, M - 1>): the index is a constant
// expression in the body (mode degrees, so that they cost nothing at run time).
template <int M, int I = 0, typename F>
__device__ __forceinline__ void static_for(F&& f) {
  if constexpr (I < M) {
    f(std::integral_constant<int, I>{});
    static_for<M, I + 1>(f);
  }
}

// v <- M v (or M^T v) for a line of N values in registers.
template <typename T, int N, bool TR>
__device__ __forceinline__ void line_mul(const T (&M)[MAXN][MAXN], T (&v)[N]) {
  T o[N];
#pragma unroll
  for (int q = 0; q < N; ++q) {
    T acc = (TR ? M[0][q] : M[q][0]) * v[0];
#pragma unroll
    for (int j = 1; j < N; ++j) acc += (TR ? M[j][q] : M[q][j]) * v[j];
    o[q] = acc;
  }
#pragma unroll
  for (int q = 0; q < N; ++q) v[q] = o[q];
}

// The interpolation B (and its transpose) and the collocation derivative Dc on a line.  Nodes and
// Gauss points are symmetric, so B commutes with the reflection of the line and Dc changes sign under
// it: for odd N the even and odd parts go through half-size tables, and the middle Gauss point of an
// odd rule is a node, so interpolation there is a copy.  6 and 7 operations instead of 9 for N = 3,
// 18 and 20 instead of 25 for N = 5; for N = 4 the split needs the same 16, so the plain product stays.
template <typename T, int N, bool TR>
__device__ __forceinline__ void line_B(const Tab<T>& tb, T (&v)[N]) {
  if constexpr (N % 2 == 0) {
    line_mul<T, N, TR>(tb.B, v);
  } else {
    constexpr int H = N / 2;
    T e[H], o[H], r[N];
#pragma unroll
    for (int j = 0; j < H; ++j) { e[j] = v[j] + v[N - 1 - j]; o[j] = v[j] - v[N - 1 - j]; }
    r[H] = v[H];
#pragma unroll
    for (int q = 0; q < H; ++q) {
      T s = TR ? tb.Be[0][q] * e[0] : tb.Bm[q] * v[H];
#pragma unroll
      for (int j = TR ? 1 : 0; j < H; ++j) s += (TR ? tb.Be[j][q] : tb.Be[q][j]) * e[j];
      T d = s;
#pragma unroll
      for (int j = 0; j < H; ++j) {
        const T c = TR ? tb.Bo[j][q] : tb.Bo[q][j];
        s += c * o[j];
        d -= c * o[j];
      }
      r[q] = s;
      r[N - 1 - q] = d;
      if (TR) r[H] += tb.Bm[q] * e[q];
    }
#pragma unroll
    for (int q = 0; q < N; ++q) v[q] = r[q];
  }
}
template <typename T, int N, bool TR>
__device__ __forceinline__ void line_D(const Tab<T>& tb, T (&v)[N]) {
  if constexpr (N % 2 == 0) {
    line_mul<T, N, TR>(tb.Dc, v);
  } else {
    constexpr int H = N / 2;
    T e[H], o[H], r[N];
#pragma unroll
    for (int j = 0; j < H; ++j) { e[j] = v[j] + v[N - 1 - j]; o[j] = v[j] - v[N - 1 - j]; }
    T mid = (TR ? tb.Dm[0] : tb.Dh[0]) * o[0];
#pragma unroll
    for (int j = 1; j < H; ++j) mid += (TR ? tb.Dm[j] : tb.Dh[j]) * o[j];
    r[H] = mid;
#pragma unroll
    for (int q = 0; q < H; ++q) {
      // the part that keeps its sign under the reflection (s) and the one that changes it (d)
      T d = (TR ? tb.Dh[q] : tb.Dm[q]) * v[H];
#pragma unroll
      for (int j = 0; j < H; ++j) d += (TR ? tb.Do[j][q] : tb.De[q][j]) * e[j];
      T s = -d;
#pragma unroll
      for (int j = 0; j < H; ++j) {
        const T c = TR ? tb.De[j][q] : tb.Do[q][j];
        d += c * o[j];
        s += c * o[j];
      }
      r[q] = d;
      r[N - 1 - q] = s;
    }
#pragma unroll
    for (int q = 0; q < N; ++q) v[q] = r[q];
  }
}

// Lines of a [..][N] shared array: N entries at `stride`; unit-stride lines of four floats are one
// 16-byte access (the arrays are 16-byte aligned with rows of four).
template <typename T, int N>
__device__ __forceinline__ void line_ld(const T* s, int stride, T (&v)[N]) {
#pragma unroll
  for (int i = 0; i < N; ++i) v[i] = s[i * stride];
}
template <typename T, int N>
__device__ __forceinline__ void line_st(T* s, int stride, const T (&v)[N]) {
#pragma unroll
  for (int i = 0; i < N; ++i) s[i * stride] = v[i];
}
template <typename T, int N>
__device__ __forceinline__ void row_ld(const T* s, T (&v)[N]) {
  if constexpr (N == 4 && sizeof(T) == 4) {
    const float4 f = *reinterpret_cast<const float4*>(s);
    v[0] = f.x; v[1] = f.y; v[2] = f.z; v[3] = f.w;
  } else {
    line_ld<T, N>(s, 1, v);
  }
}
template <typename T, int N>
__device__ __forceinline__ void row_st(T* s, const T (&v)[N]) {
  if constexpr (N == 4 && sizeof(T) == 4) {
    *reinterpret_cast<float4*>(s) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
    line_st<T, N>(s, 1, v);
  }
}

// Sizes of the shared buffers, in entries.  3D: planes of N = 4 lines are padded to 20 entries, so
// that the lines along y of a warp's threads fall into different banks.
template <int N> __host__ __device__ constexpr int plane3() { return N == 4 ? 20 : N * N; }
template <int N> __host__ __device__ constexpr int arr3() { return plane3<N>() * N; }
__host__ __device__ constexpr int even4(int e) { return (e + 3) & ~3; }
// Smallest stride >= e that is `want` mod 32: neighbouring groups of a warp, `stride` entries apart, then
// use different banks for their lines along every axis (with a stride of a multiple of 32 the lines of
// 2D Q2/P1 collided: 256^2 Q2/P1 DG(2) FP32 apply 88 us instead of 35).
__host__ __device__ constexpr int bank_stride(int e, int want) {
  while (e % 32 != want) ++e;
  return e;
}
// One group's part of the 3D buffers: three arrays of values (B0), two times three of derivatives /
// fluxes (B1, B2), pressure modes, a reduction line.
template <int N> __host__ __device__ constexpr int group3() {
  return bank_stride(9 * arr3<N>() + MAXNP + N * N, N == 3 ? 27 : (N == 4 ? 16 : 13));
}
// 2D: values, derivatives / fluxes, a reduction line, face arrays, pressure modes.
template <int N> __host__ __device__ constexpr int group2() {
  return bank_stride(4 * N * N + 13 * N + MAXNP, N == 3 ? 9 : (N == 4 ? 20 : 25));
}

template <typename T, int N, int MODE>
__host__ __device__ inline size_t cells3d_smem(int cpb, int kp1) {
  constexpr int QP = arr3<N>(), Q = N * N * N;
  const size_t cell = even4(10 * Q + 24 + (MODE == MR ? 3 * QP : 0));  // geometry, map, V_{n-1}
  return sizeof(T) * ((size_t)cpb * kp1 * group3<N>() + (size_t)cpb * cell + 2 * MAXN * MAXN + MAXN * 4 + 2 * MAXN);
}
template <typename T, int N>
__host__ __device__ inline size_t cells2d_smem(int cpb, int kp1) {
  return sizeof(T) * ((size_t)cpb * kp1 * group2<N>() + 2 * MAXN * MAXN + MAXN * 4 + 2 * MAXN);
}

template <typename T>
__device__ __forceinline__ T rcp_t(T v) { return (T)1 / v; }
template <>
__device__ __forceinline__ float rcp_t<float>(float v) { return __fdividef(1.0f, v); }

// Small lookup tables indexed by a thread's own point: copied to shared memory, since constant-bank
// reads serialise over different addresses.
template <typename T>
struct LaneTab {
  T (*B)[MAXN];
  T (*Dc)[MAXN];
  T (*P1)[4];
  T *qx, *qw;
};
template <typename T>
__device__ __forceinline__ LaneTab<T> stage_lane_tab(const Tab<T>& tb, T* s) {
  LaneTab<T> t;
  t.B = reinterpret_cast<T(*)[MAXN]>(s);
  t.Dc = reinterpret_cast<T(*)[MAXN]>(s + MAXN * MAXN);
  t.P1 = reinterpret_cast<T(*)[4]>(s + 2 * MAXN * MAXN);
  t.qx = s + 2 * MAXN * MAXN + MAXN * 4;
  t.qw = t.qx + MAXN;
  for (int e = threadIdx.x; e < MAXN * MAXN; e += blockDim.x) {
    t.B[e / MAXN][e % MAXN] = tb.B[e / MAXN][e % MAXN];
    t.Dc[e / MAXN][e % MAXN] = tb.Dc[e / MAXN][e % MAXN];
  }
  for (int e = threadIdx.x; e < MAXN * 4; e += blockDim.x) t.P1[e / 4][e % 4] = tb.P1[e / 4][e % 4];
  for (int e = threadIdx.x; e < MAXN; e += blockDim.x) { t.qx[e] = tb.qx[e]; t.qw[e] = tb.qw[e]; }
  return t;
}

// ---------------------------------------------------------------------------- 3D
// Trilinear map x_i = m[i][0] + m[i][1] X + m[i][2] Y + m[i][3] Z + m[i][4] XY + m[i][5] XZ + m[i][6] YZ
// + m[i][7] XYZ: its Jacobian at a reference point.
template <typename T>
__device__ __forceinline__ void map3_jacobian(const T* m, T X, T Y, T Z, T (&J)[3][3]) {
  const T yz = Y * Z, xz = X * Z, xy = X * Y;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const T* c = m + 8 * i;
    J[i][0] = c[1] + c[4] * Y + c[5] * Z + c[7] * yz;
    J[i][1] = c[2] + c[4] * X + c[6] * Z + c[7] * xz;
    J[i][2] = c[3] + c[5] * X + c[6] * Y + c[7] * xy;
  }
}
template <typename T>
__device__ __forceinline__ T map3_point(const T* m, int i, T X, T Y, T Z) {
  const T* c = m + 8 * i;
  return c[0] + c[1] * X + c[2] * Y + c[3] * Z + c[4] * (X * Y) + c[5] * (X * Z) + c[6] * (Y * Z) + c[7] * (X * Y * Z);
}

// One boundary face (normal axis AX, side) of the cells of a block that have it (Nitsche and
// boundary-convection terms: Eq. def-a-gam-tp, def-b-gam, bttp; Appendix A).  Thread (u, v) is
// node and Gauss point (u, v) of the face, u along the lower tangential axis.  At a face point
// (weight JxW_f):
//   J: a_c = w_a[-nu d_n dv_c + nu g1/h dv_c + g2/h (dv.n) n_c + dp n_c
//               + (y+ - 2y-) dv_c + (3 - sgn y)/2 (dv.n) v_c],  b_c = -w_a nu dv_c,  s = w_a dv.n
//   R: a_c = w_a[-nu d_n v_c + nu g1/h e_c + g2/h (e.n) n_c + p n_c + (y+ - 2y-) v_c + (g.n)- g_c],
//      b_c = -w_a nu e_c,  s = w_a e.n,  e = v - g
// with y = v.n, tested as  a_c z_c + b_c d_n z_c  and  s q.  h = |K| / |F| * hscale.
// W: 18 planar arrays of the group, red: N^2 entries, out: the group's nodal result (3 arrays,
// plane3 layout), pp: this thread's part of the pressure integrals.  Block-uniform calls.
template <typename T, int N, int MODE, int AX>
__device__ __forceinline__ void face3d(const OpArgs<T>& A, const Tab<T>& tb, const LaneTab<T>& lt, bool has, int side,
                                       const int (&cc)[3], int64_t cell, int a, int u, int v, const T* map,
                                       const T* pm, T vol, T nu, T* W, T* red, T* out, T (&pp)[npress<3, N>()]) {
  constexpr int NN = N * N, NPC = npress<3, N>(), PL = plane3<N>();
  constexpr int T1 = AX == 0 ? 1 : 0, T2 = AX == 2 ? 1 : 2;
  constexpr bool RES = MODE == MR;
  const LevelArgs<T>& L = A.L;
  const int p = u + N * v, e = side * (N - 1);
  T* W2 = W + 9 * NN;
  T nrm[3] = {0, 0, 0}, G[3][3], jf = 0, xf[3];
  if (has) {
    const int64_t n1 = L.N1, sx[3] = {1, n1, n1 * n1};
    const int64_t base = (int64_t)cc[0] * (N - 1) + n1 * ((int64_t)cc[1] * (N - 1) + n1 * ((int64_t)cc[2] * (N - 1))) +
                         u * sx[T1] + v * sx[T2] + (int64_t)a * L.Nv;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const T* src = A.x + base + c * L.nnodes;
      T ve = 0, vd = 0;
#pragma unroll
      for (int m = 0; m < N; ++m) {
        const T t = src[m * sx[AX]];
        vd += tb.Dend[side][m] * t;
        if (m == e) ve = t;
      }
      W[c * NN + p] = ve;
      W[(3 + c) * NN + p] = vd;
      if (!RES) W[(6 + c) * NN + p] = A.state[base + c * L.nnodes + e * sx[AX]];
    }
    const T q1 = lt.qx[u], q2 = lt.qx[v], sd = (T)side;
    const T X = AX == 0 ? sd : q1, Y = AX == 0 ? q1 : (AX == 1 ? sd : q2), Z = AX == 2 ? sd : q2;
    T J[3][3];
    map3_jacobian<T>(map, X, Y, Z, J);
    const T det = invert<T, 3>(J, G);
    const T nh = side ? (T)1 : (T)-1;
    T len2 = 0;
#pragma unroll
    for (int i = 0; i < 3; ++i) { nrm[i] = det * G[AX][i] * nh; len2 += nrm[i] * nrm[i]; }
    const T dS = sqrt(len2), is = (T)1 / dS;
#pragma unroll
    for (int i = 0; i < 3; ++i) nrm[i] *= is;
    jf = dS * (lt.qw[u] * lt.qw[v]);
    red[p] = jf;
    if (RES)
#pragma unroll
      for (int i = 0; i < 3; ++i) xf[i] = map3_point<T>(map, i, X, Y, Z);
  }
  __syncthreads();
  constexpr int NA = RES ? 6 : 9;
  T f[NA], area = 0;
  if (has) {
#pragma unroll
    for (int k = 0; k < NA; ++k) {
      T acc = 0;
#pragma unroll
      for (int i = 0; i < N; ++i) acc += lt.B[u][i] * W[k * NN + i + N * v];
      W2[k * NN + p] = acc;
    }
    for (int i = 0; i < NN; ++i) area += red[i];
  }
  __syncthreads();
  if (has) {
#pragma unroll
    for (int k = 0; k < NA; ++k) {
      T acc = 0;
#pragma unroll
      for (int i = 0; i < N; ++i) acc += lt.B[v][i] * W2[k * NN + u + N * i];
      f[k] = acc;
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) W[c * NN + p] = f[c];
  }
  __syncthreads();
  T ac[3], bn[3];
  if (has) {
    T gr[3][3];                                       // reference gradient [c][axis]
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      T d1 = 0, d2 = 0;
#pragma unroll
      for (int i = 0; i < N; ++i) {
        d1 += lt.Dc[u][i] * W[c * NN + i + N * v];
        d2 += lt.Dc[v][i] * W[c * NN + u + N * i];
      }
      gr[c][AX] = f[3 + c];
      gr[c][T1] = d1;
      gr[c][T2] = d2;
    }
    T fp = 0;
    static_for<NPC>([&](auto m) {
      fp += tb.Pend[side][Mode<3, decltype(m)::value>::deg(AX)] * lt.P1[u][Mode<3, decltype(m)::value>::deg(T1)] * lt.P1[v][Mode<3, decltype(m)::value>::deg(T2)] * pm[decltype(m)::value];
    });
    const T rh = area / (vol * L.hscale);             // 1 / h_{Gamma_D}
    T ghat[3], dn[3];
#pragma unroll
    for (int m = 0; m < 3; ++m) ghat[m] = G[m][0] * nrm[0] + G[m][1] * nrm[1] + G[m][2] * nrm[2];
#pragma unroll
    for (int c = 0; c < 3; ++c) dn[c] = gr[c][0] * ghat[0] + gr[c][1] * ghat[1] + gr[c][2] * ghat[2];
    T y = 0;
    T fs[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) { fs[c] = RES ? f[c] : f[(RES ? 0 : 6) + c]; y += fs[c] * nrm[c]; }
    const T ypos = (T)0.5 * (fabs(y) + y), yneg = (T)0.5 * (fabs(y) - y);
    const T sgn = (y > 0) ? (T)1 : ((y < 0) ? (T)-1 : (T)0);
    T ev[3], gd[3] = {0, 0, 0};
    if (RES) {
      double xd[3] = {(double)xf[0], (double)xf[1], (double)xf[2]}, gv[3];
      const double ta = (double)L.t0 + 0.5 * (double)L.tau * ((double)tb.that[a] + 1.0);
      if (L.problem == kProblemUser) {
        const int64_t nf = (int64_t)L.n * L.n, fi = face_index<3>(cc, AX, L.n);
        for (int c = 0; c < 3; ++c) gv[c] = L.gtab[(((((int64_t)a * 3 + AX) * 2 + side) * nf + fi) * 3 + c) * NN + p];
      } else {
        problem_g<3>(L.problem, xd, ta, (double)L.nu, gv);
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) { gd[c] = (T)gv[c]; ev[c] = f[c] - gd[c]; }
    } else {
#pragma unroll
      for (int c = 0; c < 3; ++c) ev[c] = f[c];
    }
    const T en = ev[0] * nrm[0] + ev[1] * nrm[1] + ev[2] * nrm[2];
    const T gn = gd[0] * nrm[0] + gd[1] * nrm[1] + gd[2] * nrm[2];
    const T wJ = tb.w[a] * jf;
    const T p1 = nu * L.gamma1 * rh, p2 = L.gamma2 * rh;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      T t = -nu * dn[c] + p1 * ev[c] + p2 * en * nrm[c] + fp * nrm[c];
      if (L.bconv) {
        if (RES) t += (ypos - 2 * yneg) * f[c] + (T)0.5 * (fabs(gn) - gn) * gd[c];
        else t += (ypos - 2 * yneg) * f[c] + (T)0.5 * ((T)3 - sgn) * en * fs[c];
      }
      ac[c] = wJ * t;
      const T bc = -wJ * nu * ev[c];
      bn[c] = bc * ghat[AX];
      W2[c * NN + p] = bc * ghat[T1];
      W2[(3 + c) * NN + p] = bc * ghat[T2];
    }
    const T sp = wJ * en;
    static_for<NPC>([&](auto m) {
      pp[decltype(m)::value] += tb.Pend[side][Mode<3, decltype(m)::value>::deg(AX)] * lt.P1[u][Mode<3, decltype(m)::value>::deg(T1)] * lt.P1[v][Mode<3, decltype(m)::value>::deg(T2)] * sp;
    });
  }
  __syncthreads();
  if (has) {
    // tangential gradients of the test function: transposed collocation derivatives
#pragma unroll
    for (int c = 0; c < 3; ++c) {
#pragma unroll
      for (int i = 0; i < N; ++i)
        ac[c] += lt.Dc[i][u] * W2[c * NN + i + N * v] + lt.Dc[i][v] * W2[(3 + c) * NN + u + N * i];
      W[c * NN + p] = ac[c];
      W[(3 + c) * NN + p] = bn[c];
    }
  }
  __syncthreads();
  if (has) {
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      T acc = 0;
#pragma unroll
      for (int i = 0; i < N; ++i) acc += lt.B[i][u] * W[k * NN + i + N * v];
      W2[k * NN + p] = acc;
    }
  }
  __syncthreads();
  if (has) {
    constexpr int st[3] = {1, N, PL};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      T tA = 0, tB = 0;
#pragma unroll
      for (int i = 0; i < N; ++i) {
        tA += lt.B[i][v] * W2[c * NN + u + N * i];
        tB += lt.B[i][v] * W2[(3 + c) * NN + u + N * i];
      }
      T* o = out + c * arr3<N>() + u * st[T1] + v * st[T2];
#pragma unroll
      for (int m = 0; m < N; ++m) o[m * st[AX]] += (m == e ? tA : (T)0) + tb.Dend[side][m] * tB;
    }
  }
  __syncthreads();
}

template <typename T, int N, int MODE, int BT, int MINB>
__global__ void __launch_bounds__(BT, MINB) k_cells3d(OpArgs<T> A, const __grid_constant__ Tab<T> tb, CellBuf<T> cb,
                                                      int64_t c0, int64_t c1, int cpb, const T* rhs) {
  chain_begin();
  constexpr bool RES = MODE == MR, MASS = MODE == MM, JAC = MODE == MJ;
  constexpr int NN = N * N, Q = N * NN, PL = plane3<N>(), QP = arr3<N>(), NPC = npress<3, N>();
  constexpr int GS = group3<N>();
  constexpr int CS = even4(10 * Q + 24 + (RES ? 3 * QP : 0));
  const LevelArgs<T>& L = A.L;
  const int kp1 = tb.k + 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* sm = reinterpret_cast<T*>(smem_raw);
  const int g = threadIdx.x / NN, p = threadIdx.x - g * NN;
  const int u = p % N, v = p / N;
  const bool in = g < cpb * kp1;                      // threads beyond the block's groups only join barriers
  const int gc = in ? g : 0;
  const int lc = gc / kp1, a = gc - lc * kp1;
  T* B0 = sm + (size_t)gc * GS;
  T* B1 = B0 + 3 * QP;
  T* B2 = B1 + 3 * QP;
  T* s_pm = B2 + 3 * QP;
  T* s_red = s_pm + MAXNP;
  T* cellm = sm + (size_t)cpb * kp1 * GS + (size_t)lc * CS;
  T* s_geo = cellm;                                   // [10][Q]: G, JxW at Gauss point u + N v + NN j = (u, j, v)
  T* s_map = cellm + 10 * Q;
  T* s_vp = s_map + 24;                               // [3][QP] V_{n-1} (residual)
  const LaneTab<T> lt = stage_lane_tab<T>(tb, sm + (size_t)cpb * kp1 * GS + (size_t)cpb * CS);
  A.x += blockIdx.y * A.xs;
  A.y += blockIdx.y * A.ys;
  if (A.state) A.state += blockIdx.y * A.ss;
  if (rhs) rhs += blockIdx.y * A.ys;
  const T nu = column_nu(A);
  const int64_t cell = c0 + (int64_t)blockIdx.x * cpb + lc;
  const bool on = in && cell < c1;
  int cc[3] = {0, 0, 0};
  if (on) {
    unsigned t = (unsigned)cell, n = (unsigned)L.n;   // n^3 <= 2^31 / 3 (vertex count of the handle)
    cc[0] = (int)(t % n); t /= n;
    cc[1] = (int)(t % n);
    cc[2] = (int)(t / n);
  }
  const int64_t n1 = L.N1;
  const int64_t nbase = (int64_t)cc[0] * (N - 1) + n1 * ((int64_t)cc[1] * (N - 1) + n1 * ((int64_t)cc[2] * (N - 1)));
  const int64_t poff = (int64_t)kp1 * L.Nv;
  const T wa = tb.w[a];

  // ---- nodal lines along z: load and interpolate; the map's coefficients; the pressure modes
  if (on) {
    const int64_t zb = nbase + u + n1 * v, n2 = n1 * n1;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      T w[N];
      const T* src = A.x + (int64_t)a * L.Nv + c * L.nnodes + zb;
#pragma unroll
      for (int k = 0; k < N; ++k) w[k] = src[k * n2];
      line_B<T, N, false>(tb, w);
      line_st<T, N>(B0 + c * QP + u + N * v, PL, w);
      if (JAC) {
        const T* st = A.state + (int64_t)a * L.Nv + c * L.nnodes + zb;
#pragma unroll
        for (int k = 0; k < N; ++k) w[k] = st[k * n2];
        line_B<T, N, false>(tb, w);
        line_st<T, N>(B1 + c * QP + u + N * v, PL, w);
      }
      if (RES && c % kp1 == a) {                      // V_{n-1}: one component per time node's group
        const T* st = A.vprev + c * L.nnodes + zb;
#pragma unroll
        for (int k = 0; k < N; ++k) w[k] = st[k * n2];
        line_B<T, N, false>(tb, w);
        line_st<T, N>(s_vp + c * QP + u + N * v, PL, w);
      }
    }
    for (int m = p; m < NPC; m += NN) s_pm[m] = A.x[poff + (int64_t)a * L.Np + cell * NPC + m];
    if (a == 0 && p < 3) {
      const int64_t m1 = L.n + 1, v0 = cc[0] + m1 * (cc[1] + m1 * (int64_t)cc[2]);
      T q[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) q[k] = L.verts[(v0 + (k & 1) + m1 * ((k >> 1) & 1) + m1 * m1 * (k >> 2)) * 3 + p];
      T* m = s_map + 8 * p;
      m[0] = q[0]; m[1] = q[1] - q[0]; m[2] = q[2] - q[0]; m[3] = q[4] - q[0];
      m[4] = (q[3] - q[2]) - (q[1] - q[0]);
      m[5] = (q[5] - q[4]) - (q[1] - q[0]);
      m[6] = (q[6] - q[4]) - (q[2] - q[0]);
      m[7] = ((q[7] - q[6]) - (q[5] - q[4])) - ((q[3] - q[2]) - (q[1] - q[0]));
    }
  }
  __syncthreads();
  // ---- lines along x; the geometry at the Gauss points (the time nodes' groups take turns)
  if (on) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      T w[N];
      T* s = B0 + c * QP + N * u + PL * v;
      row_ld<T, N>(s, w);
      line_B<T, N, false>(tb, w);
      row_st<T, N>(s, w);
      if (JAC) {
        s = B1 + c * QP + N * u + PL * v;
        row_ld<T, N>(s, w);
        line_B<T, N, false>(tb, w);
        row_st<T, N>(s, w);
      }
      if (RES && c % kp1 == a) {
        s = s_vp + c * QP + N * u + PL * v;
        row_ld<T, N>(s, w);
        line_B<T, N, false>(tb, w);
        row_st<T, N>(s, w);
      }
    }
#pragma unroll
    for (int j = 0; j < N; ++j)
      if (j % kp1 == a) {
        T J[3][3], G[3][3];
        map3_jacobian<T>(s_map, lt.qx[u], tb.qx[j], lt.qx[v], J);
        const T det = invert<T, 3>(J, G);
        T* o = s_geo + p + NN * j;
#pragma unroll
        for (int m = 0; m < 3; ++m)
#pragma unroll
          for (int l = 0; l < 3; ++l) o[(3 * m + l) * Q] = G[m][l];
        o[9 * Q] = det * (lt.qw[u] * tb.qw[j] * lt.qw[v]);
      }
  }
  __syncthreads();
  // ---- lines along y, kept in registers from here: values at the Gauss points (u, 0..N-1, v)
  const int yl = u + PL * v;                          // first entry of this thread's line along y
  T xq[3][N], sq[3][N];
  if (on) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      line_ld<T, N>(B0 + c * QP + yl, N, xq[c]);
      line_B<T, N, false>(tb, xq[c]);
      line_st<T, N>(B0 + c * QP + yl, N, xq[c]);
      if (JAC) {
        line_ld<T, N>(B1 + c * QP + yl, N, sq[c]);
        line_B<T, N, false>(tb, sq[c]);
      }
      if (RES && c % kp1 == a) {
        T w[N];
        line_ld<T, N>(s_vp + c * QP + yl, N, w);
        line_B<T, N, false>(tb, w);
        line_st<T, N>(s_vp + c * QP + yl, N, w);
      }
    }
  }
  __syncthreads();
  // pressure along the line: p(u, j, v) = sum_my P_my(j) cy[my]
  T cy[N - 1], ty[N - 1];
#pragma unroll
  for (int m = 0; m < N - 1; ++m) { cy[m] = 0; ty[m] = 0; }
  T z[3][N];
  if (on) {
    static_for<NPC>([&](auto m) {
      cy[Mode<3, decltype(m)::value>::deg(1)] += lt.P1[u][Mode<3, decltype(m)::value>::deg(0)] * lt.P1[v][Mode<3, decltype(m)::value>::deg(2)] * s_pm[decltype(m)::value];
    });
    if (MASS) {
#pragma unroll
      for (int j = 0; j < N; ++j) {
        const T w = wa * s_geo[9 * Q + p + NN * j];
#pragma unroll
        for (int c = 0; c < 3; ++c) z[c][j] = w * xq[c][j];
        T pq = 0;
#pragma unroll
        for (int m = 0; m < N - 1; ++m) pq += tb.P1[j][m] * cy[m];
#pragma unroll
        for (int m = 0; m < N - 1; ++m) ty[m] += tb.P1[j][m] * (w * pq);
      }
    } else {
      // time mixing of the values: all time nodes of the cell are in this block
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int j = 0; j < N; ++j) z[c][j] = 0;
      for (int b = 0; b < kp1; ++b) {
        const T kab = tb.K[a][b];
        const T* s = B0 + (b - a) * GS + yl;
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
          for (int j = 0; j < N; ++j) z[c][j] += kab * s[c * QP + N * j];
      }
      if (RES) {
        const T ca = tb.C[a];
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
          for (int j = 0; j < N; ++j) z[c][j] -= ca * s_vp[c * QP + yl + N * j];
      }
      // reference derivatives along x and z (own lines in those directions)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        T w[N];
        row_ld<T, N>(B0 + c * QP + N * u + PL * v, w);
        line_D<T, N, false>(tb, w);
        row_st<T, N>(B1 + c * QP + N * u + PL * v, w);
        line_ld<T, N>(B0 + c * QP + u + N * v, PL, w);
        line_D<T, N, false>(tb, w);
        line_st<T, N>(B2 + c * QP + u + N * v, PL, w);
      }
    }
  }
  if (!MASS) {
    __syncthreads();
    // ---- pointwise fluxes; along x and z they go back in place of the derivatives
    if (on) {
      double st = 0, ct = 0;
      if (RES && L.problem == kProblemMms3d) sincos((double)L.t0 + 0.5 * (double)L.tau * ((double)tb.that[a] + 1.0), &st, &ct);
      T fy[3][N];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
#pragma unroll
        for (int j = 0; j < N; ++j) fy[c][j] = xq[c][j];
        line_D<T, N, false>(tb, fy[c]);
      }
#pragma unroll
      for (int j = 0; j < N; ++j) {
        const T* gg = s_geo + p + NN * j;
        T G[3][3];
#pragma unroll
        for (int m = 0; m < 3; ++m)
#pragma unroll
          for (int l = 0; l < 3; ++l) G[m][l] = gg[(3 * m + l) * Q];
        const T jw = gg[9 * Q];
        T gp[3][3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const T gx = B1[c * QP + yl + N * j], gy = fy[c][j], gz = B2[c * QP + yl + N * j];
#pragma unroll
          for (int l = 0; l < 3; ++l) gp[c][l] = G[0][l] * gx + G[1][l] * gy + G[2][l] * gz;
        }
        T pq = 0;
#pragma unroll
        for (int m = 0; m < N - 1; ++m) pq += tb.P1[j][m] * cy[m];
        const T wj = wa * jw;
        T F[3][3];
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
          for (int l = c; l < 3; ++l) {
            const T cv = RES ? xq[c][j] * xq[l][j] : xq[c][j] * sq[l][j] + sq[c][j] * xq[l][j];
            F[c][l] = nu * gp[c][l] - cv;
            if (l != c) F[l][c] = nu * gp[l][c] - cv;
            else F[c][c] -= pq;
          }
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
          for (int l = 0; l < 3; ++l) F[c][l] *= wj;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          B1[c * QP + yl + N * j] = G[0][0] * F[c][0] + G[0][1] * F[c][1] + G[0][2] * F[c][2];
          fy[c][j] = G[1][0] * F[c][0] + G[1][1] * F[c][1] + G[1][2] * F[c][2];
          B2[c * QP + yl + N * j] = G[2][0] * F[c][0] + G[2][1] * F[c][1] + G[2][2] * F[c][2];
        }
        if (RES) {
          T fq[3] = {0, 0, 0};
          if (L.problem == kProblemUser) {
            const int64_t nc = (int64_t)L.n * L.n * L.n;
            for (int c = 0; c < 3; ++c) fq[c] = (T)L.ftab[(((int64_t)a * nc + cell) * 3 + c) * Q + u + N * j + NN * v];
          } else if (L.problem == kProblemMms3d) {
            const T X = lt.qx[u], Y = tb.qx[j], Z = lt.qx[v];
            double xd[3], fd[3];
            for (int l = 0; l < 3; ++l) xd[l] = (double)map3_point<T>(s_map, l, X, Y, Z);
            problem_f<3>(L.problem, xd, st, ct, (double)L.nu, fd);
            for (int c = 0; c < 3; ++c) fq[c] = (T)fd[c];
          }
#pragma unroll
          for (int c = 0; c < 3; ++c) z[c][j] -= wa * fq[c];
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) z[c][j] *= jw;
        const T sp = -wj * (gp[0][0] + gp[1][1] + gp[2][2]);
#pragma unroll
        for (int m = 0; m < N - 1; ++m) ty[m] += tb.P1[j][m] * sp;
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        line_D<T, N, true>(tb, fy[c]);
#pragma unroll
        for (int j = 0; j < N; ++j) z[c][j] += fy[c][j];
      }
    }
    __syncthreads();
    // ---- gradient test functions along x and z
    if (on) {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        T w[N];
        T* s = B1 + c * QP + N * u + PL * v;
        row_ld<T, N>(s, w);
        line_D<T, N, true>(tb, w);
        row_st<T, N>(s, w);
        s = B2 + c * QP + u + N * v;
        line_ld<T, N>(s, PL, w);
        line_D<T, N, true>(tb, w);
        line_st<T, N>(s, PL, w);
      }
    }
    __syncthreads();
    if (on) {
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int j = 0; j < N; ++j) z[c][j] += B1[c * QP + yl + N * j] + B2[c * QP + yl + N * j];
    }
  }
  // ---- quadrature -> nodes: transposed interpolation along y, x, z
  T* S = B0;                                          // last read (by the mixing) before the barriers above
  if (on) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      line_B<T, N, true>(tb, z[c]);
      line_st<T, N>(S + c * QP + yl, N, z[c]);
    }
  }
  __syncthreads();
  if (on) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      T w[N];
      T* s = S + c * QP + N * u + PL * v;
      row_ld<T, N>(s, w);
      line_B<T, N, true>(tb, w);
      row_st<T, N>(s, w);
    }
  }
  __syncthreads();
  if (on) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      line_ld<T, N>(S + c * QP + u + N * v, PL, z[c]);
      line_B<T, N, true>(tb, z[c]);
    }
  }
  T pp[NPC];
  static_for<NPC>([&](auto m) {
    pp[decltype(m)::value] = on ? lt.P1[u][Mode<3, decltype(m)::value>::deg(0)] * lt.P1[v][Mode<3, decltype(m)::value>::deg(2)] * ty[Mode<3, decltype(m)::value>::deg(1)] : (T)0;
  });
  // ---- boundary faces of the block's boundary cells
  if (!MASS) {
    const bool bnd = on && (cc[0] == 0 || cc[1] == 0 || cc[2] == 0 || cc[0] == L.n - 1 || cc[1] == L.n - 1 || cc[2] == L.n - 1);
    if (__syncthreads_or(bnd)) {
      T vol = 0;
      if (on) {
#pragma unroll
        for (int c = 0; c < 3; ++c) line_st<T, N>(S + c * QP + u + N * v, PL, z[c]);
        for (int j = 0; j < N; ++j) vol += s_geo[9 * Q + p + NN * j];
        s_red[p] = vol;
      }
      __syncthreads();
      if (bnd) {
        vol = 0;
        for (int i = 0; i < NN; ++i) vol += s_red[i];
      }
      __syncthreads();
      T* W = B1;
#pragma unroll 1
      for (int side = 0; side < 2; ++side) {
        const int edge = side ? L.n - 1 : 0;
        bool has = on && cc[0] == edge;
        if (__syncthreads_or(has))
          face3d<T, N, MODE, 0>(A, tb, lt, has, side, cc, cell, a, u, v, s_map, s_pm, vol, nu, W, s_red, S, pp);
        has = on && cc[1] == edge;
        if (__syncthreads_or(has))
          face3d<T, N, MODE, 1>(A, tb, lt, has, side, cc, cell, a, u, v, s_map, s_pm, vol, nu, W, s_red, S, pp);
        has = on && cc[2] == edge;
        if (__syncthreads_or(has))
          face3d<T, N, MODE, 2>(A, tb, lt, has, side, cc, cell, a, u, v, s_map, s_pm, vol, nu, W, s_red, S, pp);
      }
      if (on)
#pragma unroll
        for (int c = 0; c < 3; ++c) line_ld<T, N>(S + c * QP + u + N * v, PL, z[c]);
    }
  }
  // ---- results: nodal lines to the cell buffer, the cell's pressure rows to y
  if (on) {
    const int64_t row = (int64_t)L.n * N;
    T* o = cb.s + blockIdx.y * cb.col + (int64_t)(cc[2] % cb.P) * cb.plane + (int64_t)cc[0] * N + u;
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int k = 0; k < N; ++k) o[(int64_t)(a * 3 + c) * cb.comp + (((int64_t)cc[1] * N + k) * N + v) * row] = z[c][k];
  }
  __syncthreads();
  T* R = B1;                                          // [NN][NPC] partial pressure integrals (B1, B2: 6 QP entries)
  if (on)
#pragma unroll
    for (int m = 0; m < NPC; ++m) R[p + NN * m] = pp[m];
  __syncthreads();
  if (on)
    for (int m = p; m < NPC; m += NN) {
      T acc = 0;
      for (int i = 0; i < NN; ++i) acc += R[i + NN * m];
      const int64_t gi = poff + (int64_t)a * L.Np + cell * NPC + m;
      A.y[gi] = rhs ? rhs[gi] - acc : acc;
    }
}

// ---------------------------------------------------------------------------- 2D
// One boundary face (axis, side) for the threads of the cells that have it: thread u is node and
// Gauss point u of the face.  W: 12 line arrays of the group, red: N entries, out: the group's nodal
// result (2 arrays [j][i]).  Same integrand as face3d.
// Geometry of a 2D boundary face (axis AX, side) at its point q: G n, n, length element, det J there.
template <typename T, int AX>
__device__ __forceinline__ void face_geometry2d(const T (&mp)[2][4], int side, T q, T (&ghat)[2], T (&nrm)[2], T& dS) {
  const T X = AX == 0 ? (T)side : q, Y = AX == 0 ? q : (T)side;
  T J[3][3], G[3][3];
#pragma unroll
  for (int i = 0; i < 2; ++i) { J[i][0] = mp[i][1] + mp[i][3] * Y; J[i][1] = mp[i][2] + mp[i][3] * X; }
  const T det = invert<T, 2>(J, G), nh = side ? (T)1 : (T)-1;
  nrm[0] = det * G[AX][0] * nh;
  nrm[1] = det * G[AX][1] * nh;
  dS = sqrt(nrm[0] * nrm[0] + nrm[1] * nrm[1]);
  const T is = (T)1 / dS;
  nrm[0] *= is;
  nrm[1] *= is;
#pragma unroll
  for (int m = 0; m < 2; ++m) ghat[m] = G[m][0] * nrm[0] + G[m][1] * nrm[1];
}

template <typename T, int N, int MODE, int AX>
__device__ __forceinline__ void face2d(const OpArgs<T>& A, const Tab<T>& tb, const LaneTab<T>& lt, bool has, int side,
                                       const int (&cc)[3], int a, int u, const T (&mp)[2][4], const T* pm, T vol, T nu,
                                       T* W, T* red, T* out, T (&pp)[npress<2, N>()]) {
  constexpr int NPC = npress<2, N>(), TX = 1 - AX;
  constexpr bool RES = MODE == MR;
  const LevelArgs<T>& L = A.L;
  const int e = side * (N - 1);
  T* W2 = W + 6 * N;
  constexpr bool TABLE = sizeof(T) == 8;              // FP64: divisions and roots come from the face table
  T nrm[2] = {0, 0}, ghat[2] = {0, 0}, jf = 0, rht = 0, xf[2];
  if (has) {
    const int64_t n1 = L.N1, sx[2] = {1, n1};
    const int64_t base = (int64_t)cc[0] * (N - 1) + n1 * ((int64_t)cc[1] * (N - 1)) + u * sx[TX] + (int64_t)a * L.Nv;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const T* src = A.x + base + c * L.nnodes;
      T ve = 0, vd = 0;
#pragma unroll
      for (int m = 0; m < N; ++m) {
        const T t = src[m * sx[AX]];
        vd += tb.Dend[side][m] * t;
        if (m == e) ve = t;
      }
      W[c * N + u] = ve;
      W[(2 + c) * N + u] = vd;
      if (!RES) W[(4 + c) * N + u] = A.state[base + c * L.nnodes + e * sx[AX]];
    }
    if constexpr (TABLE) {
      const T* g = A.fgeo + ((int64_t)(2 * AX + side) * L.n + cc[TX]) * (6 * N) + u;
      ghat[0] = g[0]; ghat[1] = g[N]; nrm[0] = g[2 * N]; nrm[1] = g[3 * N]; jf = g[4 * N]; rht = g[5 * N];
    } else {
      T dS;
      face_geometry2d<T, AX>(mp, side, lt.qx[u], ghat, nrm, dS);
      jf = dS * lt.qw[u];
      red[u] = jf;
    }
    const T X = AX == 0 ? (T)side : lt.qx[u], Y = AX == 0 ? lt.qx[u] : (T)side;
    if (RES)
#pragma unroll
      for (int i = 0; i < 2; ++i) xf[i] = mp[i][0] + mp[i][1] * X + mp[i][2] * Y + mp[i][3] * (X * Y);
  }
  __syncthreads();
  if (has) {
    T fv[2], fdn[2], fdt[2], fs[2], area = 0;
#pragma unroll
    for (int c = 0; c < 2; ++c) { fv[c] = 0; fdn[c] = 0; fdt[c] = 0; fs[c] = 0; }
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const T b = lt.B[u][i], d = lt.Dc[u][i];        // lt.Dc holds D here (set by the caller)
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        fv[c] += b * W[c * N + i];
        fdt[c] += d * W[c * N + i];
        fdn[c] += b * W[(2 + c) * N + i];
        if (!RES) fs[c] += b * W[(4 + c) * N + i];
      }
      if (!TABLE) area += red[i];
    }
    if (RES) { fs[0] = fv[0]; fs[1] = fv[1]; }
    T fp = 0;
    static_for<NPC>([&](auto m) { fp += tb.Pend[side][Mode<2, decltype(m)::value>::deg(AX)] * lt.P1[u][Mode<2, decltype(m)::value>::deg(TX)] * pm[decltype(m)::value]; });
    const T rh = TABLE ? rht : area / (vol * L.hscale);   // 1 / h_{Gamma_D}
    T dn[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) dn[c] = fdn[c] * ghat[AX] + fdt[c] * ghat[TX];
    const T y = fs[0] * nrm[0] + fs[1] * nrm[1];
    const T ypos = (T)0.5 * (fabs(y) + y), yneg = (T)0.5 * (fabs(y) - y);
    const T sgn = (y > 0) ? (T)1 : ((y < 0) ? (T)-1 : (T)0);
    T ev[2], gd[2] = {0, 0};
    if (RES) {
      double xd[3] = {(double)xf[0], (double)xf[1], 0.0}, gv[3];
      const double ta = (double)L.t0 + 0.5 * (double)L.tau * ((double)tb.that[a] + 1.0);
      if (L.problem == kProblemUser) {
        const int64_t gb = ((((int64_t)a * 2 + AX) * 2 + side) * L.n + cc[TX]) * 2 * N + u;
        gv[0] = L.gtab[gb];
        gv[1] = L.gtab[gb + N];
      } else {
        problem_g<2>(L.problem, xd, ta, (double)L.nu, gv);
      }
      gd[0] = (T)gv[0]; gd[1] = (T)gv[1];
    }
    ev[0] = fv[0] - gd[0]; ev[1] = fv[1] - gd[1];
    const T en = ev[0] * nrm[0] + ev[1] * nrm[1];
    const T gn = gd[0] * nrm[0] + gd[1] * nrm[1];
    const T wJ = tb.w[a] * jf;
    const T p1 = nu * L.gamma1 * rh, p2 = L.gamma2 * rh;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      T t = -nu * dn[c] + p1 * ev[c] + p2 * en * nrm[c] + fp * nrm[c];
      if (L.bconv) {
        if (RES) t += (ypos - 2 * yneg) * fs[c] + (T)0.5 * (fabs(gn) - gn) * gd[c];
        else t += (ypos - 2 * yneg) * fv[c] + (T)0.5 * ((T)3 - sgn) * en * fs[c];
      }
      const T bc = -wJ * nu * ev[c];
      W2[c * N + u] = wJ * t;
      W2[(2 + c) * N + u] = bc * ghat[TX];
      W2[(4 + c) * N + u] = bc * ghat[AX];
    }
    const T sp = wJ * en;
    static_for<NPC>([&](auto m) { pp[decltype(m)::value] += tb.Pend[side][Mode<2, decltype(m)::value>::deg(AX)] * lt.P1[u][Mode<2, decltype(m)::value>::deg(TX)] * sp; });
  }
  __syncthreads();
  if (has) {
    constexpr int st[2] = {1, N};
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      T tA = 0, tB = 0;
#pragma unroll
      for (int i = 0; i < N; ++i) {
        tA += lt.B[i][u] * W2[c * N + i] + lt.Dc[i][u] * W2[(2 + c) * N + i];
        tB += lt.B[i][u] * W2[(4 + c) * N + i];
      }
      T* o = out + c * N * N + u * st[TX];
#pragma unroll
      for (int m = 0; m < N; ++m) o[m * st[AX]] += (m == e ? tA : (T)0) + tb.Dend[side][m] * tB;
    }
  }
  __syncthreads();
}

template <typename T, int N, int MODE, int BT, int MINB>
__global__ void __launch_bounds__(BT, MINB) k_cells2d(OpArgs<T> A, const __grid_constant__ Tab<T> tb, CellBuf<T> cb,
                                                      int64_t c0, int64_t c1, int cpb, const T* rhs) {
  chain_wait();
  const bool late = chain_late<T, 2>(tb.k + 1);
  if (!late) chain_release();
  constexpr bool RES = MODE == MR, MASS = MODE == MM, JAC = MODE == MJ;
  constexpr int Q = N * N, NPC = npress<2, N>();
  constexpr int GS = group2<N>();
  const LevelArgs<T>& L = A.L;
  const int kp1 = tb.k + 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* sm = reinterpret_cast<T*>(smem_raw);
  const int g = threadIdx.x / N, u = threadIdx.x - g * N;
  const bool in = g < cpb * kp1;
  const int gc = in ? g : 0;
  const int lc = gc / kp1, a = gc - lc * kp1;
  T* B0 = sm + (size_t)gc * GS;                       // [2][Q] values, then the integration passes
  T* B1 = B0 + 2 * Q;                                 // [2][Q] derivatives / fluxes along y
  T* s_red = B1 + 2 * Q;                              // [N]
  T* W = s_red + N;                                   // [12][N] face arrays
  T* s_pm = W + 12 * N;
  const LaneTab<T> lt = stage_lane_tab<T>(tb, sm + (size_t)cpb * kp1 * GS);
  A.x += blockIdx.y * A.xs;
  A.y += blockIdx.y * A.ys;
  if (A.state) A.state += blockIdx.y * A.ss;
  if (rhs) rhs += blockIdx.y * A.ys;
  const T nu = column_nu(A);
  const int64_t cell = c0 + (int64_t)blockIdx.x * cpb + lc;
  const bool on = in && cell < c1;
  int cc[3] = {0, 0, 0};
  if (on) { cc[0] = (int)((unsigned)cell % (unsigned)L.n); cc[1] = (int)((unsigned)cell / (unsigned)L.n); }
  const int64_t n1 = L.N1;
  const int64_t nbase = (int64_t)cc[0] * (N - 1) + n1 * ((int64_t)cc[1] * (N - 1));
  const int64_t poff = (int64_t)kp1 * L.Nv;
  const T wa = tb.w[a];
  // the bilinear map x_l = mp[l][0] + mp[l][1] X + mp[l][2] Y + mp[l][3] XY.  FP32 evaluates its Jacobian
  // at every point (a dozen operations against five loads of a table); FP64 reads the level's table,
  // since every operation on its pipe counts (and needs the map for the residual's boundary data only).
  constexpr bool TABLE = sizeof(T) == 8;
  const bool bnd = !MASS && on && (cc[0] == 0 || cc[1] == 0 || cc[0] == L.n - 1 || cc[1] == L.n - 1);
  T mp[2][4] = {{0, 1, 0, 0}, {0, 0, 1, 0}};
  if (TABLE ? bnd : on) {
    const int64_t v0 = (int64_t)cc[0] + (int64_t)(L.n + 1) * cc[1];
#pragma unroll
    for (int l = 0; l < 2; ++l) {
      const T q0 = L.verts[2 * v0 + l], q1 = L.verts[2 * v0 + 2 + l];
      const T q2 = L.verts[2 * (v0 + L.n + 1) + l], q3 = L.verts[2 * (v0 + L.n + 2) + l];
      mp[l][0] = q0; mp[l][1] = q1 - q0; mp[l][2] = q2 - q0; mp[l][3] = (q3 - q2) - (q1 - q0);
    }
  }
  // G (row-major) and JxW at the Gauss point (i, u)
  const T* geo = TABLE ? A.geo + cell * 5 * Q + N * u : nullptr;
  const auto geometry = [&](int i, T (&G)[4]) -> T {
    if constexpr (TABLE) {
#pragma unroll
      for (int x = 0; x < 4; ++x) G[x] = geo[x * Q + i];
      return geo[4 * Q + i];
    } else {
      const T X = tb.qx[i], Y = lt.qx[u];
      const T J00 = mp[0][1] + mp[0][3] * Y, J01 = mp[0][2] + mp[0][3] * X;
      const T J10 = mp[1][1] + mp[1][3] * Y, J11 = mp[1][2] + mp[1][3] * X;
      const T det = J00 * J11 - J01 * J10, id = rcp_t<T>(det);
      G[0] = J11 * id; G[1] = -J01 * id; G[2] = -J10 * id; G[3] = J00 * id;
      return det * (tb.qw[i] * lt.qw[u]);
    }
  };
  // ---- nodal lines along y
  if (on) {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      T w[N];
      const T* src = A.x + (int64_t)a * L.Nv + c * L.nnodes + nbase + u;
#pragma unroll
      for (int k = 0; k < N; ++k) w[k] = src[k * n1];
      line_B<T, N, false>(tb, w);
      line_st<T, N>(B0 + c * Q + u, N, w);
      if (!MASS && (JAC || a == 0)) {
        const T* st = (JAC ? A.state + (int64_t)a * L.Nv : A.vprev) + c * L.nnodes + nbase + u;
#pragma unroll
        for (int k = 0; k < N; ++k) w[k] = st[k * n1];
        line_B<T, N, false>(tb, w);
        line_st<T, N>(B1 + c * Q + u, N, w);
      }
    }
    for (int m = u; m < NPC; m += N) s_pm[m] = A.x[poff + (int64_t)a * L.Np + cell * NPC + m];
  }
  __syncthreads();
  // ---- lines along x, kept in registers: values at the Gauss points (0..N-1, u)
  T xq[2][N], sq[2][N], z[2][N], cx[N - 1], tx[N - 1];
#pragma unroll
  for (int m = 0; m < N - 1; ++m) { cx[m] = 0; tx[m] = 0; }
  if (on) {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      row_ld<T, N>(B0 + c * Q + N * u, xq[c]);
      line_B<T, N, false>(tb, xq[c]);
      row_st<T, N>(B0 + c * Q + N * u, xq[c]);
      if (JAC) {
        row_ld<T, N>(B1 + c * Q + N * u, sq[c]);
        line_B<T, N, false>(tb, sq[c]);
      } else if (RES) {
        // V_{n-1}: group 0 interpolated it along y; every time node takes it from there
        row_ld<T, N>(B0 - a * GS + 2 * Q + c * Q + N * u, sq[c]);
        line_B<T, N, false>(tb, sq[c]);
      }
    }
    static_for<NPC>([&](auto m) { cx[Mode<2, decltype(m)::value>::deg(0)] += lt.P1[u][Mode<2, decltype(m)::value>::deg(1)] * s_pm[decltype(m)::value]; });
  }
  __syncthreads();
  if (on) {
    if (MASS) {
#pragma unroll
      for (int i = 0; i < N; ++i) {
        T G[4];
        const T w = wa * geometry(i, G);
        z[0][i] = w * xq[0][i];
        z[1][i] = w * xq[1][i];
        T pq = 0;
#pragma unroll
        for (int m = 0; m < N - 1; ++m) pq += tb.P1[i][m] * cx[m];
#pragma unroll
        for (int m = 0; m < N - 1; ++m) tx[m] += tb.P1[i][m] * (w * pq);
      }
    } else {
#pragma unroll
      for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int i = 0; i < N; ++i) z[c][i] = RES ? -tb.C[a] * sq[c][i] : (T)0;
      if (kp1 == 1) {                                 // the thread's own line
        const T k00 = tb.K[0][0];
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
          for (int i = 0; i < N; ++i) z[c][i] += k00 * xq[c][i];
      } else {
        for (int b = 0; b < kp1; ++b) {
          const T kab = tb.K[a][b];
          const T* s = B0 + (b - a) * GS + N * u;
#pragma unroll
          for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int i = 0; i < N; ++i) z[c][i] += kab * s[c * Q + i];
        }
      }
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        T w[N];
        line_ld<T, N>(B0 + c * Q + u, N, w);
        line_D<T, N, false>(tb, w);
        line_st<T, N>(B1 + c * Q + u, N, w);
      }
    }
  }
  if (!MASS) {
    __syncthreads();
    if (on) {
      double st = 0, ct = 0;
      if (RES && L.problem == kProblemMms2d) sincos((double)L.t0 + 0.5 * (double)L.tau * ((double)tb.that[a] + 1.0), &st, &ct);
      T fx[2][N];
#pragma unroll
      for (int c = 0; c < 2; ++c) {
#pragma unroll
        for (int i = 0; i < N; ++i) fx[c][i] = xq[c][i];
        line_D<T, N, false>(tb, fx[c]);
      }
#pragma unroll
      for (int i = 0; i < N; ++i) {
        T G[4];
        const T jw = geometry(i, G), G00 = G[0], G01 = G[1], G10 = G[2], G11 = G[3];
        T gp[2][2];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const T gx = fx[c][i], gy = B1[c * Q + N * u + i];
          gp[c][0] = G00 * gx + G10 * gy;
          gp[c][1] = G01 * gx + G11 * gy;
        }
        T pq = 0;
#pragma unroll
        for (int m = 0; m < N - 1; ++m) pq += tb.P1[i][m] * cx[m];
        const T wj = wa * jw;
        const T x0 = xq[0][i], x1 = xq[1][i];
        const T s0 = RES ? x0 : sq[0][i], s1 = RES ? x1 : sq[1][i];
        const T c01 = RES ? x0 * x1 : x0 * s1 + s0 * x1;
        const T F00 = wj * (nu * gp[0][0] - (RES ? x0 * x0 : 2 * (x0 * s0)) - pq), F01 = wj * (nu * gp[0][1] - c01);
        const T F10 = wj * (nu * gp[1][0] - c01), F11 = wj * (nu * gp[1][1] - (RES ? x1 * x1 : 2 * (x1 * s1)) - pq);
        fx[0][i] = G00 * F00 + G01 * F01;
        fx[1][i] = G00 * F10 + G01 * F11;
        B1[N * u + i] = G10 * F00 + G11 * F01;
        B1[Q + N * u + i] = G10 * F10 + G11 * F11;
        if (RES) {
          T f0 = 0, f1 = 0;
          if (L.problem == kProblemUser) {
            const int64_t fb = (((int64_t)a * L.n * L.n + cell) * 2) * Q + N * u + i;
            f0 = (T)L.ftab[fb];
            f1 = (T)L.ftab[fb + Q];
          } else if (L.problem == kProblemMms2d) {
            const int64_t v0 = (int64_t)cc[0] + (int64_t)(L.n + 1) * cc[1];
            const T X = tb.qx[i], Y = lt.qx[u];
            double xd[3] = {0, 0, 0}, fd[3];
            for (int l = 0; l < 2; ++l)
              xd[l] = (double)(L.verts[2 * v0 + l] * ((1 - X) * (1 - Y)) + L.verts[2 * v0 + 2 + l] * (X * (1 - Y)) +
                               L.verts[2 * (v0 + L.n + 1) + l] * ((1 - X) * Y) + L.verts[2 * (v0 + L.n + 2) + l] * (X * Y));
            problem_f<2>(L.problem, xd, st, ct, (double)L.nu, fd);
            f0 = (T)fd[0];
            f1 = (T)fd[1];
          }
          z[0][i] -= wa * f0;
          z[1][i] -= wa * f1;
        }
        z[0][i] *= jw;
        z[1][i] *= jw;
        const T sp = -wj * (gp[0][0] + gp[1][1]);
#pragma unroll
        for (int m = 0; m < N - 1; ++m) tx[m] += tb.P1[i][m] * sp;
      }
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        line_D<T, N, true>(tb, fx[c]);
#pragma unroll
        for (int i = 0; i < N; ++i) z[c][i] += fx[c][i];
      }
    }
    __syncthreads();
    if (on) {
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        T w[N];
        line_ld<T, N>(B1 + c * Q + u, N, w);
        line_D<T, N, true>(tb, w);
        line_st<T, N>(B1 + c * Q + u, N, w);
      }
    }
    __syncthreads();
    if (on) {
#pragma unroll
      for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int i = 0; i < N; ++i) z[c][i] += B1[c * Q + N * u + i];
    }
  }
  // ---- quadrature -> nodes
  T* S = B0;
  if (on) {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      line_B<T, N, true>(tb, z[c]);
      row_st<T, N>(S + c * Q + N * u, z[c]);
    }
  }
  __syncthreads();
  if (on) {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      line_ld<T, N>(S + c * Q + u, N, z[c]);
      line_B<T, N, true>(tb, z[c]);
    }
  }
  T pp[NPC];
  static_for<NPC>([&](auto m) { pp[decltype(m)::value] = on ? lt.P1[u][Mode<2, decltype(m)::value>::deg(1)] * tx[Mode<2, decltype(m)::value>::deg(0)] : (T)0; });
  if (!MASS) {
    if (__syncthreads_or(bnd)) {
      T vol = 0;
      if (bnd) {
#pragma unroll
        for (int c = 0; c < 2; ++c) line_st<T, N>(S + c * Q + u, N, z[c]);
        // |K|: det J of the bilinear map at the centre
        vol = (mp[0][1] + (T)0.5 * mp[0][3]) * (mp[1][2] + (T)0.5 * mp[1][3]) -
              (mp[0][2] + (T)0.5 * mp[0][3]) * (mp[1][1] + (T)0.5 * mp[1][3]);
      }
      // D at the lane's own point replaces Dc in the lane table: the faces differentiate nodal values
      for (int e = threadIdx.x; e < MAXN * MAXN; e += blockDim.x) lt.Dc[e / MAXN][e % MAXN] = tb.D[e / MAXN][e % MAXN];
      __syncthreads();
#pragma unroll 1
      for (int side = 0; side < 2; ++side) {
        const int edge = side ? L.n - 1 : 0;
        bool has = on && cc[0] == edge;
        if (__syncthreads_or(has))
          face2d<T, N, MODE, 0>(A, tb, lt, has, side, cc, a, u, mp, s_pm, vol, nu, W, s_red, S, pp);
        has = on && cc[1] == edge;
        if (__syncthreads_or(has))
          face2d<T, N, MODE, 1>(A, tb, lt, has, side, cc, a, u, mp, s_pm, vol, nu, W, s_red, S, pp);
      }
      if (bnd)
#pragma unroll
        for (int c = 0; c < 2; ++c) line_ld<T, N>(S + c * Q + u, N, z[c]);
    }
  }
  if (late) chain_release();
  if (on) {
    const int64_t row = (int64_t)L.n * N;
    T* o = cb.s + blockIdx.y * cb.col + (int64_t)(cc[1] % cb.P) * cb.plane + (int64_t)cc[0] * N + u;
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int j = 0; j < N; ++j) o[(int64_t)(a * 2 + c) * cb.comp + j * row] = z[c][j];
  }
  __syncthreads();
  T* R = B0;                                          // [N][NPC] partial pressure integrals: N NPC <= 4 Q
  if (on)
#pragma unroll
    for (int m = 0; m < NPC; ++m) R[u + N * m] = pp[m];
  __syncthreads();
  if (on)
    for (int m = u; m < NPC; m += N) {
      T acc = 0;
#pragma unroll
      for (int i = 0; i < N; ++i) acc += R[i + N * m];
      const int64_t gi = poff + (int64_t)a * L.Np + cell * NPC + m;
      A.y[gi] = rhs ? rhs[gi] - acc : acc;
    }
}

// ---------------------------------------------------------------------------- node sums
// y (velocity part, node planes g0 .. g1-1 of the last axis) = src + alpha * the sum of the cells'
// contributions at each node (src null: zero; src may be y).  One thread per node, all components and
// time nodes; the cells of a node in ascending order.
template <typename T, int D, int N, int KP1>
__global__ void k_node_sum(CellBuf<T> cb, const T* src, T* y, T alpha, int n, int N1, int64_t nnodes, int64_t Nv,
                           int64_t ys, int g0, int64_t count) {
  chain_wait();
  constexpr bool late = chain_late<T, D>(KP1);
  if (!late) chain_release();
  y += blockIdx.y * ys;
  if (src) src += blockIdx.y * ys;
  const T* s = cb.s + blockIdx.y * cb.col;
  const int64_t row = (int64_t)n * N;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < count; t += (int64_t)gridDim.x * blockDim.x) {
    int gm[3];
    int64_t rem;
    if (count <= 0xffffffffll) { rem = (unsigned)t / (unsigned)N1; }
    else { rem = t / N1; }
    gm[0] = (int)(t - rem * N1);
    if (D == 3) { gm[2] = (int)((unsigned)rem / (unsigned)N1); gm[1] = (int)rem - gm[2] * N1; gm[2] += g0; }
    else { gm[1] = g0 + (int)rem; gm[2] = 0; }
    // per axis: offsets of the (one or two) cell lines that hold the node
    int64_t o0[3] = {0, 0, 0}, o1[3] = {0, 0, 0};
    bool two[3] = {false, false, false};
#pragma unroll
    for (int l = 0; l < D; ++l) {
      const int c = gm[l] / (N - 1), i = gm[l] - c * (N - 1);
      const auto at = [&](int cell, int loc) -> int64_t {
        if (l == 0) return (int64_t)cell * N + loc;
        if (l == D - 1) return (int64_t)(cell % cb.P) * cb.plane + (int64_t)loc * (D == 3 ? N : 1) * row;
        return ((int64_t)cell * N * N + loc) * row;
      };
      const bool low = i == 0 && c > 0;
      two[l] = low && c < n;
      o0[l] = low ? at(c - 1, N - 1) : at(c, i);
      o1[l] = two[l] ? at(c, 0) : 0;
    }
    const int64_t node = gm[0] + (int64_t)N1 * (gm[1] + (int64_t)N1 * gm[2]);
    T old[KP1 * D], v[KP1 * D];
#pragma unroll
    for (int ac = 0; ac < KP1 * D; ++ac) {
      old[ac] = src ? src[(int64_t)(ac / D) * Nv + (int64_t)(ac % D) * nnodes + node] : (T)0;
      const T* sc = s + (int64_t)ac * cb.comp;
      v[ac] = 0;
#pragma unroll
      for (int k2 = 0; k2 < (D == 3 ? 2 : 1); ++k2)
#pragma unroll
        for (int k1 = 0; k1 < 2; ++k1) {
          const bool on = !(k2 && !two[2]) && !(k1 && !two[1]);
          const T* q = sc + (k1 ? o1[1] : o0[1]) + (k2 ? o1[2] : o0[2]);
          v[ac] += on ? q[o0[0]] : (T)0;
          v[ac] += on && two[0] ? q[o1[0]] : (T)0;
        }
    }
#pragma unroll
    for (int ac = 0; ac < KP1 * D; ++ac)
      y[(int64_t)(ac / D) * Nv + (int64_t)(ac % D) * nnodes + node] = old[ac] + alpha * v[ac];
  }
  if (late) chain_release();
}

// Face table (FP64) of a 2D level, one thread per boundary face: see OpArgs::fgeo.  With it the longest
// chain of dependent FP64 operations of a boundary cell (two divisions, a root, a third division) is
// gone from every call: 2D 8^2 Q2/P1 DG(1) apply 34.8 -> 30.7 us.
template <typename T, int N>
__global__ void k_face_geo2d(LevelArgs<T> L, Tab<T> tb, T* __restrict__ fgeo) {
  const int f = blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= 4 * L.n) return;
  const int as = f / L.n, pos = f - as * L.n, axis = as >> 1, side = as & 1, edge = side ? L.n - 1 : 0;
  const int cx = axis == 0 ? edge : pos, cy = axis == 0 ? pos : edge;
  const int64_t v0 = (int64_t)cx + (int64_t)(L.n + 1) * cy;
  T mp[2][4];
  for (int l = 0; l < 2; ++l) {
    const T q0 = L.verts[2 * v0 + l], q1 = L.verts[2 * v0 + 2 + l];
    const T q2 = L.verts[2 * (v0 + L.n + 1) + l], q3 = L.verts[2 * (v0 + L.n + 2) + l];
    mp[l][0] = q0; mp[l][1] = q1 - q0; mp[l][2] = q2 - q0; mp[l][3] = (q3 - q2) - (q1 - q0);
  }
  const T vol = (mp[0][1] + (T)0.5 * mp[0][3]) * (mp[1][2] + (T)0.5 * mp[1][3]) -
                (mp[0][2] + (T)0.5 * mp[0][3]) * (mp[1][1] + (T)0.5 * mp[1][3]);
  T* g = fgeo + (int64_t)f * (6 * N);
  T area = 0;
  for (int p = 0; p < N; ++p) {
    T ghat[2], nrm[2], dS;
    if (axis == 0) face_geometry2d<T, 0>(mp, side, tb.qx[p], ghat, nrm, dS);
    else face_geometry2d<T, 1>(mp, side, tb.qx[p], ghat, nrm, dS);
    const T jf = dS * tb.qw[p];
    g[p] = ghat[0]; g[N + p] = ghat[1]; g[2 * N + p] = nrm[0]; g[3 * N + p] = nrm[1]; g[4 * N + p] = jf;
    area += jf;
  }
  for (int p = 0; p < N; ++p) g[5 * N + p] = area / (vol * L.hscale);
}

// Geometry table (FP64) of a 2D level: per cell and Gauss point t the inverse Jacobian G (dxhat_m/dx_l)
// and JxW of the multilinear map.
template <typename T, int N>
__global__ void k_geo2d(LevelArgs<T> L, Tab<T> tb, T* __restrict__ geo, int64_t ncells) {
  constexpr int Q = N * N;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < ncells * Q;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t cell = e / Q;
    const int t = (int)(e % Q), tx = t % N, ty = t / N;
    const int cx = (int)(cell % L.n), cy = (int)(cell / L.n);
    const int64_t v0 = (int64_t)cx + (int64_t)(L.n + 1) * cy;
    const int64_t vv[4] = {v0, v0 + 1, v0 + L.n + 1, v0 + L.n + 2};
    T corner[4][3];
    for (int q = 0; q < 4; ++q) {
      for (int i = 0; i < 2; ++i) corner[q][i] = L.verts[vv[q] * 2 + i];
      corner[q][2] = 0;
    }
    T xh[3] = {tb.qx[tx], tb.qx[ty], 0}, J[3][3], G[3][3], xq[3];
    map_jacobian<T, 2>(corner, xh, J, xq);
    const T JxW = invert<T, 2>(J, G) * tb.qw[tx] * tb.qw[ty];
    T* gg = geo + cell * 5 * Q + t;
    gg[0] = G[0][0]; gg[Q] = G[0][1]; gg[2 * Q] = G[1][0]; gg[3 * Q] = G[1][1]; gg[4 * Q] = JxW;
  }
}

}  // namespace stmg
