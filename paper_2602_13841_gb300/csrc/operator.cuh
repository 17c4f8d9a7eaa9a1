// Small helpers shared by the cell kernels: points per cell, node numbering, and the basis functions
// on a boundary face (values, reference gradients, pressure modes).
#pragma once
#include "common.cuh"

namespace stmg {

template <int D, int N>
struct Shape {
  static constexpr int Q = (D == 2) ? N * N : N * N * N;
  static constexpr int NF = (D == 2) ? N : N * N;    // points on one face
};

template <int D>
__device__ inline int64_t global_node(int N1, const int* cc, int r1, int t, int N) {
  int64_t g = 0, stride = 1;
  for (int l = 0; l < D; ++l) {
    int il = (l == 0) ? t % N : (l == 1 ? (t / N) % N : t / (N * N));
    g += (int64_t)(cc[l] * r1 + il) * stride;
    stride *= N1;
  }
  return g;
}

// Node j's basis function at face point pq of the face (axis, side): value and reference gradient.
template <typename T, int D, int N>
__device__ inline void face_weights(const Tab<T>& tb, int axis, int side, const int* pq, int j,
                                    T& val, T* grad) {
  int jm[3];
  jm[0] = j % N; jm[1] = (j / N) % N; jm[2] = (D == 3) ? j / (N * N) : 0;
  // tangential coordinates: dimensions other than `axis` in increasing order
  int qq[3] = {0, 0, 0};
  { int ti = 0; for (int l = 0; l < D; ++l) if (l != axis) qq[l] = pq[ti++]; }
  const bool onf = (jm[axis] == side * (N - 1));
  val = 1;
  for (int m = 0; m < D; ++m) grad[m] = 1;
  for (int l = 0; l < D; ++l) {
    T v = (l == axis) ? (onf ? (T)1 : (T)0) : tb.B[qq[l]][jm[l]];
    T dv = (l == axis) ? tb.Dend[side][jm[l]] : tb.D[qq[l]][jm[l]];
    val *= v;
    for (int m = 0; m < D; ++m) grad[m] *= (m == l) ? dv : v;
  }
}

template <typename T, int D, int N>
__device__ inline T face_psi(const Tab<T>& tb, int axis, int side, const int* pq, int mo) {
  int qq[3] = {0, 0, 0};
  { int ti = 0; for (int l = 0; l < D; ++l) if (l != axis) qq[l] = pq[ti++]; }
  T psi = 1;
  for (int l = 0; l < D; ++l)
    psi *= (l == axis) ? tb.Pend[side][tb.modes[mo][l]] : tb.P1[qq[l]][tb.modes[mo][l]];
  return psi;
}

}  // namespace stmg
