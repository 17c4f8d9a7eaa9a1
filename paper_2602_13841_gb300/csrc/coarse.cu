// Coarsest-level direct solve (Sec. 4.2, "solved directly").  The coarse Jacobian is assembled
// column by column by a batched matrix-free apply to the identity, bordered with one mean-zero
// pressure row and column per time node (pure Dirichlet: pressure in L^2_0), inverted once per
// smoother build by Gauss-Jordan elimination with partial pivoting in FP64, and applied in FP64
// with one step of iterative refinement against the bordered matrix.
#include "mg.hpp"
#include "op_launch.cuh"
#include "chain.cuh"
#include "counters.hpp"

namespace stmg {

// A (Nb x Nb, column-major) = [[J, C^T], [C, 0]] with C_a = (pressure part of M e_a), e_a the
// constant pressure at time node a.  J: N x N column-major.
__global__ void k_border_copy(const double* __restrict__ J, double* __restrict__ A, int N, int Nb) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < (int64_t)Nb * Nb;
       e += (int64_t)gridDim.x * blockDim.x) {
    int col = (int)(e / Nb), row = (int)(e % Nb);
    A[e] = (col < N && row < N) ? J[(int64_t)col * N + row] : 0.0;
  }
}

__global__ void k_const_pressure(double* __restrict__ e, int64_t poff, int64_t Np, int npc, int a, int N) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
    int64_t rel = i - poff - (int64_t)a * Np;
    e[i] = (rel >= 0 && rel < Np && rel % npc == 0) ? 1.0 : 0.0;
  }
}

__global__ void k_border_rows(const double* __restrict__ Me, double* __restrict__ A, int N, int Nb, int a) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
    A[(int64_t)(N + a) * Nb + i] = Me[i];     // column N+a, row i   (C^T)
    A[(int64_t)i * Nb + N + a] = Me[i];       // column i, row N+a   (C)
  }
}

cudaError_t coarse_border(const Level& lv, const Problem& pb, const double* J, double* A, int N, int Nb,
                          cudaStream_t s) {
  k_border_copy<<<152 * 4, 256, 0, s>>>(J, A, N, Nb);
  note_launch();
  // scratch: the two columns after J (caller allocates Nb*Nb + 2*N for J's buffer)
  double* e = const_cast<double*>(J) + (int64_t)N * N;
  double* Me = e + N;
  for (int a = 0; a <= lv.k; ++a) {
    k_const_pressure<<<64, 256, 0, s>>>(e, (int64_t)(lv.k + 1) * lv.Nv, lv.Np, lv.npc, a, N);
  note_launch();
    cudaError_t err = launch_operator<double>(lv, pb, OP_MASS, 0.0, e, nullptr, nullptr, Me, s);
    if (err != cudaSuccess) return err;
    k_border_rows<<<64, 256, 0, s>>>(Me, A, N, Nb, a);
  note_launch();
  }
  return cudaGetLastError();
}

__global__ void k_to_rowmajor(const double* __restrict__ A, double* __restrict__ S, int n) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < (int64_t)n * n;
       e += (int64_t)gridDim.x * blockDim.x) {
    int row = (int)(e / n), col = (int)(e % n);
    S[e] = A[(int64_t)col * n + row];
  }
}

// Inverse of the coarse matrix S (n x n row-major) by Gauss-Jordan exchange steps in panels of kPanel
// columns, without row interchanges (see vanka_patch.cuh for the form): k_gj_panel (one block) runs the
// steps of a panel on its n x kPanel columns, choosing each pivot among the rows not used yet, and
// leaves the exchange matrix W (by columns), a copy R of the pivot rows, the pivot rows' numbers and
// each row's panel; k_gj_update (all SMs) applies S_i <- [i not a pivot row] S_i + W_i R to the other
// columns; k_gj_permute writes the column-major inverse.  A zero pivot sets *status and turns the
// remaining launches into no-ops.
// Bound by FP64 (2 multiply-adds per clock and SM): a panel's steps cost n kPanel^2 of them on one SM,
// the updates n^2 kPanel over all, so narrow panels win until the launches show; one pass over S per
// panel instead of one per column.  n = 816 (3D Q2/P1 DG(1), 2^3 cells): 4.7 ms against 14.1 ms with a
// pivot and an elimination launch per column; n = 126 (2D): 0.37 ms against 1.0 ms in one block.
constexpr int kPanel = 8;

// key of a pivot candidate: leading bits of |a|, then the row in the bits of `low` (lower rows win).  A pivot may
// miss the largest candidate by a factor of 1 - 2^(b - 20), b the bits of the row numbers (n = 816: 2^-10).
__device__ __forceinline__ unsigned gj_key(double a, int row, unsigned low) {
  // integer comparisons: the FP64 pipe is what the panel steps wait for
  const unsigned hi = (unsigned)__double2hiint(a) & 0x7fffffffu, lo = (unsigned)__double2loint(a);
  const bool zero = (hi | lo) == 0u, nan = hi > 0x7ff00000u || (hi == 0x7ff00000u && lo != 0u);
  return zero || nan ? 0u : ((hi & ~low) | (low - (unsigned)row));
}

// Rows in registers: thread t of the block owns rows t, t + 1024, ... (ROWS of them).
template <int ROWS>
__global__ void __launch_bounds__(1024) k_gj_panel(const double* __restrict__ S, int n, int p0, double* __restrict__ W,
                                                   double* __restrict__ R, int* piv, int* pan, int* status,
                                                   unsigned low) {
  __shared__ double prow[kPanel];
  __shared__ unsigned keys[2][32];
  __shared__ int spiv[kPanel];
  if (*status) return;
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warps = nt >> 5;
  const int nb = n - p0 < kPanel ? n - p0 : kPanel;
  double w[ROWS][kPanel];
  bool open[ROWS];
#pragma unroll
  for (int x = 0; x < ROWS; ++x) {
    const int i = tid + x * nt;
    open[x] = i < n && pan[i] < 0;
#pragma unroll
    for (int k = 0; k < kPanel; ++k) w[x][k] = i < n && k < nb ? S[(int64_t)i * n + p0 + k] : 0.0;
  }
  // the columns rotate by one place per step: the current one is always w[.][0]
#pragma unroll 1
  for (int s = 0; s < nb; ++s) {
    unsigned best = 0u;
#pragma unroll
    for (int x = 0; x < ROWS; ++x)
      if (open[x]) best = max(best, gj_key(w[x][0], tid + x * nt, low));
    best = __reduce_max_sync(0xffffffffu, best);
    if (lane == 0) keys[s & 1][tid >> 5] = best;
    __syncthreads();
    best = __reduce_max_sync(0xffffffffu, lane < warps ? keys[s & 1][lane] : 0u);
    if (best == 0u) {
      if (tid == 0) *status = 1;
      return;
    }
    const int r = (int)(low - (best & low));
#pragma unroll
    for (int x = 0; x < ROWS; ++x)
      if (tid + x * nt == r) {
        open[x] = false;
        spiv[s] = r;
        prow[0] = 1.0 / w[x][0];                      // the reciprocal in the pivot's place
#pragma unroll
        for (int k = 1; k < kPanel; ++k) { prow[k] = w[x][k]; w[x][k] = 0.0; }
      }
    __syncthreads();
    const double iv = prow[0];
#pragma unroll
    for (int x = 0; x < ROWS; ++x) {
      const double f = tid + x * nt == r ? -iv : w[x][0] * iv;
#pragma unroll
      for (int k = 1; k < kPanel; ++k) w[x][k - 1] = w[x][k] - f * prow[k];
      w[x][kPanel - 1] = -f;
    }
  }
  __syncthreads();
#pragma unroll
  for (int x = 0; x < ROWS; ++x) {
    const int i = tid + x * nt;
    if (i >= n) continue;
#pragma unroll
    for (int k = 0; k < kPanel; ++k) W[(int64_t)((k + nb) % kPanel) * n + i] = w[x][k];
  }
  if (tid < nb) { piv[p0 + tid] = spiv[tid]; pan[spiv[tid]] = p0 / kPanel; }
  for (int t = tid; t < nb * n; t += nt) {
    const int k = t / n, j = t - k * n;
    R[t] = S[(int64_t)spiv[k] * n + j];
  }
}

// The same with the panel in global memory (W), for more rows than registers hold.
__global__ void __launch_bounds__(1024) k_gj_panel_global(const double* __restrict__ S, int n, int p0, double* W, double* R,
                                                          int* piv, int* pan, int* status, unsigned low) {
  __shared__ double prow[kPanel];
  __shared__ unsigned keys[32];
  if (*status) return;
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warps = nt >> 5;
  const int nb = n - p0 < kPanel ? n - p0 : kPanel;
  for (int64_t t = tid; t < (int64_t)n * kPanel; t += nt) {
    const int i = (int)(t / kPanel), k = (int)(t % kPanel);
    W[(int64_t)k * n + i] = k < nb ? S[(int64_t)i * n + p0 + k] : 0.0;
  }
  __syncthreads();
  for (int s = 0; s < nb; ++s) {
    unsigned best = 0u;
    for (int i = tid; i < n; i += nt)
      if (pan[i] < 0) best = max(best, gj_key(W[(int64_t)s * n + i], i, low));
    best = __reduce_max_sync(0xffffffffu, best);
    if (lane == 0) keys[tid >> 5] = best;
    __syncthreads();
    best = __reduce_max_sync(0xffffffffu, lane < warps ? keys[lane] : 0u);
    if (best == 0u) {
      if (tid == 0) *status = 1;
      return;
    }
    const int r = (int)(low - (best & low));
    if (tid < kPanel) {
      const double w = W[(int64_t)tid * n + r];
      prow[tid] = tid == s ? 1.0 / w : w;
    }
    __syncthreads();
    if (tid == 0) { piv[p0 + s] = r; pan[r] = p0 / kPanel; }
    const double iv = prow[s];
    for (int i = tid; i < n; i += nt) {
      const bool own = i == r;
      const double f = own ? -iv : W[(int64_t)s * n + i] * iv;
#pragma unroll
      for (int k = 0; k < kPanel; ++k) {
        const double w = own ? 0.0 : W[(int64_t)k * n + i];
        W[(int64_t)k * n + i] = k == s ? -f : w - f * prow[k];
      }
    }
    __syncthreads();
  }
  for (int64_t t = tid; t < (int64_t)nb * n; t += nt) {
    const int k = (int)(t / n), j = (int)(t - (int64_t)k * n);
    R[t] = S[(int64_t)piv[p0 + k] * n + j];
  }
}

constexpr int kGjTile = 32;
__global__ void __launch_bounds__(128) k_gj_update(double* __restrict__ S, int n, int p0, const double* __restrict__ W,
                                                   const double* __restrict__ R, const int* __restrict__ pan,
                                                   const int* status) {
  if (*status) return;
  __shared__ double sw[kPanel][kGjTile], sr[kPanel][kGjTile];
  const int nb = n - p0 < kPanel ? n - p0 : kPanel, ip = p0 / kPanel;
  const int i0 = blockIdx.y * kGjTile, j0 = blockIdx.x * kGjTile, tid = threadIdx.x;
  for (int t = tid; t < kPanel * kGjTile; t += 128) {
    const int k = t / kGjTile, x = t % kGjTile;
    sw[k][x] = k < nb && i0 + x < n ? W[(int64_t)k * n + i0 + x] : 0.0;
    sr[k][x] = k < nb && j0 + x < n ? R[(int64_t)k * n + j0 + x] : 0.0;
  }
  __syncthreads();
  const int jj = tid & 31, ib = tid >> 5, j = j0 + jj;
  if (j >= n) return;
  double r[kPanel];
#pragma unroll
  for (int k = 0; k < kPanel; ++k) r[k] = sr[k][jj];
  const bool in = j >= p0 && j < p0 + nb;             // the panel's own columns take W
#pragma unroll
  for (int x = 0; x < kGjTile / 4; ++x) {
    const int ii = ib + 4 * x, i = i0 + ii;
    if (i >= n) break;
    double acc;
    if (in) {
      acc = W[(int64_t)(j - p0) * n + i];
    } else {
      acc = pan[i] == ip ? 0.0 : S[(int64_t)i * n + j];
#pragma unroll
      for (int k = 0; k < kPanel; ++k) acc += sw[k][ii] * r[k];
    }
    S[(int64_t)i * n + j] = acc;
  }
}

// out (column-major): inverse[p][piv[q]] = S[piv[p]][q]
__global__ void k_gj_permute(const double* __restrict__ S, double* __restrict__ out, int n, const int* __restrict__ piv,
                             const int* status) {
  if (*status) return;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < (int64_t)n * n;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int q = (int)(e / n), p = (int)(e % n);
    out[(int64_t)piv[q] * n + p] = S[(int64_t)piv[p] * n + q];
  }
}

__global__ void k_gj_reset(int* pan, int n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) pan[i] = -1;
}

size_t coarse_panel_entries(int Nb) { return (size_t)2 * kPanel * Nb; }

cudaError_t coarse_invert(const double* A, double* Ainv, double* work, double* panel, int* piv, int Nb, int* status,
                          cudaStream_t s) {
  k_to_rowmajor<<<152 * 4, 256, 0, s>>>(A, work, Nb);
  int* pan = piv + Nb;
  k_gj_reset<<<(Nb + 255) / 256, 256, 0, s>>>(pan, Nb);
  double* W = panel;
  double* R = panel + (size_t)kPanel * Nb;
  unsigned low = 1;
  while (low < (unsigned)Nb) low = 2 * low + 1;
  const int threads = Nb >= 1024 ? 1024 : (Nb + 31) / 32 * 32;
  const unsigned tiles = (unsigned)((Nb + kGjTile - 1) / kGjTile);
  int panels = 0;
  for (int p = 0; p < Nb; p += kPanel, ++panels) {
    if (Nb <= 1024) k_gj_panel<1><<<1, threads, 0, s>>>(work, Nb, p, W, R, piv, pan, status, low);
    else if (Nb <= 2048) k_gj_panel<2><<<1, threads, 0, s>>>(work, Nb, p, W, R, piv, pan, status, low);
    else k_gj_panel_global<<<1, threads, 0, s>>>(work, Nb, p, W, R, piv, pan, status, low);
    k_gj_update<<<dim3(tiles, tiles), 128, 0, s>>>(work, Nb, p, W, R, pan, status);
  }
  k_gj_permute<<<152 * 4, 256, 0, s>>>(work, Ainv, Nb, piv, status);
  note_launch(3 + 2 * panels);
  return cudaGetLastError();
}

// One product of the coarse solve, y = A x (A column-major n x n) with what stands around it:
//   step 0: x1 = Ainv b        step 1: r = b - A x1        step 2: out = x1 + Ainv r
// b: the right-hand side (T, nc entries) continued by zeros, out: nc entries of T.  A block owns 8 rows,
// its 32 groups of 8 threads every 32nd column; their sums meet in shared memory in a fixed order.
// FP64 on few SMs is slow, so small systems are spread over n / 8 blocks (n = 126: 10.2 -> 3.7 us).
template <typename T, int STEP>
__global__ void __launch_bounds__(256) k_coarse_mv(const double* A, int n, int nc, const T* b, const double* x1,
                                                   const double* r, double* y, T* out) {
  chain_begin();
  __shared__ double part[32][9];
  A += (int64_t)blockIdx.y * n * n;                   // blockIdx.y: independent slot
  b += (int64_t)blockIdx.y * nc;
  if (STEP > 0) x1 += (int64_t)blockIdx.y * n;
  if (STEP == 2) { r += (int64_t)blockIdx.y * n; out += (int64_t)blockIdx.y * nc; }
  else y += (int64_t)blockIdx.y * n;
  const int lr = threadIdx.x & 7, g = threadIdx.x >> 3, i = blockIdx.x * 8 + lr;
  double acc = 0.0;
  if (i < n) {
#pragma unroll 4
    for (int j = g; j < n; j += 32) {
      const double x = STEP == 0 ? (j < nc ? (double)b[j] : 0.0) : (STEP == 1 ? x1[j] : r[j]);
      acc += A[(int64_t)j * n + i] * x;
    }
  }
  part[g][lr] = acc;
  __syncthreads();
  if (threadIdx.x < 64) {                             // 8 rows x 8 sums of four, then 8 rows
    double s = part[g][lr];
    s += part[g + 8][lr];
    s += part[g + 16][lr];
    s += part[g + 24][lr];
    part[g][lr] = s;
  }
  __syncthreads();
  if (threadIdx.x < 8 && i < n) {
    double s = part[0][lr];
#pragma unroll
    for (int k = 1; k < 8; ++k) s += part[k][lr];
    if (STEP == 0) y[i] = s;
    else if (STEP == 1) y[i] = (i < nc ? (double)b[i] : 0.0) - s;
    else if (i < nc) out[i] = (T)(x1[i] + s);
  }
}

template <typename T>
cudaError_t coarse_apply(const double* Ainv, const double* A, int n, int nc, const T* b, T* out, double* x1, double* r,
                         cudaStream_t s, int slots) {
  const dim3 grid((n + 7) / 8, slots);
  launch_chained(k_coarse_mv<T, 0>, grid, 256, 0, s, Ainv, n, nc, b, nullptr, nullptr, x1, nullptr);
  launch_chained(k_coarse_mv<T, 1>, grid, 256, 0, s, A, n, nc, b, x1, nullptr, r, nullptr);
  launch_chained(k_coarse_mv<T, 2>, grid, 256, 0, s, Ainv, n, nc, b, x1, r, nullptr, out);
  note_launch(3);
  return cudaGetLastError();
}
template cudaError_t coarse_apply<float>(const double*, const double*, int, int, const float*, float*, double*, double*,
                                         cudaStream_t, int);
template cudaError_t coarse_apply<double>(const double*, const double*, int, int, const double*, double*, double*,
                                          double*, cudaStream_t, int);


}  // namespace stmg
