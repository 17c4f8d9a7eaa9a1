// Vector kernels (see vec.cuh).  Grid-stride loops sized as a multiple of the SM count;
// reductions in a fixed order (block partial sums, then one block per result).
#include <algorithm>
#include "vec.cuh"
#include "chain.cuh"
#include "counters.hpp"

namespace stmg {

static inline int grid_for(int64_t n) {
  int64_t g = (n + 255) / 256;
  if (g > 152 * 16) g = 152 * 16;
  if (g < 1) g = 1;
  return (int)g;
}

template <typename T>
__global__ void k_axpby(int64_t n, T a, const T* x, T b, T* y) {
  chain_begin();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] = a * x[i] + b * y[i];
}

template <typename T>
cudaError_t vaxpby(int64_t n, T a, const T* x, T b, T* y, cudaStream_t s) {
  launch_chained(k_axpby<T>, grid_for(n), 256, 0, s, n, a, x, b, y);
  note_launch();
  return cudaGetLastError();
}

template <typename S, typename T>
__global__ void k_copy(int64_t n, const S* x, T* y) {
  chain_begin();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] = (T)x[i];
}

template <typename S, typename T>
cudaError_t vcopy(int64_t n, const S* x, T* y, cudaStream_t s) {
  launch_chained(k_copy<S, T>, grid_for(n), 256, 0, s, n, x, y);
  note_launch();
  return cudaGetLastError();
}

// Dot products in one launch: each block forms the partial sums of up to DOTS_PER_ROW basis vectors with
// w (w[i] is read once for all of them); the last block of a row of blocks to finish adds the partial
// sums, in block order.  Each thread accumulates its strided elements in index order and every sum
// has a fixed tree, so the result does not depend on which block is last.  Short vectors take few
// blocks: the launch is then over as soon as the data have been read.
constexpr int DOTS_PER_ROW = 4;

// Sums red[0 .. RED_THREADS) per row of `red`, rows q < cnt, into the first warp's lane 0 (v[q]).
template <int Q>
__device__ __forceinline__ void block_sums(double (*red)[RED_THREADS], double (&v)[Q]) {
  __syncthreads();
  if (threadIdx.x < 32) {
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      // a tree: FP64 additions are slow one after another
      double t[RED_THREADS / 32];
#pragma unroll
      for (int k = 0; k < RED_THREADS / 32; ++k) t[k] = red[q][threadIdx.x + 32 * k];
#pragma unroll
      for (int h = RED_THREADS / 64; h > 0; h >>= 1)
#pragma unroll
        for (int k = 0; k < h; ++k) t[k] += t[k + h];
      double s = t[0];
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
      v[q] = s;
    }
  }
}

// After a block has written its partial sums: true in the last of gridDim.x blocks (and resets count).
__device__ __forceinline__ bool last_block(unsigned* count) {
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    last = atomicAdd(count, 1u) == gridDim.x - 1;
    if (last) *count = 0;
  }
  __syncthreads();
  if (last) __threadfence();
  return last;
}

template <typename T>
__global__ void k_dots(int64_t n, int m, const T* X, int64_t ldx, const T* w, double* part,
                       double* out, unsigned* count) {
  chain_begin();
  __shared__ double red[DOTS_PER_ROW][RED_THREADS];
  const int l0 = blockIdx.y * DOTS_PER_ROW;
  const int cnt = m - l0 < DOTS_PER_ROW ? m - l0 : DOTS_PER_ROW;
  double acc[DOTS_PER_ROW] = {0.0, 0.0, 0.0, 0.0};
  const int64_t stride = (int64_t)gridDim.x * RED_THREADS;
  for (int64_t i = blockIdx.x * (int64_t)RED_THREADS + threadIdx.x; i < n; i += stride) {
    const double wi = (double)w[i];
    double xv[DOTS_PER_ROW];
#pragma unroll
    for (int q = 0; q < DOTS_PER_ROW; ++q) xv[q] = q < cnt ? (double)X[(l0 + q) * ldx + i] : 0.0;
#pragma unroll
    for (int q = 0; q < DOTS_PER_ROW; ++q) acc[q] += xv[q] * wi;
  }
#pragma unroll
  for (int q = 0; q < DOTS_PER_ROW; ++q) red[q][threadIdx.x] = acc[q];
  block_sums<DOTS_PER_ROW>(red, acc);
  if (threadIdx.x == 0)
    for (int q = 0; q < cnt; ++q) part[(int64_t)(l0 + q) * RED_BLOCKS + blockIdx.x] = acc[q];
  if (!last_block(count + blockIdx.y)) return;
#pragma unroll
  for (int q = 0; q < DOTS_PER_ROW; ++q) {
    double s = 0.0;
    if (q < cnt)
      for (int i = threadIdx.x; i < (int)gridDim.x; i += RED_THREADS) s += __ldcg(part + (int64_t)(l0 + q) * RED_BLOCKS + i);
    red[q][threadIdx.x] = s;
  }
  block_sums<DOTS_PER_ROW>(red, acc);
  if (threadIdx.x == 0)
    for (int q = 0; q < cnt; ++q) out[l0 + q] = acc[q];
}

// Short vectors: two elements a thread, up to two blocks an SM (eight a thread left most SMs idle; 2D 32^2
// Q2/P1 DG(1) slab solve 8.09 -> 7.87 ms).  Long ones: eight a thread, so that the last block has fewer partial
// sums to add (two a thread throughout: 2D 128^2 Q3/P2 DG(2) slab solve 1-2 % slower).
static inline int red_grid(int64_t n) {
  const int64_t g2 = std::min<int64_t>((n + 2 * RED_THREADS - 1) / (2 * RED_THREADS), 304);
  const int64_t g = std::max<int64_t>(g2, (n + 8 * RED_THREADS - 1) / (8 * RED_THREADS));
  return (int)(g < 1 ? 1 : (g > RED_BLOCKS ? RED_BLOCKS : g));
}
static inline unsigned* red_counters(double* scratch) { return reinterpret_cast<unsigned*>(scratch + (size_t)RED_BLOCKS * 64); }

template <typename T>
cudaError_t vdots(int64_t n, int m, const T* X, int64_t ldx, const T* w, double* out, double* scratch,
                  cudaStream_t s) {
  if (m <= 0) return cudaSuccess;
  if (m > 64) return cudaErrorInvalidValue;
  launch_chained(k_dots<T>, dim3(red_grid(n), (m + DOTS_PER_ROW - 1) / DOTS_PER_ROW), RED_THREADS, 0, s, n, m, X, ldx, w, scratch, out, red_counters(scratch));
  note_launch();
  return cudaGetLastError();
}

// w -= sum_l h[l] X[l]; NORM: also out = sum_i w_i^2 of the result (the same two-stage sum).
template <typename T, bool NORM>
__global__ void k_sub_comb(int64_t n, int m, const T* X, int64_t ldx, const double* h,
                           T* w, double* part, double* out, unsigned* count) {
  chain_begin();
  __shared__ double hs[64];
  __shared__ double red[1][RED_THREADS];
  if (threadIdx.x < m) hs[threadIdx.x] = h[threadIdx.x];
  __syncthreads();
  double sq[1] = {0.0};
  for (int64_t i = blockIdx.x * (int64_t)RED_THREADS + threadIdx.x; i < n; i += (int64_t)gridDim.x * RED_THREADS) {
    double acc = (double)w[i];
#pragma unroll 8
    for (int l = 0; l < m; ++l) acc -= hs[l] * (double)X[l * ldx + i];
    const T wi = (T)acc;
    w[i] = wi;
    if (NORM) sq[0] += (double)wi * (double)wi;
  }
  if (NORM) {
    red[0][threadIdx.x] = sq[0];
    block_sums<1>(red, sq);
    if (threadIdx.x == 0) part[blockIdx.x] = sq[0];
    if (!last_block(count)) return;
    double s = 0.0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += RED_THREADS) s += __ldcg(part + i);
    red[0][threadIdx.x] = s;
    block_sums<1>(red, sq);
    if (threadIdx.x == 0) *out = sq[0];
  }
}

template <typename T>
cudaError_t vsub_comb(int64_t n, int m, const T* X, int64_t ldx, const double* h, T* w, cudaStream_t s) {
  if (m <= 0) return cudaSuccess;
  if (m > 64) return cudaErrorInvalidValue;
  launch_chained(k_sub_comb<T, false>, grid_for(n), RED_THREADS, 0, s, n, m, X, ldx, h, w, (double*)nullptr, (double*)nullptr, (unsigned*)nullptr);
  note_launch();
  return cudaGetLastError();
}

template <typename T>
cudaError_t vsub_comb_norm(int64_t n, int m, const T* X, int64_t ldx, const double* h, T* w, double* out, double* scratch,
                           cudaStream_t s) {
  if (m <= 0 || m > 64) return cudaErrorInvalidValue;
  launch_chained(k_sub_comb<T, true>, red_grid(n), RED_THREADS, 0, s, n, m, X, ldx, h, w, scratch, out, red_counters(scratch));
  note_launch();
  return cudaGetLastError();
}

struct Coef64 { double v[64]; };

__global__ void k_add_comb(int64_t n, int m, const double* Z, int64_t ldz, Coef64 y,
                           double* x) {
  chain_begin();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    double acc = x[i];
    for (int l = 0; l < m; ++l) acc += y.v[l] * Z[l * ldz + i];
    x[i] = acc;
  }
}

cudaError_t vadd_comb_host(int64_t n, int m, const double* Z, int64_t ldz, const double* y, double* x,
                           cudaStream_t s) {
  if (m <= 0) return cudaSuccess;
  if (m > 64) return cudaErrorInvalidValue;
  Coef64 c{};
  for (int l = 0; l < m; ++l) c.v[l] = y[l];
  launch_chained(k_add_comb, grid_for(n), 256, 0, s, n, m, Z, ldz, c, x);
  note_launch();
  return cudaGetLastError();
}

template <typename T>
__global__ void k_scale_inv_dev(int64_t n, const T* x, const double* nrm, T* y) {
  chain_begin();
  const double f = 1.0 / *nrm;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] = (T)((double)x[i] * f);
}

template <typename T>
cudaError_t vscale_inv_dev(int64_t n, const T* x, const double* nrm, T* y, cudaStream_t s) {
  launch_chained(k_scale_inv_dev<T>, grid_for(n), 256, 0, s, n, x, nrm, y);
  note_launch();
  return cudaGetLastError();
}

template <typename T>
__global__ void k_scale(int64_t n, T a, const T* x, T* y) {
  chain_begin();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] = a * x[i];
}

template <typename T>
cudaError_t vscale(int64_t n, T a, const T* x, T* y, cudaStream_t s) {
  launch_chained(k_scale<T>, grid_for(n), 256, 0, s, n, a, x, y);
  note_launch();
  return cudaGetLastError();
}

__global__ void k_finite(int64_t n, const double* x, int* flag) {
  chain_begin();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    if (!isfinite(x[i])) *flag = 1;
}

cudaError_t vfinite(int64_t n, const double* x, int* flag, cudaStream_t s) {
  launch_chained(k_finite, grid_for(n), 256, 0, s, n, x, flag);
  note_launch();
  return cudaGetLastError();
}

template cudaError_t vaxpby<float>(int64_t, float, const float*, float, float*, cudaStream_t);
template cudaError_t vaxpby<double>(int64_t, double, const double*, double, double*, cudaStream_t);
template cudaError_t vcopy<double, float>(int64_t, const double*, float*, cudaStream_t);
template cudaError_t vcopy<float, double>(int64_t, const float*, double*, cudaStream_t);
template cudaError_t vcopy<double, double>(int64_t, const double*, double*, cudaStream_t);
template cudaError_t vcopy<float, float>(int64_t, const float*, float*, cudaStream_t);
template cudaError_t vdots<float>(int64_t, int, const float*, int64_t, const float*, double*, double*, cudaStream_t);
template cudaError_t vdots<double>(int64_t, int, const double*, int64_t, const double*, double*, double*, cudaStream_t);
template cudaError_t vsub_comb<float>(int64_t, int, const float*, int64_t, const double*, float*, cudaStream_t);
template cudaError_t vsub_comb<double>(int64_t, int, const double*, int64_t, const double*, double*, cudaStream_t);
template cudaError_t vsub_comb_norm<double>(int64_t, int, const double*, int64_t, const double*, double*, double*, double*,
                                            cudaStream_t);
template cudaError_t vscale_inv_dev<double>(int64_t, const double*, const double*, double*, cudaStream_t);
template cudaError_t vscale_inv_dev<float>(int64_t, const float*, const double*, float*, cudaStream_t);
template cudaError_t vscale<float>(int64_t, float, const float*, float*, cudaStream_t);
template cudaError_t vscale<double>(int64_t, double, const double*, double*, cudaStream_t);

}  // namespace stmg
