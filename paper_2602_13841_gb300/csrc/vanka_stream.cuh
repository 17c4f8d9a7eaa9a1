// Additive Vanka sweep with stored patch inverses (Eq. vanka0): the patch solves of all cells in one
// launch (k_vanka_stream), then d += omega * the sum of each node's cells (k_node_sum).
//
// Per cell, through the time-diagonalised inverse (vanka_patch.cuh):
//   rt_e = sum_a F[e][a] res_a  (per spatial patch DoF),  yhat_e = T_e^{-1} rt_e,
//   y_a = sum_e Re(G[a][e] yhat_e).
// The sweep is a stream of the stored inverses, each entry read once and used in one or two
// multiply-adds, so it is bound by HBM and the kernel's work is to keep enough loads in flight at few
// instructions: the columns of an inverse are contiguous, P chunks each (16 bytes of a complex, 8 of
// a real block: RC rows), so P x JS threads take JS columns per step by consecutive chunks, straight
// into registers, U steps ahead; the transformed residual comes from shared memory (broadcast
// reads), and the JS partial sums of a row meet there at the end of a block.  Rows of the velocity go
// to the cell buffer of the operator kernels, pressure rows (each in one patch) update d directly.
// No colouring: one launch over all cells has one ramp and one tail instead of 2^D, and no patch waits
// for another colour; the buffer adds 5 % to the traffic in 2D, 1 % in 3D.
// Measured, all cells of a level, patch solves + node sums (of the 6.80 TB/s copy peak): 2D 256^2 Q3/P2
// DG(2) 170 + 10 us (0.98 for the solves), against 234 us for the four colours of a persistent kernel
// that staged the inverses in a shared-memory ring; 3D 32^3 Q2/P1 DG(2) 462 + 13 us (0.91), against 622
// (one staged cell per block); 3D 16^3 Q3/P2 DG(2) 340 + 7 us (0.87), against 600 (a row per thread).
// Smaller teams did better than larger ones (m = 85: 96 threads 462 us, 224 threads 610 us): more blocks
// in flight, none of whose phases waits for another's barrier.
#pragma once
#include "operator_cells.cuh"
#include "vanka.cuh"

namespace stmg {

// Columns per step: the count whose threads fill whole warps best within `target` threads.
__host__ __device__ constexpr int stream_columns(int P, int target) {
  int best = 1, bt = 0, bw = 1;
  for (int js = 1; js * P <= target; ++js) {
    const int t = js * P, w = (t + 31) / 32;
    if ((long long)t * bw >= (long long)bt * w) { best = js; bt = t; bw = w; }
  }
  return best;
}

template <typename T, typename SI, int D, int N>
struct StreamShape {
  static constexpr int MS = patch_rows<D, N>(), MV = D * Shape<D, N>::Q, ST = inv_stride(MS, (int)sizeof(SI));
  static constexpr int RC = 8 / (int)sizeof(SI);      // rows per chunk
  static constexpr int P = ST / RC;
  static constexpr int TARGET = MS <= 64 ? (sizeof(SI) == 8 ? 128 : 64) : MS <= 128 ? 96 : (P <= 256 ? 256 : 512);
  static constexpr int JS = stream_columns(P, TARGET);
  static constexpr int THREADS = (P * JS + 31) / 32 * 32;
  static constexpr int NIT = (MS + JS - 1) / JS;
  static constexpr int NB = NIT <= 13 ? 1 : (NIT + 7) / 8, U = (NIT + NB - 1) / NB;   // batches of U steps
  static constexpr int MP = JS * U * NB;              // columns incl. the steps past the end (zero residual)
  static constexpr int BLOCKS = THREADS <= 64 ? 9 : THREADS <= 96 ? 6 : THREADS <= 128 ? 4 : 2;
  static_assert(ST % RC == 0, "chunks do not straddle columns");
};

// A batch of U chunks of a thread: 16 bytes each of a complex block, 8 of a real one.
template <bool C, int U> struct ChunkBatch { uint32_t w[U][C ? 4 : 2]; };

// The inverses are written by kernels that end before this one starts (they are not chained), so they may
// take the non-coherent path; volatile keeps the loads after chain_begin().
// q: the thread's chunk of the batch's first column; STEP bytes between its columns; `left` columns from
// the first one on exist (chunks past them are zero).
template <bool C, int U, int STEP>
__device__ __forceinline__ void load_batch(ChunkBatch<C, U>& c, const unsigned char* q, int left, int js_step,
                                           uint64_t pol) {
#pragma unroll
  for (int u = 0; u < U; ++u) {
    if (u * js_step < left) {
      if constexpr (C)
        asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
            : "=r"(c.w[u][0]), "=r"(c.w[u][1]), "=r"(c.w[u][2]), "=r"(c.w[u][3]) : "l"(q + u * STEP), "l"(pol));
      else
        asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v2.u32 {%0, %1}, [%2], %3;"
            : "=r"(c.w[u][0]), "=r"(c.w[u][1]) : "l"(q + u * STEP), "l"(pol));
    } else {
#pragma unroll
      for (int x = 0; x < (C ? 4 : 2); ++x) c.w[u][x] = 0;
    }
  }
}

// Entries of a chunk: row r of a real block, (re, im) of row r of a complex block.
template <typename SI> struct ChunkOf;
template <> struct ChunkOf<float> {
  __device__ static float re(const uint32_t* w, int r) { return __uint_as_float(w[r]); }
  __device__ static float2 cx(const uint32_t* w, int r) { return {__uint_as_float(w[2 * r]), __uint_as_float(w[2 * r + 1])}; }
};
template <> struct ChunkOf<double> {
  __device__ static double re(const uint32_t* w, int) { return __hiloint2double((int)w[1], (int)w[0]); }
  __device__ static double2 cx(const uint32_t* w, int) {
    return {__hiloint2double((int)w[1], (int)w[0]), __hiloint2double((int)w[3], (int)w[2])};
  }
};
template <> struct ChunkOf<__half> {
  __device__ static float2 pair(uint32_t w) { return __half22float2(*reinterpret_cast<const __half2*>(&w)); }
  __device__ static float re(const uint32_t* w, int r) { const float2 p = pair(w[r >> 1]); return (r & 1) ? p.y : p.x; }
  __device__ static float2 cx(const uint32_t* w, int r) { return pair(w[r]); }
};

template <typename T, typename SI, bool C, int U, int JS, int RC>
__device__ __forceinline__ void use_batch(const ChunkBatch<C, U>& c, const T* r, T (&ar)[RC], T (&ai)[RC]) {
#pragma unroll
  for (int u = 0; u < U; ++u) {
    if constexpr (C) {
      const T xr = r[2 * JS * u], xi = r[2 * JS * u + 1];
#pragma unroll
      for (int q = 0; q < RC; ++q) {
        const auto v = ChunkOf<SI>::cx(c.w[u], q);
        const T vr = (T)v.x, vi = (T)v.y;
        ar[q] += vr * xr - vi * xi;
        ai[q] += vr * xi + vi * xr;
      }
    } else {
      const T x = r[JS * u];
#pragma unroll
      for (int q = 0; q < RC; ++q) ar[q] += (T)ChunkOf<SI>::re(c.w[u], q) * x;
    }
  }
}

// Grid: the cells c0, c0 + 1, ... (one block each) x slots.  KP1 = 1: one real block; 2: one complex
// block; 3: one of each, in the order the eigenvalues come.  first: the correction is zero on entry and
// not read.  stream: the inverses of the level exceed what L2 keeps, so they pass through it evicted
// first; smaller levels are read again by the next sweep and stay.
template <typename T, typename SI, int D, int N, int KP1>
__global__ void __launch_bounds__(StreamShape<T, SI, D, N>::THREADS, StreamShape<T, SI, D, N>::BLOCKS)
k_vanka_stream(LevelArgs<T> L, const SI* inv, const float* scale, const T* res,
               T* d, T omega_p, const __grid_constant__ TEig<T> te, CellBuf<T> cb, int64_t c0,
               SlotStrides zs, int first, int stream) {
  chain_begin();
  using Sh = StreamShape<T, SI, D, N>;
  constexpr int MS = Sh::MS, MV = Sh::MV, ST = Sh::ST, RC = Sh::RC, P = Sh::P, JS = Sh::JS, U = Sh::U, NB = Sh::NB;
  constexpr int NL = Shape<D, N>::Q, NPC = MS - MV, NT = Sh::THREADS, MP = Sh::MP, ROWS = (MS + NT - 1) / NT;
  constexpr bool HAS_C = KP1 > 1, HAS_R = KP1 != 2;
  // transformed residual of the complex block (pairs) and of the real one, zero past the last row
  __shared__ __align__(16) T rtc[HAS_C ? 2 * MP : 2];
  __shared__ __align__(16) T rtr[HAS_R ? MP : 2];
  __shared__ __align__(16) T red[JS][KP1][ST];        // partial sums: complex re, im, then real
  inv += blockIdx.y * zs.inv;
  if (scale) scale += blockIdx.y * zs.scale;
  res += blockIdx.y * zs.vec;
  d += blockIdx.y * zs.vec;
  const int tid = threadIdx.x;
  const int64_t cell = c0 + blockIdx.x;
  uint64_t pol;
  if (stream) asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  else asm("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(pol));
  const int p = tid % P, js = tid / P;
  const bool on = js < JS;
  const int ec = KP1 == 3 && !te.cplx[0] ? 1 : 0, er = KP1 == 3 ? 1 - ec : 0;      // complex and real block
  constexpr int CS = ST * (int)sizeof(SI);            // bytes of a real column
  const unsigned char* blob = reinterpret_cast<const unsigned char*>(inv + cell * (int64_t)KP1 * MS * ST);
  const unsigned char* qc = blob + (size_t)(ec ? MS * CS : 0) + (size_t)js * (2 * CS) + p * 16;
  const unsigned char* qr = blob + (size_t)(KP1 == 3 && er ? 2 * MS * CS : 0) + (size_t)js * CS + p * 8;
  const int left = on ? MS - js : 0;                  // columns js, js + JS, ... < MS
  // the first batches are on their way before anything else
  ChunkBatch<true, U> bc;
  ChunkBatch<false, U> br;
  if constexpr (HAS_C) load_batch<true, U, JS * 2 * CS>(bc, qc, left, JS, pol);
  if constexpr (HAS_R && (NB == 1 || !HAS_C)) load_batch<false, U, JS * CS>(br, qr, left, JS, pol);
  // ---- residual on the patch, in the time eigenbasis
  int cc[3];
  {
    unsigned t = (unsigned)cell, n = (unsigned)L.n;
    cc[0] = (int)(t % n); t /= n;
    cc[1] = D == 3 ? (int)(t % n) : (int)t;
    cc[2] = D == 3 ? (int)(t / n) : 0;
  }
  const int64_t n1 = L.N1;
  const int64_t corner = (int64_t)cc[0] * (N - 1) + n1 * ((int64_t)cc[1] * (N - 1) + (D == 3 ? n1 * ((int64_t)cc[2] * (N - 1)) : 0));
#pragma unroll
  for (int x = 0; x < ROWS; ++x) {
    const int i = tid + x * NT;
    if (i < MS) {
      int64_t g, sa;
      if (i < MV) {
        const int c = i / NL, ni = i - c * NL;
        g = c * L.nnodes + corner + ni % N + n1 * ((ni / N) % N + (D == 3 ? n1 * (ni / (N * N)) : 0));
        sa = L.Nv;
      } else {
        g = (int64_t)KP1 * L.Nv + cell * NPC + (i - MV);
        sa = L.Np;
      }
      T ra[KP1];
#pragma unroll
      for (int a = 0; a < KP1; ++a) ra[a] = res[g + a * sa];
      if constexpr (HAS_C) {
        T fr = 0, fi = 0;
#pragma unroll
        for (int a = 0; a < KP1; ++a) { fr += te.Fre[ec][a] * ra[a]; fi += te.Fim[ec][a] * ra[a]; }
        rtc[2 * i] = fr;
        rtc[2 * i + 1] = fi;
      }
      if constexpr (HAS_R) {
        T fr = 0;
#pragma unroll
        for (int a = 0; a < KP1; ++a) fr += te.Fre[er][a] * ra[a];
        rtr[i] = fr;
      }
    }
  }
  for (int i = MS + tid; i < MP; i += NT) {
    if constexpr (HAS_C) { rtc[2 * i] = 0; rtc[2 * i + 1] = 0; }
    if constexpr (HAS_R) rtr[i] = 0;
  }
  __syncthreads();
  // ---- the products; the next batch is loaded while one is used
  if (on) {
    if constexpr (HAS_C) {
      T ar[RC], ai[RC];
#pragma unroll
      for (int r = 0; r < RC; ++r) { ar[r] = 0; ai[r] = 0; }
      const T* r = rtc + 2 * js;
#pragma unroll 1
      for (int b = 1; b < NB; ++b) {
        ChunkBatch<true, U> nx;
        load_batch<true, U, JS * 2 * CS>(nx, qc + (size_t)b * (U * JS * 2 * CS), left - b * (U * JS), JS, pol);
        use_batch<T, SI, true, U, JS, RC>(bc, r, ar, ai);
        r += 2 * JS * U;
        bc = nx;
      }
      if constexpr (HAS_R && NB > 1) load_batch<false, U, JS * CS>(br, qr, left, JS, pol);
      use_batch<T, SI, true, U, JS, RC>(bc, r, ar, ai);
#pragma unroll
      for (int q = 0; q < RC; ++q) { red[js][0][RC * p + q] = ar[q]; red[js][1][RC * p + q] = ai[q]; }
    }
    if constexpr (HAS_R) {
      T ar[RC], ai[RC];
#pragma unroll
      for (int r = 0; r < RC; ++r) ar[r] = 0;
      const T* r = rtr + js;
#pragma unroll 1
      for (int b = 1; b < NB; ++b) {
        ChunkBatch<false, U> nx;
        load_batch<false, U, JS * CS>(nx, qr + (size_t)b * (U * JS * CS), left - b * (U * JS), JS, pol);
        use_batch<T, SI, false, U, JS, RC>(br, r, ar, ai);
        r += JS * U;
        br = nx;
      }
      use_batch<T, SI, false, U, JS, RC>(br, r, ar, ai);
#pragma unroll
      for (int q = 0; q < RC; ++q) red[js][KP1 - 1][RC * p + q] = ar[q];
    }
  }
  __syncthreads();
  // ---- back to the time nodes
#pragma unroll
  for (int x = 0; x < ROWS; ++x) {
    const int i = tid + x * NT;
    if (i >= MS) break;
    T ya[KP1];
#pragma unroll
    for (int a = 0; a < KP1; ++a) ya[a] = 0;
    if constexpr (HAS_C) {
      T yr = red[0][0][i], yi = red[0][1][i];
#pragma unroll
      for (int s = 1; s < JS; ++s) { yr += red[s][0][i]; yi += red[s][1][i]; }
      const T sc = scale ? (T)scale[cell * te.nblk + ec] : (T)1;
      yr *= sc;
      yi *= sc;
#pragma unroll
      for (int a = 0; a < KP1; ++a) ya[a] += te.Gre[a][ec] * yr - te.Gim[a][ec] * yi;
    }
    if constexpr (HAS_R) {
      T yr = red[0][KP1 - 1][i];
#pragma unroll
      for (int s = 1; s < JS; ++s) yr += red[s][KP1 - 1][i];
      yr *= scale ? (T)scale[cell * te.nblk + er] : (T)1;
#pragma unroll
      for (int a = 0; a < KP1; ++a) ya[a] += te.Gre[a][er] * yr;
    }
    if (i < MV) {
      const int c = i / NL, ni = i - c * NL, ix = ni % N, iy = (ni / N) % N, iz = ni / (N * N);
      const int64_t row = (int64_t)L.n * N;
      T* o = cb.s + blockIdx.y * cb.col + (int64_t)(cc[D - 1] % cb.P) * cb.plane + (int64_t)cc[0] * N + ix +
             (D == 3 ? (((int64_t)cc[1] * N + iz) * N + iy) : (int64_t)iy) * row;
#pragma unroll
      for (int a = 0; a < KP1; ++a) o[(int64_t)(a * D + c) * cb.comp] = ya[a];
    } else {
      const int64_t g = (int64_t)KP1 * L.Nv + cell * NPC + (i - MV);
#pragma unroll
      for (int a = 0; a < KP1; ++a) d[g + a * L.Np] = (first ? (T)0 : d[g + a * L.Np]) + omega_p * ya[a];
    }
  }
}

// Failure-test hook of sweeps whose kernels have no wait of their own: one block waits (bounded) for bytes
// that are never sent and sets the flag that every sweep's caller reads.  It stands in for the sweep, so that
// the correction is left as it was and the sweep's kernels need not read the flag (0.9 us of 50 in the node
// sums of a 2D 256^2 Q3/P2 DG(2) apply when they did).
__global__ inline void k_wait_hook(int* wstat, unsigned extra_tx) {
  __shared__ uint64_t bar;
  const uint32_t b = smem_addr(&bar);
  mbar_init(b, 1);
  mbar_expect_tx(b, extra_tx);
  if (!mbar_wait_bounded(b, 0, kWaitLimit)) atomicExch(wstat, 1);
}

}  // namespace stmg
