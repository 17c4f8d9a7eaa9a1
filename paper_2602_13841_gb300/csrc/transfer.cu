// Grid transfer kernels and their host set-up (see transfer.hpp).
#include <algorithm>
#include <cmath>
#include <vector>

#include "handle.hpp"
#include "transfer.hpp"
#include "chain.cuh"
#include "counters.hpp"

namespace stmg {

// Output nodes of a block of k_transfer_tile along x, y, z.
constexpr int kTile2[3] = {16, 8, 1}, kTile3[3] = {8, 4, 4};

// ---------------------------------------------------------------------------- host set-up
// The rows of a 1D operator as windows of columns and, FP64, as lists of the entries in them (see Line1D).
static Line1D upload_lines(Handle* h, int rows, int cols, const std::vector<std::vector<std::pair<int, double>>>& R) {
  Line1D c;
  c.rows = rows; c.cols = cols;
  std::vector<int2> win(rows);
  std::vector<int> cnt(rows);
  for (int i = 0; i < rows; ++i) {
    int lo = cols, hi = -1;
    for (auto& e : R[i]) { lo = std::min(lo, e.first); hi = std::max(hi, e.first); }
    if (hi < 0) { lo = 0; hi = 0; }
    win[i] = make_int2(lo, hi - lo + 1);
    cnt[i] = (int)R[i].size();
    c.width = std::max(c.width, win[i].y);
    c.entries = std::max(c.entries, cnt[i]);
    c.gaps = c.gaps || cnt[i] < win[i].y;
  }
  std::vector<float> v32((size_t)rows * c.width, 0.0f);
  std::vector<double> v64((size_t)rows * c.entries, 0.0);
  std::vector<int> off((size_t)rows * c.entries, 0);
  for (int i = 0; i < rows; ++i)
    for (int e = 0; e < cnt[i]; ++e) {
      const int o = R[i][e].first - win[i].x;
      v32[(size_t)i * c.width + o] = (float)R[i][e].second;
      v64[(size_t)i * c.entries + e] = R[i][e].second;
      off[(size_t)i * c.entries + e] = o;
    }
  const int tile = h->levels[0].d == 3 ? kTile3[1] : kTile2[1];
  for (int g = 0; g < rows; g += tile) {
    int lo = win[g].x, hi = lo;
    for (int i = g; i < rows && i < g + tile; ++i) { lo = std::min(lo, win[i].x); hi = std::max(hi, win[i].x + win[i].y); }
    c.span = std::max(c.span, hi - lo);
  }
  c.win = (int2*)h->dalloc(win.size() * sizeof(int2));
  c.cnt = (int*)h->dalloc(cnt.size() * sizeof(int));
  c.off = (int*)h->dalloc(off.size() * sizeof(int));
  c.val64 = (double*)h->dalloc(v64.size() * sizeof(double));
  c.val32 = (float*)h->dalloc(v32.size() * sizeof(float));
  h->upload(c.win, win.data(), win.size() * sizeof(int2));
  h->upload(c.cnt, cnt.data(), cnt.size() * sizeof(int));
  h->upload(c.off, off.data(), off.size() * sizeof(int));
  h->upload(c.val64, v64.data(), v64.size() * sizeof(double));
  h->upload(c.val32, v32.data(), v32.size() * sizeof(float));
  return c;
}

// rows: value at positions x (in cells of the `n`-cell line) of the global 1D basis of degree r+1
static std::vector<std::vector<std::pair<int, double>>> eval_rows(int n, int r, const std::vector<double>& x) {
  auto g = gauss_lobatto_nodes(r + 2);
  for (auto& v : g) v = 0.5 * (v + 1.0);
  std::vector<std::vector<std::pair<int, double>>> R(x.size());
  for (size_t p = 0; p < x.size(); ++p) {
    int c = (int)std::floor(x[p]);
    if (c > n - 1) c = n - 1;
    if (c < 0) c = 0;
    double xi = x[p] - c;
    for (int j = 0; j < r + 2; ++j) {
      double v = lagrange(g, j, xi);
      if (std::fabs(v) > 1e-14) R[p].push_back({c * (r + 1) + j, v});
    }
  }
  return R;
}

static std::vector<double> node_positions(int n, int r, double scale) {
  auto g = gauss_lobatto_nodes(r + 2);
  std::vector<double> x;
  for (int c = 0; c < n; ++c)
    for (int i = 0; i <= r; ++i) x.push_back((c + 0.5 * (g[i] + 1.0)) * scale);
  x.push_back(n * scale);
  return x;
}

void build_transfer(Handle* h, Transfer& tr, const Level& f, const Level& c) {
  tr.fine = &f; tr.coarse = &c;
  const double cf = (double)c.n / f.n;
  auto R = eval_rows(c.n, c.r, node_positions(f.n, f.r, cf));
  tr.P1 = upload_lines(h, f.N1, c.N1, R);
  std::vector<std::vector<std::pair<int, double>>> RT(c.N1);
  for (int i = 0; i < (int)R.size(); ++i)
    for (auto& e : R[i]) RT[e.first].push_back({i, e.second});
  tr.P1T = upload_lines(h, c.N1, f.N1, RT);
  tr.I1 = upload_lines(h, c.N1, f.N1, eval_rows(f.n, f.r, node_positions(c.n, c.r, 1.0 / cf)));
  // time
  auto tf = radau_right_nodes(f.k), tc = radau_right_nodes(c.k);
  for (int i = 0; i <= f.k; ++i)
    for (int j = 0; j <= c.k; ++j) {
      tr.E[i][j] = (c.k == 0) ? 1.0 : lagrange(tc, j, tf[i]);
      tr.Et[j][i] = (f.k == 0) ? 1.0 : lagrange(tf, i, tc[j]);
    }
  // pressure child expansions: T1[b][i][j] = coeff of P_j(2x-1) in P_i(2 (b+x)/2 - 1)
  tr.ratio = f.n / c.n;
  tr.ntypes = (tr.ratio == 2) ? (1 << f.d) : 1;
  const int rr = f.r > c.r ? f.r : c.r;
  auto gx = gauss_legendre_nodes(rr + 2);
  auto gw = gauss_legendre_weights(gx);
  double T1[2][4][4] = {};
  for (int b = 0; b < 2; ++b)
    for (int i = 0; i <= rr; ++i)
      for (int j = 0; j <= rr; ++j) {
        double s = 0;
        for (size_t q = 0; q < gx.size(); ++q) {
          double x = 0.5 * (gx[q] + 1.0), w = 0.5 * gw[q];
          double pi, dpi, pj, dpj;
          legendre(i, 2.0 * (0.5 * (b + x)) - 1.0, &pi, &dpi);
          legendre(j, 2.0 * x - 1.0, &pj, &dpj);
          s += w * pi * pj;
        }
        T1[b][i][j] = s * (2 * j + 1);
      }
  const int npf = f.npc, npc = c.npc;
  std::vector<double> PT(tr.ntypes * npf * npc, 0.0);
  for (int t = 0; t < tr.ntypes; ++t)
    for (int mf = 0; mf < npf; ++mf)
      for (int mc = 0; mc < npc; ++mc) {
        double v;
        if (tr.ratio == 1) {
          v = 1.0;
          for (int l = 0; l < f.d; ++l) if (f.tabs.modes[mf][l] != c.tabs.modes[mc][l]) v = 0.0;
        } else {
          v = 1.0;
          for (int l = 0; l < f.d; ++l) v *= T1[(t >> l) & 1][c.tabs.modes[mc][l]][f.tabs.modes[mf][l]];
        }
        PT[(t * npf + mf) * npc + mc] = v;
      }
  std::vector<float> PT32(PT.begin(), PT.end());
  tr.PT64 = (double*)h->dalloc(PT.size() * sizeof(double));
  tr.PT32 = (float*)h->dalloc(PT.size() * sizeof(float));
  h->upload(tr.PT64, PT.data(), PT.size() * sizeof(double));
  h->upload(tr.PT32, PT32.data(), PT32.size() * sizeof(float));
}

// ---------------------------------------------------------------------------- kernels
// One transfer in one launch: out = (M (x) L (x) .. (x) L) in on the velocity, L the 1D operator along
// every axis and M the time matrix, and the pressure modes (op: prolongation, restriction or none), added
// to out where `add`.  Nothing passes through memory between axes, time and pressure.  Two forms:
//   k_transfer       a thread owns one output node and component and sums the product of its D row windows
//                    for every input time node; rows without gaps only (every column of a window counts).
//   k_transfer_tile  a block owns a tile of output nodes of one component and sums axis by axis, the lines in
//                    between in shared memory: a window of w entries costs D w products instead of w^D, a zero
//                    in a window none (nor does it carry an infinity over from its column).
// See transfer_launch for which is taken.
template <typename T> struct MatT { T m[MAXKP1][MAXKP1]; };
enum { P_NONE = 0, P_PROLONG = 1, P_RESTRICT = 2 };

template <typename T>
struct TransferArgs {
  const T* in;
  T* out;
  const int2* win;
  const int *cnt, *off;
  const T* val;
  int width, nin1, nout1, kin, kout, add, mix;        // mix: M is not the identity
  int64_t nin, nout, vin, vout;                       // nodes and velocity entries per time node
  int64_t nvel, total;                                // entries of the velocity per time node, and with the pressure
  MatT<T> M;
  int pop, nf, ratio, npf, npc;                       // pressure: kind, fine cells per axis, modes fine / coarse
  const T* PT;
  int64_t pin, pout, zin, zout;                       // pressure entries per time node; slot strides
  int span, tx, ty, tz;                               // tiles: input lines per axis at most, tiles per axis
  int64_t nvb;                                        // ... and velocity blocks (the others do pressure)
};

// Mix the sums of the input time nodes and write entry o (stride so between time nodes).
template <typename T>
__device__ __forceinline__ void transfer_store(const TransferArgs<T>& A, T* out, int64_t o, int64_t so,
                                               const T (&acc)[MAXKP1]) {
#pragma unroll
  for (int a = 0; a < MAXKP1; ++a) {
    if (a >= A.kout) break;
    T r = acc[a];
    if (A.mix) {
      r = A.M.m[a][0] * acc[0];
#pragma unroll
      for (int b = 1; b < MAXKP1; ++b)
        if (b < A.kin) r += A.M.m[a][b] * acc[b];
    }
    out[o + a * so] = A.add ? out[o + a * so] + r : r;
  }
}

// Output pressure entry i of every time node.
template <typename T, int D>
__device__ __forceinline__ void transfer_pressure(const TransferArgs<T>& A, const T* in, T* out, int64_t i) {
  T acc[MAXKP1];
#pragma unroll
  for (int b = 0; b < MAXKP1; ++b) acc[b] = 0;
  const T* p = in + A.kin * A.vin;
  const bool pro = A.pop == P_PROLONG;
  const int no = pro ? A.npf : A.npc, n = pro ? A.nf : A.nf / A.ratio;
  const int m = (int)(i % no);
  unsigned rem = (unsigned)(i / no);
  int cm[3] = {0, 0, 0};
#pragma unroll
  for (int l = 0; l < D; ++l) { cm[l] = (int)(rem % (unsigned)n); rem /= (unsigned)n; }
  // prolongation: the coarse cell that holds the fine one; restriction: the fine cells of the coarse one
  const int children = !pro && A.ratio == 2 ? (1 << D) : 1, no2 = pro ? A.nf / A.ratio : A.nf;
  for (int ch = 0; ch < children; ++ch) {
    int64_t cell = 0, s = 1;
    int type = ch;
    if (pro) type = 0;
#pragma unroll
    for (int l = 0; l < D; ++l) {
      const int x = pro ? cm[l] / A.ratio : cm[l] * A.ratio + ((ch >> l) & 1);
      if (pro && A.ratio == 2) type |= (cm[l] & 1) << l;
      cell += x * s;
      s *= no2;
    }
    const T* P = A.PT + (int64_t)type * A.npf * A.npc;
    const int ni = pro ? A.npc : A.npf;
    const T* q = p + cell * ni;
    for (int k = 0; k < ni; ++k) {
      const T f = pro ? P[m * A.npc + k] : P[k * A.npc + m];
#pragma unroll
      for (int b = 0; b < MAXKP1; ++b)
        if (b < A.kin) acc[b] += f * q[b * A.pin + k];
    }
  }
  transfer_store(A, out, A.kout * A.vout + i, A.pout, acc);
}

template <typename T, int D>
__global__ void k_transfer(const __grid_constant__ TransferArgs<T> A) {
  chain_begin();
  const T* in = A.in + blockIdx.y * A.zin;            // blockIdx.y: independent slot
  T* out = A.out + blockIdx.y * A.zout;
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= A.total) return;
  if (t >= A.nvel) { transfer_pressure<T, D>(A, in, out, t - A.nvel); return; }
  T acc[MAXKP1];
#pragma unroll
  for (int b = 0; b < MAXKP1; ++b) acc[b] = 0;
  const int c = (int)(t / A.nout);
  unsigned rem = (unsigned)(t - c * A.nout);
  int2 w[3];
  const T* v[3];
#pragma unroll
  for (int l = 0; l < D; ++l) {
    const unsigned q = rem / (unsigned)A.nout1, g = rem - q * (unsigned)A.nout1;
    rem = q;
    w[l] = A.win[g];
    v[l] = A.val + (int64_t)g * A.width;
  }
  const int64_t n1 = A.nin1;
  const T* src = in + c * A.nin + w[0].x + n1 * (w[1].x + (D == 3 ? n1 * w[2].x : 0));
  for (int z = 0; z < (D == 3 ? w[2].y : 1); ++z)
    for (int y = 0; y < w[1].y; ++y) {
      const T wyz = D == 3 ? v[2][z] * v[1][y] : v[1][y];
      const T* s = src + n1 * (y + (D == 3 ? n1 * z : 0));
#pragma unroll 2
      for (int x = 0; x < w[0].y; ++x) {
        const T f = wyz * v[0][x];
#pragma unroll
        for (int b = 0; b < MAXKP1; ++b)
          if (b < A.kin) acc[b] += f * s[b * A.vin + x];
      }
    }
  transfer_store(A, out, t, A.vout, acc);
}

// Up to kRun entries of a row from entry e0 on.  Rows with gaps (GAPS): FP32 takes the window and skips
// the zeros in it, FP64 the list of the entries, since every operation on its pipe counts.
constexpr int kRun = 8;
template <typename T, bool GAPS> struct RowRun { T c[kRun]; int off[kRun]; unsigned on; };
template <bool GAPS, typename T>
__device__ __forceinline__ RowRun<T, GAPS> row_run(const TransferArgs<T>& A, int g, bool has, int e0) {
  constexpr bool LIST = GAPS && sizeof(T) == 8;
  RowRun<T, GAPS> r;
  const int64_t row = (int64_t)g * A.width + e0;
  const int len = has ? (LIST ? A.cnt[g] : A.win[g].y) - e0 : 0;
  r.on = 0;
#pragma unroll
  for (int e = 0; e < kRun; ++e) {
    r.c[e] = e < len ? A.val[row + e] : (T)0;
    r.off[e] = LIST ? (e < len ? A.off[row + e] : 0) : e;
    if (e < len && (LIST || !GAPS || r.c[e] != (T)0)) r.on |= 1u << e;
  }
  return r;
}
// n: entries of the longest row from the run's first one on (the same for all threads).  e0: the run's first.
template <typename T, bool GAPS>
__device__ __forceinline__ T run_sum(const RowRun<T, GAPS>& r, int e0, int n, const T* s, int stride, T acc) {
  if (!(GAPS && sizeof(T) == 8)) s += e0 * stride;
  T t[kRun];
#pragma unroll
  for (int e = 0; e < kRun; ++e) t[e] = (r.on >> e) & 1u ? s[r.off[e] * stride] : (T)0;
#pragma unroll
  for (int e = 0; e < kRun; ++e) {
    if (sizeof(T) == 8 && e >= n) break;
    acc += r.c[e] * t[e];
  }
  return acc;
}

// Lines of the tile's input box, x -> y -> z: S1 [time node][z][y][TX] holds the sums along x, S2 (3D) [time
// node][z][TY][TX] those along y.  A thread keeps its x (and y) of the tile, so its weights stay in
// registers; the loads of an x sum are independent and straight from global memory (neighbouring sums
// share them through L1).  Bound by load latency up to 16^3 cells and by L1 and the FP64 pipe above.
template <typename T, int D, bool GAPS>
__global__ void __launch_bounds__(256) k_transfer_tile(const __grid_constant__ TransferArgs<T> A) {
  chain_begin();
  constexpr int TX = D == 3 ? kTile3[0] : kTile2[0], TY = D == 3 ? kTile3[1] : kTile2[1], TZ = D == 3 ? kTile3[2] : 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const T* in = A.in + blockIdx.y * A.zin;            // blockIdx.y: independent slot
  T* out = A.out + blockIdx.y * A.zout;
  const int tid = threadIdx.x, nt = blockDim.x;       // a multiple of TX * TY
  if (blockIdx.x >= A.nvb) {
    const int64_t i = (blockIdx.x - A.nvb) * (int64_t)nt + tid;
    if (i < A.total - A.nvel) transfer_pressure<T, D>(A, in, out, i);
    return;
  }
  unsigned b = blockIdx.x;
  const int x0 = (int)(b % (unsigned)A.tx) * TX; b /= (unsigned)A.tx;
  const int y0 = (int)(b % (unsigned)A.ty) * TY; b /= (unsigned)A.ty;
  const int z0 = D == 3 ? (int)(b % (unsigned)A.tz) * TZ : 0;
  const int c = D == 3 ? (int)(b / (unsigned)A.tz) : (int)b;
  // input lines of the tile along y and z
  int ylo = A.nin1, yhi = 0, zlo = D == 3 ? A.nin1 : 0, zhi = D == 3 ? 0 : 1;
#pragma unroll
  for (int j = 0; j < TY; ++j)
    if (y0 + j < A.nout1) { const int2 w = A.win[y0 + j]; ylo = min(ylo, w.x); yhi = max(yhi, w.x + w.y); }
  if (D == 3)
#pragma unroll
    for (int j = 0; j < TZ; ++j)
      if (z0 + j < A.nout1) { const int2 w = A.win[z0 + j]; zlo = min(zlo, w.x); zhi = max(zhi, w.x + w.y); }
  const int ny = yhi - ylo, nz = zhi - zlo;           // <= A.span
  T* S1 = reinterpret_cast<T*>(smem_raw);
  T* S2 = S1 + (size_t)A.kin * nz * ny * TX;
  const int ox = tid % TX, q0 = tid / TX, dq = nt / TX, oy = q0 % TY;
  const int64_t n1 = A.nin1;
  {
    const bool has = x0 + ox < A.nout1;
    const T* src = in + c * A.nin + (has ? A.win[x0 + ox].x : 0) + n1 * (ylo + n1 * zlo);
    const int lines = A.kin * nz * ny;
    for (int e = 0; e < A.width; e += kRun) {         // (one pass for windows of up to kRun entries)
      const auto r = row_run<GAPS>(A, x0 + ox, has, e);
      for (int q = q0; q < lines; q += dq) {
        const unsigned t = (unsigned)q / (unsigned)ny, y = q - t * ny;
        const unsigned a = D == 3 ? t / (unsigned)nz : t, z = D == 3 ? t - a * nz : 0;
        S1[q * TX + ox] = run_sum(r, e, A.width - e, src + a * A.vin + n1 * (y + n1 * z), 1, e ? S1[q * TX + ox] : (T)0);
      }
    }
  }
  __syncthreads();
  const bool hasy = y0 + oy < A.nout1;
  const int yo = hasy ? A.win[y0 + oy].x - ylo : 0;
  T acc[MAXKP1];
#pragma unroll
  for (int a = 0; a < MAXKP1; ++a) acc[a] = 0;
  const int oz = q0 / TY;
  if constexpr (D == 3) {
    const T* s1 = S1 + yo * TX + ox;
    for (int e = 0; e < A.width; e += kRun) {
      const auto r = row_run<GAPS>(A, y0 + oy, hasy, e);
      for (int q = oz; q < A.kin * nz; q += dq / TY) {
        T* o = S2 + (q * TY + oy) * TX + ox;
        *o = run_sum(r, e, A.width - e, s1 + q * ny * TX, TX, e ? *o : (T)0);
      }
    }
    __syncthreads();
    if (oz >= TZ || z0 + oz >= A.nout1) return;
    const T* s2 = S2 + ((A.win[z0 + oz].x - zlo) * TY + oy) * TX + ox;
    for (int e = 0; e < A.width; e += kRun) {
      const auto r = row_run<GAPS>(A, z0 + oz, true, e);
#pragma unroll
      for (int a = 0; a < MAXKP1; ++a)
        if (a < A.kin) acc[a] = run_sum(r, e, A.width - e, s2 + a * nz * TY * TX, TY * TX, acc[a]);
    }
  } else {
    if (oz >= 1) return;
    const T* s1 = S1 + yo * TX + ox;
    for (int e = 0; e < A.width; e += kRun) {
      const auto r = row_run<GAPS>(A, y0 + oy, hasy, e);
#pragma unroll
      for (int a = 0; a < MAXKP1; ++a)
        if (a < A.kin) acc[a] = run_sum(r, e, A.width - e, s1 + a * ny * TX, TX, acc[a]);
    }
  }
  if (x0 + ox >= A.nout1 || !hasy) return;
  const int64_t m1 = A.nout1;
  transfer_store(A, out, c * A.nout + x0 + ox + m1 * (y0 + oy + (D == 3 ? m1 * (z0 + oz) : 0)), A.vout, acc);
}

template <typename T> static const T* vals(const Line1D& c);
template <> const double* vals<double>(const Line1D& c) { return c.val64; }
template <> const float* vals<float>(const Line1D& c) { return c.val32; }
template <typename T> static const T* ptab(const Transfer& t);
template <> const double* ptab<double>(const Transfer& t) { return t.PT64; }
template <> const float* ptab<float>(const Transfer& t) { return t.PT32; }

// 256 threads where the tile's input box is larger than the tile (restriction, interpolation), else 128.
template <typename T>
static cudaError_t launch_tile(TransferArgs<T>& A, const Line1D& op, int d, cudaStream_t s, int slots) {
  const int* tile = d == 3 ? kTile3 : kTile2;
  const auto tiles = [&](int t) { return (A.nout1 + t - 1) / t; };
  A.span = op.span;
  A.tx = tiles(tile[0]); A.ty = tiles(tile[1]); A.tz = d == 3 ? tiles(tile[2]) : 1;
  A.nvb = (int64_t)A.tx * A.ty * A.tz * d;
  const int threads = A.nin1 > A.nout1 ? 256 : 128;
  const int64_t blocks = A.nvb + (A.total - A.nvel + threads - 1) / threads;
  const size_t lines = d == 3 ? (size_t)op.span * (op.span + tile[1]) : op.span;
  const size_t smem = sizeof(T) * A.kin * tile[0] * lines;
  auto kern = d == 3 ? (op.gaps ? k_transfer_tile<T, 3, true> : k_transfer_tile<T, 3, false>) : k_transfer_tile<T, 2, true>;
  if constexpr (sizeof(T) == 8)                       // (2D FP32: rows with gaps only, see transfer_launch)
    if (d == 2 && !op.gaps) kern = k_transfer_tile<T, 2, false>;
  if (smem > 48 * 1024) {
    cudaError_t e = allow_smem(kern, smem);
    if (e != cudaSuccess) return e;
  }
  launch_chained(kern, dim3((unsigned)blocks, (unsigned)slots), threads, smem, s, A);
  note_launch();
  return cudaGetLastError();
}

// in on level li -> out on level lo through the 1D operator op and the time matrix M [lo.k+1][li.k+1].
template <typename T>
static cudaError_t transfer_launch(const Transfer& tr, const Line1D& op, const Level& li, const Level& lo,
                                   const double (*M)[MAXKP1], bool transposed, int pop, bool add, const T* in, T* out,
                                   cudaStream_t s, int slots) {
  TransferArgs<T> A{};
  A.in = in; A.out = out;
  A.win = op.win; A.cnt = op.cnt; A.off = op.off; A.val = vals<T>(op);
  A.width = sizeof(T) == 8 ? op.entries : op.width;
  A.nin1 = li.N1; A.nout1 = lo.N1; A.kin = li.k + 1; A.kout = lo.k + 1; A.add = add;
  A.nin = li.nnodes; A.nout = lo.nnodes; A.vin = li.Nv; A.vout = lo.Nv;
  A.nvel = lo.Nv;
  A.total = lo.Nv + (pop != P_NONE ? lo.Np : 0);
  for (int a = 0; a <= lo.k; ++a)
    for (int b = 0; b <= li.k; ++b) A.M.m[a][b] = (T)(transposed ? M[b][a] : M[a][b]);
  A.mix = lo.k != li.k;                               // one time basis: M is the identity
  A.pop = pop; A.nf = tr.fine->n; A.ratio = tr.ratio; A.npf = tr.fine->npc; A.npc = tr.coarse->npc;
  A.PT = ptab<T>(tr);
  A.pin = li.Np; A.pout = lo.Np; A.zin = li.Nst; A.zout = lo.Nst;
  // Tiles for everything but injections (k_transfer reads and writes each entry once: 3D 64^3 DG(2) -> DG(1)
  // 80 us against 285 us axis by axis through memory) and 2D FP32 rows without gaps (at most 9 or 16 cheap
  // products; 2D 256^2 Q3/P2 DG(2) state interpolation 12.5 us, as tiles 18.1, prolongation 22 and 24).  Before,
  // one launch per axis, time and pressure -> k_transfer -> tiles, in a graph: FP64 3D 32^3 -> 16^3 Q2/P1 DG(1)
  // restriction 49 -> 389 -> 44 us, prolongation 49 -> 117 -> 32; FP64 3D 32^3 Q3/P2 -> Q2/P1 DG(1) 145 -> 500
  // -> 123 and 136 -> 422 -> 118; FP64 2D 256^2 -> 128^2 restriction 35 -> 61 -> 20; FP32 3D 16^3 -> 8^3 restriction
  // 19 -> 31 -> 5.6; FP32 2D 32^2 -> 16^2 13.5 -> 5.9 -> 3.1.  Slower than axis by axis: FP64 3D 16^3 Q4/P3 DG(2)
  // restriction 48 -> 51, FP64 2D 256^2 Q3/P2 DG(2) state interpolation 45 -> 51.
  if (op.width > 1 && (li.d == 3 || sizeof(T) == 8 || op.gaps)) return launch_tile(A, op, li.d, s, slots);
  const dim3 grid((unsigned)((A.total + 127) / 128), (unsigned)slots);
  if (li.d == 2) launch_chained(k_transfer<T, 2>, grid, 128, 0, s, A);
  else launch_chained(k_transfer<T, 3>, grid, 128, 0, s, A);
  note_launch();
  return cudaGetLastError();
}

template <typename T>
cudaError_t Transfer::prolong(const T* xc, T* xf, cudaStream_t s, int slots, bool add) const {
  return transfer_launch<T>(*this, P1, *coarse, *fine, E, false, P_PROLONG, add, xc, xf, s, slots);
}

template <typename T>
cudaError_t Transfer::restrict_(const T* xf, T* xc, cudaStream_t s, int slots) const {
  return transfer_launch<T>(*this, P1T, *fine, *coarse, E, true, P_RESTRICT, false, xf, xc, s, slots);
}

template <typename T>
cudaError_t Transfer::interp_state(const T* Vf, T* Vc, cudaStream_t s) const {
  return transfer_launch<T>(*this, I1, *fine, *coarse, Et, false, P_NONE, false, Vf, Vc, s, 1);
}

template cudaError_t Transfer::prolong<float>(const float*, float*, cudaStream_t, int, bool) const;
template cudaError_t Transfer::prolong<double>(const double*, double*, cudaStream_t, int, bool) const;
template cudaError_t Transfer::restrict_<float>(const float*, float*, cudaStream_t, int) const;
template cudaError_t Transfer::restrict_<double>(const double*, double*, cudaStream_t, int) const;
template cudaError_t Transfer::interp_state<float>(const float*, float*, cudaStream_t) const;
template cudaError_t Transfer::interp_state<double>(const double*, double*, cudaStream_t) const;

}  // namespace stmg
