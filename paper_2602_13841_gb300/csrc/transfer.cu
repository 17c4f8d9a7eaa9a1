// Grid transfer kernels and their host set-up (see transfer.hpp).
#include <algorithm>
#include <cmath>
#include <vector>

#include "handle.hpp"
#include "transfer.hpp"
#include "chain.cuh"
#include "counters.hpp"

namespace stmg {

// ---------------------------------------------------------------------------- host set-up
// The rows of a 1D operator as contiguous windows of columns.
static Line1D upload_lines(Handle* h, int rows, int cols, const std::vector<std::vector<std::pair<int, double>>>& R) {
  Line1D c;
  c.rows = rows; c.cols = cols;
  std::vector<int2> win(rows);
  for (int i = 0; i < rows; ++i) {
    int lo = cols, hi = -1;
    for (auto& e : R[i]) { lo = std::min(lo, e.first); hi = std::max(hi, e.first); }
    if (hi < 0) { lo = 0; hi = 0; }
    win[i] = make_int2(lo, hi - lo + 1);
    c.width = std::max(c.width, hi - lo + 1);
  }
  std::vector<double> v((size_t)rows * c.width, 0.0);
  for (int i = 0; i < rows; ++i)
    for (auto& e : R[i]) v[(size_t)i * c.width + e.first - win[i].x] += e.second;
  std::vector<float> v32(v.begin(), v.end());
  c.win = (int2*)h->dalloc(win.size() * sizeof(int2));
  c.val64 = (double*)h->dalloc(v.size() * sizeof(double));
  c.val32 = (float*)h->dalloc(v.size() * sizeof(float));
  h->upload(c.win, win.data(), win.size() * sizeof(int2));
  h->upload(c.val64, v.data(), v.size() * sizeof(double));
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
// to out where `add`.  A thread owns one output node and component: it sums the product of its D row
// windows for every input time node and mixes the sums in time, so that nothing passes through memory
// between axes, time and pressure (five launches before, six with the correction's update).  A window
// holds up to 7 entries, so a 3D restriction reads up to 343 neighbouring values per input; those of
// neighbouring threads coincide and stay in L1.  Bound by launch and load latency on the small levels
// that most transfers are for: 5.8 us a launch on the levels of a 2D 32^2 solve, against chains of five
// and six launches of 3 us each.
template <typename T> struct MatT { T m[MAXKP1][MAXKP1]; };
enum { P_NONE = 0, P_PROLONG = 1, P_RESTRICT = 2 };

template <typename T>
struct TransferArgs {
  const T* in;
  T* out;
  const int2* win;
  const T* val;
  int width, nin1, nout1, kin, kout, add;
  int64_t nin, nout, vin, vout;                       // nodes and velocity entries per time node
  int64_t nvel, total;                                // threads for the velocity, and with the pressure
  MatT<T> M;
  int pop, nf, ratio, npf, npc;                       // pressure: kind, fine cells per axis, modes fine / coarse
  const T* PT;
  int64_t pin, pout, zin, zout;                       // pressure entries per time node; slot strides
};

template <typename T, int D>
__global__ void k_transfer(const __grid_constant__ TransferArgs<T> A) {
  chain_begin();
  const T* in = A.in + blockIdx.y * A.zin;            // blockIdx.y: independent slot
  T* out = A.out + blockIdx.y * A.zout;
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= A.total) return;
  T acc[MAXKP1];
#pragma unroll
  for (int b = 0; b < MAXKP1; ++b) acc[b] = 0;
  int64_t o, so;                                      // output entry and its stride between time nodes
  if (t < A.nvel) {
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
          if (f == (T)0) continue;                    // a gap in the row: its entry does not count, whatever it is
#pragma unroll
          for (int b = 0; b < MAXKP1; ++b)
            if (b < A.kin) acc[b] += f * s[b * A.vin + x];
        }
      }
    o = t;
    so = A.vout;
  } else {
    const int64_t i = t - A.nvel;
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
    o = A.kout * A.vout + i;
    so = A.pout;
  }
#pragma unroll
  for (int a = 0; a < MAXKP1; ++a) {
    if (a >= A.kout) break;
    T r = 0;
#pragma unroll
    for (int b = 0; b < MAXKP1; ++b)
      if (b < A.kin) r += A.M.m[a][b] * acc[b];
    out[o + a * so] = A.add ? out[o + a * so] + r : r;
  }
}

template <typename T> static const T* vals(const Line1D& c);
template <> const double* vals<double>(const Line1D& c) { return c.val64; }
template <> const float* vals<float>(const Line1D& c) { return c.val32; }
template <typename T> static const T* ptab(const Transfer& t);
template <> const double* ptab<double>(const Transfer& t) { return t.PT64; }
template <> const float* ptab<float>(const Transfer& t) { return t.PT32; }

// in on level li -> out on level lo through the 1D operator op and the time matrix M [lo.k+1][li.k+1].
template <typename T>
static cudaError_t transfer_launch(const Transfer& tr, const Line1D& op, const Level& li, const Level& lo,
                                   const double (*M)[MAXKP1], bool transposed, int pop, bool add, const T* in, T* out,
                                   cudaStream_t s, int slots) {
  TransferArgs<T> A{};
  A.in = in; A.out = out;
  A.win = op.win; A.val = vals<T>(op); A.width = op.width;
  A.nin1 = li.N1; A.nout1 = lo.N1; A.kin = li.k + 1; A.kout = lo.k + 1; A.add = add;
  A.nin = li.nnodes; A.nout = lo.nnodes; A.vin = li.Nv; A.vout = lo.Nv;
  A.nvel = lo.Nv;
  A.total = lo.Nv + (pop != P_NONE ? lo.Np : 0);
  for (int a = 0; a <= lo.k; ++a)
    for (int b = 0; b <= li.k; ++b) A.M.m[a][b] = (T)(transposed ? M[b][a] : M[a][b]);
  A.pop = pop; A.nf = tr.fine->n; A.ratio = tr.ratio; A.npf = tr.fine->npc; A.npc = tr.coarse->npc;
  A.PT = ptab<T>(tr);
  A.pin = li.Np; A.pout = lo.Np; A.zin = li.Nst; A.zout = lo.Nst;
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
