// Exact local solves of the FP64 RAS smoother (Section 4.2) in 64-bit fixed
// point; in 2D with the residual of the step formed in the same kernel.
//
// On a level whose stencil is the Q1 Laplacian / d (checked at setup), a
// box's local matrix R_i Z_k R_i^T is (1/d) sum_i (x)_ax {K_l if ax = i else
// M_l} with the 1D Dirichlet matrices K_l = (1/h) tridiag(-1, 2, -1) and
// M_l = (h/6) tridiag(1, 4, 1) of the box extents l, both diagonalised by the
// orthonormal sine matrix S_l. The exact solve (A_k)_i^{-1} r is then: S
// along every axis but x, one tridiagonal solve per line along x (elimination
// factors precomputed), S back.
//
// What bounds it. In FP64 the solve is bound by FP64 issue (2 lanes per
// clock per SM): about 2,450 FP64 instructions per 12 x 12 box. The box data
// therefore goes to fixed point (fix64.cuh), where a multiply-add costs three
// integer multiply-adds on a pipe 32 times as wide; what is left is integer
// issue (ALU pipe 57% busy: conversions, 64-bit additions and shifts beside
// the multiply-adds) and the load phase. Measured per launch: 2D 1024^2, 8 x 8
// cores with overlap 2: 85.8 + 17.4 us (solve and residual kernels in FP64)
// -> 49.4 us, residual included, 41.8 us from a zero iterate; 3D 128^3, 4^3
// cores with overlap 1: 270 us -> 99 us, after a residual kernel of 54 us.
//
// Precision. All values of a box share one exponent, so errors are relative
// to the largest entry of the box, whose bits are (FP64: 53):
//   right-hand side alone, step from zero and 3D: 58 (4 x 4 boxes), 57 (6 x 6),
//   56 (8 to 12), 55 (16 x 16); 3D 56 (4^3, some mesh sizes 57), 55 (6^3, 56);
//   residual formed here (2D): 1.6 to 0.6 bits fewer, from z and f with 58.
// The residual is small against z near convergence, so quantising it against
// the exponent of z would lose what FP64 keeps. In 2D it is therefore formed
// exactly from z and f (entries within 2^5 of the largest lose nothing) and
// gets an exponent of its own before the solve. 3D coefficients are no small
// integers, and quantised at 56 bits a large entry over small noise left ten
// times the error of FP64; there the residual comes from the FP64 kernel of
// mg.cu, which also is the faster form on large grids (166 us against 99 + 54
// at 128^3; below 48^3 a W-cycle takes up to 11% longer for the launch).
// Error of a step against extended precision over the largest entry, FP64
// kernels -> here: random data 1.8e-15 -> 1.8e-16 (12 x 12), 6.4e-16 -> 2.8e-16
// (6^3); smooth z with f = Z z 1.9e-15 -> 1.7e-18, 2.1e-15 -> 1.6e-15; z falling
// by e^1/2 per node 9.2e-17 -> 5.9e-17, 3.7e-16 -> 2.6e-16.
//
// Scaling. The scaled operator A / hs, hs = 1 in 2D and the power of two next
// below h in 3D, has entries of order one whatever the level. The host
// chooses the bits from the row sums of the tables so that no intermediate
// value can leave the range of fix64.cuh: fold of two entries, transform
// |S|_inf, forward elimination, and the inverse line operators ||T_j^-1||_inf,
// which a transformed line j may grow by. In 2D line j is stored in units of
// 2^K_j, K_j = ceil log2 ||T_j^-1||_inf, and the transform back multiplies
// by S 2^(K_j - kout); in 3D the growth is small and one K serves all. A box
// with a non-finite entry returns NaN everywhere.
//
// Mapping. A CTA takes one work item (boxes of one class). In 2D a box belongs
// to a group of 8, 16 or 32 lanes, one per column of the box and its halo: a
// lane loads its column of z and f into registers (every load of the box in
// flight together), the box maximum and the neighbouring columns come by
// shuffles, the y transform runs down the lane's own column, the x line solve
// takes one row per lane, and only the two transpositions between them go
// through shared memory; no barrier wider than a warp. In 3D a box has one
// thread per column along z and every phase gives each thread one grid line.
// Rows are padded to an odd pitch (conflict-free 8-byte accesses).
// A transform folds its line by the symmetry S[j][l-1-x] = (-1)^j S[j][x] (on
// the inputs forward, on the outputs back): l^2 / 2 multiply-adds. Short
// lines of a class are padded by zero table entries up to the compile-time
// LM. Results go to y box-major (y[item][b][i]).
#include "common.cuh"
#include "ras_fix.cuh"

#include <algorithm>
#include <cmath>
#include <map>
#include <memory>
#include <utility>

namespace dcg {
namespace {

struct FixArgs {
  const int* work;           // [nwork*3]: class, first index into class_patches, count
  const int* class_patches;
  const RasClass* classes;
  const int4* origin;        // [npatch] box origin (x, y, z) and its node index
  const long long* item_off; // [nwork]
  const int2* tab;
  int m;
  FxScale sc;
};

// EX: the boxes have extent LM along every axis
template <int LM, bool ZZERO, bool EX>
__device__ __forceinline__ void fx_boxes_2d(const FixArgs& A, const RasClass& C, const int2* s_tab, long long* smem,
                                            int first, int cnt, const double* __restrict__ f,
                                            const double* __restrict__ z, double* __restrict__ yi) {
  constexpr int G = fx_group(LM), HP = fx_hm(LM), NF = LM * HP;
  const int lane = threadIdx.x & (G - 1), b = threadIdx.x / G;
  const int lx = EX ? LM : C.len[0], ly = EX ? LM : C.len[1], m = A.m;
  const bool live = b < cnt;                 // groups past the item's boxes only take part in the shuffles
  const int x = lane - 1;                    // column of the box, -1 and lx are its halo
  const bool own = live && x >= 0 && x < lx;
  const int4 og = live ? __ldg(A.origin + __ldg(A.class_patches + first + b)) : make_int4(0, 0, 0, 0);
  long long zv[LM + 2], fv[LM];
  {
    const int gx = og.x + x;
    const bool col = live && !ZZERO && x <= lx && gx >= 0 && gx < m;
    const int base = gx + m * (og.y - 1);
#pragma unroll
    for (int q = 0; q < LM + 2; ++q) {
      const int gy = og.y - 1 + q;
      // rows 1 .. ly of the halo lie in the box and so in the grid
      zv[q] = (col && q <= ly + 1 && (EX && q >= 1 && q <= LM ? true : gy >= 0 && gy < m)) ? __double_as_longlong(__ldg(z + base + q * m)) : 0;
    }
#pragma unroll
    for (int q = 0; q < LM; ++q)
      fv[q] = (own && q < ly) ? __double_as_longlong(__ldg(f + base + (q + 1) * m)) : 0;
  }
  double* yb = yi + b * (lx * ly) + x;
  fx_solve_2d<LM, ZZERO, EX, true>(A.sc, lx, ly, live, zv, fv, smem + b * (ly * (lx | 1)), s_tab, s_tab + NF,
                             A.tab + C.fx_tri, [&](int q, double v) { yb[q * lx] = v; });
}

// y = the boxes' solves of the right-hand side f
template <int LM, bool EX>
__device__ __forceinline__ void fx_boxes_3d(const FixArgs& A, const RasClass& C, const int2* s_tab, long long* smem, unsigned* s_e,
                                            int first, int cnt, const double* __restrict__ f,
                                            double* __restrict__ yi) {
  constexpr int TPB = LM * LM, HP = fx_hm(LM), HM = (LM + 1) / 2, NF = LM * HP, NBK = 2 * HM * HP;
  const int b = threadIdx.x / TPB, c = threadIdx.x - b * TPB;
  const int cy = c / LM, cx = c - cy * LM;
  const int lx = EX ? LM : C.len[0], ly = EX ? LM : C.len[1], lz = EX ? LM : C.len[2], m = A.m;
  const int wp = lx | 1;
  long long* W = smem + b * (wp * ly * lz);  // [lz][ly][wp]
  const bool live = b < cnt;
  const bool own = live && cx < lx && cy < ly;
  const int4 og = live ? __ldg(A.origin + __ldg(A.class_patches + first + b)) : make_int4(0, 0, 0, 0);
  if (c == 0) s_e[b] = 0;
  __syncthreads();
  const int mm = m * m;
  long long fv[LM];
  unsigned mag = 0;
  const int base = (og.x + cx) + m * (og.y + cy) + mm * og.z;
#pragma unroll
  for (int q = 0; q < LM; ++q) {
    fv[q] = (own && q < lz) ? __double_as_longlong(__ldg(f + base + q * mm)) : 0;
    mag = max(mag, fx_mag(fv[q]));
  }
  if (live && mag) atomicMax(&s_e[b], mag);
  __syncthreads();
  mag = s_e[b];
  const bool odd = fx_odd(mag);
  int e = (int)(mag >> 20);
  if (odd) {
    const int lift = fx_lift(mag);
    const double up = fx_two320(lift);
    e = fx_odd_exponent(mag, lift);
#pragma unroll
    for (int q = 0; q < LM; ++q) fv[q] = fx_scaled(fv[q], up);
  }
  const int sh0 = 63 - A.sc.bits + e;
#pragma unroll
  for (int q = 0; q < LM; ++q)
    if (own && q < lz) W[(q * ly + cy) * wp + cx] = fx_near(fv[q], sh0);
  // column (cx, cy) along z; then line (cx, k = cy) along y; then line (j =
  // cx, k = cy) along x
  if (own) fx_forward<LM>(W + cy * wp + cx, ly * wp, lz, s_tab + NF + NBK);
  __syncthreads();
  const bool yline = live && cx < lx && cy < lz;
  if (yline) fx_forward<LM>(W + cy * ly * wp + cx, wp, ly, s_tab);
  __syncthreads();
  if (live && cx < ly && cy < lz)
    fx_line_solve<LM, EX>(W + (cy * ly + cx) * wp, lx, A.tab + C.fx_tri + cy * ly + cx, ly * lz);
  __syncthreads();
  if (yline) fx_back<LM>(W + cy * ly * wp + cx, wp, ly, s_tab + NF);
  __syncthreads();
  if (own) {
    fx_back<LM>(W + cy * wp + cx, ly * wp, lz, s_tab + NF + NBK + NF);
    const int e0 = e + A.sc.sf + 63 - A.sc.bits + A.sc.kout;
    double* yb = yi + b * (lx * ly * lz) + cy * lx + cx;
    if (!odd) {
#pragma unroll 2
      for (int q = 0; q < lz; ++q) yb[q * lx * ly] = fx_to_double(W[(q * ly + cy) * wp + cx], e0);
    } else {
      for (int q = 0; q < lz; ++q) yb[q * lx * ly] = fx_special(W[(q * ly + cy) * wp + cx], e0, mag);
    }
  }
}

template <int D, int LM, bool ZZERO>
__global__ void __launch_bounds__(fx_threads(D, LM), fx_blocks(D, LM))
    k_ras_fix(FixArgs A, const double* __restrict__ f, const double* __restrict__ z, double* __restrict__ y) {
  constexpr int HP = fx_hm(LM), HM = (LM + 1) / 2;
  constexpr int NF = LM * HP, NBK = 2 * HM * HP;  // forward / back table entries per axis
  extern __shared__ __align__(16) unsigned char fx_smem[];
  __shared__ __align__(16) int2 s_tab[(D - 1) * (NF + NBK)];
  __shared__ unsigned s_e[fx_batch(D, LM)];
  const int w = blockIdx.x;
  const int cls = A.work[3 * w], first = A.work[3 * w + 1], cnt = A.work[3 * w + 2];
  const RasClass& C = A.classes[cls];
  for (int t = threadIdx.x; t < (D - 1) * (NF + NBK); t += fx_threads(D, LM)) {
    const int ax = t / (NF + NBK), i = t - ax * (NF + NBK);
    s_tab[t] = __ldg(A.tab + (i < NF ? C.fx_f[ax] + i : C.fx_b[ax] + i - NF));
  }
  __syncthreads();
  long long* smem = reinterpret_cast<long long*>(fx_smem);
  double* yi = y + A.item_off[w];
  const bool exact = C.len[0] == LM && C.len[1] == LM && (D == 2 || C.len[2] == LM);  // the interior class
  if constexpr (D == 2) {
    if (exact) fx_boxes_2d<LM, ZZERO, true>(A, C, s_tab, smem, first, cnt, f, z, yi);
    else fx_boxes_2d<LM, ZZERO, false>(A, C, s_tab, smem, first, cnt, f, z, yi);
  } else {
    if (exact) fx_boxes_3d<LM, true>(A, C, s_tab, smem, s_e, first, cnt, f, yi);
    else fx_boxes_3d<LM, false>(A, C, s_tab, smem, s_e, first, cnt, f, yi);
  }
}

// Double-double numbers (sums of two doubles, about 104 bits, by Dekker's and
// Knuth's error-free sum and product). The tables are formed in them because
// long double is software on Arm (3D, 4^3 cores: 645 us per level with it, a
// third of the set-up at 16^3).
struct Dd {
  double h, l;
};
// (a call of its own: its operands have to be rounded before they are added,
// and compilers for Arm fuse an inlined product into the addition)
__attribute__((noinline)) Dd dd_sum(double a, double b) {
  const double s = a + b, t = s - a;
  return Dd{s, (a - (s - t)) + (b - t)};
}
Dd operator+(Dd a, Dd b) {
  const Dd s = dd_sum(a.h, b.h);
  return dd_sum(s.h, s.l + (a.l + b.l));
}
Dd operator-(Dd a) { return Dd{-a.h, -a.l}; }
Dd operator-(Dd a, Dd b) { return a + -b; }
Dd operator*(Dd a, Dd b) {
  const double p = a.h * b.h;
  return dd_sum(p, std::fma(a.h, b.h, -p) + std::fma(a.h, b.l, a.l * b.h));
}
Dd dd_inverse(Dd a) {
  const double q = 1.0 / a.h;
  const Dd r = Dd{1.0, 0.0} - a * Dd{q, 0.0};
  return dd_sum(q, q * (r.h + r.l));
}
Dd operator/(Dd a, double b) { return a * dd_inverse(Dd{b, 0.0}); }
Dd dd_root(double x) {  // of x > 0: one Newton step
  const double y = std::sqrt(x);
  return dd_sum(y, std::fma(-y, y, x) / (2.0 * y));
}
// sine and cosine of 0 < x <= pi / 4 by their series
void dd_sincos(Dd x, Dd* sn, Dd* cs) {
  const Dd x2 = -(x * x);
  Dd t{1.0, 0.0}, s{0.0, 0.0}, c{0.0, 0.0};
  for (int k = 1; std::fabs(t.h) > 1e-34; ++k) {  // t = (-1)^(k-1) x^(2k-2) / (2k - 2)!
    c = c + t;
    const Dd u = t / (2.0 * k - 1.0);
    s = s + u;
    t = u * x2 / (2.0 * k);
  }
  *sn = s * x;
  *cs = c;
}
// round(c 2^58)
long long fx_const_bits(Dd c) {
  const double v = std::nearbyint(c.h * 0x1p58);
  return (long long)v + (long long)std::nearbyint(std::fma(c.h, 0x1p58, -v) + c.l * 0x1p58);
}
// the constant C 2^-58 2^shift as the pair fx_mac takes
int2 fx_const(long long C, int shift = 0) {
  const long long v = shift >= 0 ? C << shift : (C + (1LL << (-shift - 1))) >> -shift;
  const long long lo = ((v + (1LL << 28)) & ((1LL << 29) - 1)) - (1LL << 28);  // in [-2^28, 2^28)
  return make_int2((int)((v - lo) >> 29), (int)lo);
}

template <int D, int LM>
size_t fx_smem(const Level& L) {
  size_t mx = 0;
  for (const auto& c : L.classes)
    mx = std::max(mx, sizeof(long long) * (size_t)c.nb * (c.len[0] | 1) * c.len[1] * (D > 2 ? c.len[2] : 1));
  return mx;
}
// below the 48 KB that need no limit to be raised: a limit belongs to the
// kernel and would be shared by every problem
template <int D, int LM>
constexpr bool fx_smem_fits() {
  constexpr int tab = (D - 1) * (LM + (LM + 1) / 2 * 2) * fx_hm(LM);
  return 8 * (fx_batch(D, LM) * (LM | 1) * LM * (D > 2 ? LM : 1) + tab) + 4 * fx_batch(D, LM) <= 48 * 1024;
}

// y = solves of f - Z z on the boxes (z null: of f; 3D: z null)
template <int D, int LM>
void fx_launch(const Level& L, const FixArgs& a, const double* f, const double* z, cudaStream_t s) {
  static_assert(fx_smem_fits<D, LM>(), "");
  const size_t smem = fx_smem<D, LM>(L);
  constexpr int nt = fx_threads(D, LM);
  if constexpr (D == 2) {
    if (z) {
      k_ras_fix<D, LM, false><<<L.nwork, nt, smem, s>>>(a, f, z, (double*)L.y);
      return;
    }
  }
  k_ras_fix<D, LM, true><<<L.nwork, nt, smem, s>>>(a, f, nullptr, (double*)L.y);
}

// compile-time extent that serves a level's largest box extent
int fx_lm(int dim, int lmax) {
  if (dim == 3) return lmax <= 4 ? 4 : 6;
  return lmax <= 4 ? 4 : lmax <= 6 ? 6 : lmax <= 8 ? 8 : lmax <= 10 ? 10 : lmax <= 12 ? 12 : 16;
}

}  // namespace

int ras_fix_lm(int dim, int lmax) { return fx_lm(dim, lmax); }
int ras_fix_batch(int dim, int lmax) { return fx_batch(dim, fx_lm(dim, lmax)); }

// What the levels of one hierarchy share while it is set up
struct FixExtent {
  std::vector<Dd> kap, mu;     // 1D eigenvalues at h = 1
  std::vector<long long> S;    // sine matrix
  double row = 0.0, mx = 0.0;  // largest absolute row sum and entry of S
};
// Line systems along x after the transforms along y (j) and z (k), system
// j + ly k: the tridiagonal Toeplitz part of A', the same for every extent
// along x (a shorter line takes the first of `rows` factors). Per row i: -l_i,
// winv_i, -b winv_i; and for lines of `rows` the reciprocal pivot of the row
// that meets an equal elimination of half of them from the other end.
struct FixLines {
  std::vector<long long> l, w, bw, meet;  // meet: one per system
  std::vector<double> ld, wd, b;          // |l_i|, winv_i; |b| per system
};
struct FixTables {
  double rho = 0.0;  // the lines' scale
  std::map<int, FixExtent> ext;
  std::map<std::pair<int, int>, FixLines> lines;
};
std::shared_ptr<FixTables> ras_fix_tables() { return std::make_shared<FixTables>(); }

namespace {
// sines and cosines of pi k / (2 N), N = l + 1, by the rotation from k to k + 1
FixExtent fix_extent(int l) {
  const int N = l + 1;
  const Dd pi{3.141592653589793116, 1.2246467991473531772e-16}, nrm = dd_inverse(dd_root(N / 2.0));
  std::vector<Dd> q(N + 1, Dd{0.0, 0.0});
  Dd s1, c1, c{1.0, 0.0};
  dd_sincos(pi / (2.0 * N), &s1, &c1);
  for (int k = 0; k < N; ++k) {
    q[k + 1] = q[k] * c1 + c * s1;
    c = c * c1 - q[k] * s1;
  }
  FixExtent e;
  std::vector<long long> sn(N, 0);
  for (int j = 1; j < N; ++j) sn[j] = fx_const_bits(nrm * q[2 * j <= N ? 2 * j : 2 * N - 2 * j]);
  e.S.resize((size_t)l * l);
  for (int j = 0; j < l; ++j) {
    double t = 0.0;
    for (int x = 0; x < l; ++x) {
      const int a = ((j + 1) * (x + 1)) % (2 * N);
      const long long v = a <= l ? sn[a] : a == N ? 0 : -sn[a - N];
      e.S[(size_t)j * l + x] = v;
      const double av = std::fabs((double)v * 0x1p-58);
      t += av;
      e.mx = std::max(e.mx, av);
    }
    e.row = std::max(e.row, t);
    const int k = 2 * (j + 1);
    const Dd cs = k <= N ? q[N - k] : -q[k - N], d = Dd{1.0, 0.0} - cs;
    e.kap.push_back(d + d);
    e.mu.push_back((Dd{2.0, 0.0} + cs) / 3.0);
  }
  return e;
}

FixLines fix_lines(int D, const FixExtent& ey, const FixExtent& ez, int ly, int lz, int rows, Dd rho) {
  FixLines v;
  const int nsys = ly * lz;
  v.l.resize((size_t)nsys * rows);
  v.w = v.bw = v.l;
  v.ld.resize((size_t)nsys * rows);
  v.wd = v.ld;
  v.meet.resize(nsys);
  v.b.resize(nsys);
  for (int sys = 0; sys < nsys; ++sys) {
    const int j = sys % ly, k = sys / ly;
    const Dd cm = D == 2 ? ey.kap[j] / 2.0 : (ey.kap[j] * ez.mu[k] + ey.mu[j] * ez.kap[k]) / 3.0;
    const Dd ck = D == 2 ? ey.mu[j] / 2.0 : ey.mu[j] * ez.mu[k] / 3.0;
    const Dd a = rho * (cm / 1.5 + ck + ck), bb = rho * (cm / 6.0 - ck);
    v.b[sys] = std::fabs(bb.h);
    Dd wi{0.0, 0.0};  // reciprocal pivot
    for (int i = 0; i < rows; ++i) {
      const size_t at = (size_t)sys * rows + i;
      const Dd li = bb * wi, w = a - li * bb;
      wi = dd_inverse(w);
      const Dd bw = bb * wi;
      v.l[at] = fx_const_bits(-li);
      v.w[at] = fx_const_bits(wi);
      v.bw[at] = fx_const_bits(-bw);
      v.ld[at] = std::fabs(li.h);
      v.wd[at] = wi.h;
      if (i == rows / 2 - 1) v.meet[sys] = fx_const_bits(dd_inverse(w - bb * bw));
    }
  }
  return v;
}

// ||T^-1||_inf of a line of n rows: |T^-1| is the inverse with off-diagonals
// -|b|, and its row sums solve that system for a right-hand side of ones;
// *grow: bound of the forward sweep for |g| <= 1
double fix_line_norm(const double* ld, const double* wd, double b, int n, double* grow) {
  double v[16], u = 0.0, norm = 0.0;
  for (int i = 0; i < n; ++i) {
    v[i] = u = 1.0 + ld[i] * u;
    *grow = std::max(*grow, u);
  }
  for (int i = n - 1; i >= 0; --i) {
    v[i] = (v[i] + (i + 1 < n ? b * v[i + 1] : 0.0)) * wd[i];
    norm = std::max(norm, v[i]);
  }
  return norm;
}
}  // namespace

// Tables of a level's box classes and its quantisation (see the file header).
// `shared`: what the hierarchy's other levels have formed already.
int ras_fix_setup(dcg_problem* p, Level& L, FixTables& shared, cudaStream_t s) {
  const int D = p->dim, LM = fx_lm(D, L.fdm_lmax), HM = (LM + 1) / 2, HP = fx_hm(LM);
  // A' = A / hs = rho * (the operator at h = 1)
  Dd rho{1.0, 0.0};
  L.fx_sf = 0;
  if (D == 3) {
    int e = 0;
    std::frexp(1.0 / L.n, &e);  // h = fr 2^e, fr in [0.5, 1)
    const double two = std::ldexp(1.0, 1 - e);
    rho = dd_inverse(Dd{(double)L.n, 0.0});
    rho = Dd{rho.h * two, rho.l * two};
    L.fx_sf = -(e - 1);
  }
  // Constants are formed once per extent and per pair of extents along y and
  // z, and kept as integers C = round(c 2^58); the bounds need doubles only.
  if (shared.rho != rho.h) {
    shared.lines.clear();
    shared.rho = rho.h;
  }
  std::map<int, FixExtent>& ext = shared.ext;
  auto lines_of = [&](const RasClass& c) -> const FixLines& {
    return shared.lines.at(std::pair<int, int>(c.len[1], D == 2 ? 1 : c.len[2]));
  };
  for (const auto& c : L.classes) {
    for (int k = 0; k < D; ++k)
      if (!ext.count(c.len[k])) ext.emplace(c.len[k], fix_extent(c.len[k]));
    const std::pair<int, int> key(c.len[1], D == 2 ? 1 : c.len[2]);
    if (!shared.lines.count(key))
      shared.lines.emplace(key, fix_lines(D, ext.at(c.len[1]), ext.at(c.len[D - 1]), key.first, key.second, LM, rho));
  }
  double t1 = 1.0, grow = 1.0, norm = 1.0;
  std::vector<std::vector<double>> norms(L.classes.size());
  for (size_t q = 0; q < L.classes.size(); ++q) {
    const RasClass& c = L.classes[q];
    const FixLines& ln = lines_of(c);
    for (size_t sys = 0; sys < ln.b.size(); ++sys) {
      norms[q].push_back(fix_line_norm(&ln.ld[sys * LM], &ln.wd[sys * LM], ln.b[sys], c.len[0], &grow));
      norm = std::max(norm, norms[q].back());
    }
    for (int ax = 1; ax < D; ++ax) t1 = std::max(t1, ext.at(c.len[ax]).row);
  }
  // Quantisation: every operand of a multiply-add stays 1% below 2^60.
  // g bits of residual allow the fold (2), the transforms (t1 per axis), the
  // forward elimination (grow) and, in units of 2^K, the line solutions
  // (norm) and in 3D their transform back along y, which is also the
  // transform along z of the box's solution (bounded by t1 norm_box; norm of
  // the lines times t1^2 bounds both).
  const double lim = 0.99 * std::ldexp(1.0, 60);
  auto bits_below = [&](double factor) { return (int)std::floor(std::log2(lim / factor)); };
  const double tD = D == 2 ? t1 : t1 * t1;
  double solve = std::max(2.0, tD * grow);
  if (D == 3) solve = std::max(solve, 2.0 * t1);
  L.fx_gb = bits_below(solve);
  std::vector<std::vector<int>> K(L.classes.size());
  L.fx_kout = 0;
  int k3 = 0;  // 3D: one K for every line
  if (D == 3) {
    // trade bits of the residual for bits of the solution
    const int g0 = L.fx_gb;
    auto gb_of = [&](int k) { return std::min(g0, bits_below(t1 * tD * norm * std::ldexp(1.0, -k))); };
    for (int k = 0; k < 16; ++k)
      if (gb_of(k) - k > gb_of(k3) - k3 || gb_of(k3) < g0 - 1 || norm * std::ldexp(1.0, -k3) > 1.99) k3 = k;
    L.fx_gb = gb_of(k3);
    L.fx_kout = std::max(0, k3 - 1);
  }
  for (size_t q = 0; q < L.classes.size(); ++q) {
    const FixExtent& ey = ext.at(L.classes[q].len[1]);
    for (double nr : norms[q]) {
      int k = k3;
      if (D == 2) {
        while (bits_below(t1 * nr * std::ldexp(1.0, -k)) < L.fx_gb || nr * std::ldexp(1.0, -k) > 1.99) ++k;
        // units of the results such that S 2^(K_j - kout) < 2
        while (ey.mx * std::ldexp(1.0, k - L.fx_kout) > 1.99) ++L.fx_kout;
      }
      K[q].push_back(k);
    }
  }
  L.fx_rb = std::min(L.fx_gb, 57);  // 6 r as an operand: at most 2^(fx_rb + 2)
  L.fx_sixth = fx_const(fx_const_bits(dd_inverse(Dd{6.0, 0.0})));

  std::vector<int2> tab;
  for (size_t q = 0; q < L.classes.size(); ++q) {
    RasClass& c = L.classes[q];
    const int2 none = make_int2(0, 0);
    for (int ax = 0; ax < D - 1; ++ax) {
      const int l = c.len[ax + 1], hc = (l + 1) / 2;
      const std::vector<long long>& S = ext.at(l).S;
      if (tab.size() & 1) tab.push_back(none);  // the transforms' tables are read as 16-byte pairs
      c.fx_f[ax] = (int)tab.size();
      for (int j = 0; j < LM; ++j)
        for (int x = 0; x < HP; ++x)
          tab.push_back(j < l && x < hc && !((j & 1) && 2 * x + 1 == l) ? fx_const(S[j * l + x]) : none);
      c.fx_b[ax] = (int)tab.size();
      for (int x = 0; x < HM; ++x)
        for (int par = 0; par < 2; ++par)
          for (int k = 0; k < HP; ++k) {
            const int j = 2 * k + par;
            const bool in = j < l && x < hc && !(par && 2 * x + 1 == l);
            // the last transform back (2D: y, 3D: z) goes to the units of the results
            const int sc = !in ? 0 : D == 2 ? K[q][j] - L.fx_kout : ax == 1 ? k3 - L.fx_kout : 0;
            tab.push_back(in ? fx_const(S[j * l + x], sc) : none);
          }
    }
    c.fx_tri = (int)tab.size();
    const FixLines& ln = lines_of(c);
    const int n = c.len[0], nsys = (int)ln.b.size();
    for (int sys = 0; sys < nsys; ++sys)
      if (!(norms[q][sys] * std::ldexp(1.0, -K[q][sys]) < 2.0)) {
        set_error_msg("fixed-point smoother: line factor out of range");
        return DCG_ERR_UNSUPPORTED;
      }
    for (int i = 0; i < n; ++i)
      for (int sys = 0; sys < nsys; ++sys) tab.push_back(fx_const(ln.l[(size_t)sys * LM + i]));
    for (int i = 0; i < n; ++i)
      for (int sys = 0; sys < nsys; ++sys) tab.push_back(fx_const(ln.w[(size_t)sys * LM + i], -K[q][sys]));
    for (int i = 0; i < n; ++i)
      for (int sys = 0; sys < nsys; ++sys) tab.push_back(fx_const(ln.bw[(size_t)sys * LM + i]));
    // read by lines of LM rows only
    for (int sys = 0; sys < nsys; ++sys) tab.push_back(n == LM ? fx_const(ln.meet[sys], -K[q][sys]) : none);
  }
  L.fx_ntab = (int)tab.size();
  DCG_CUDA(cudaMalloc(&L.d_fix, sizeof(int2) * tab.size()));
  DCG_CUDA(cudaMemcpyAsync(L.d_fix, tab.data(), sizeof(int2) * tab.size(), cudaMemcpyHostToDevice, s));
  DCG_CUDA(cudaStreamSynchronize(s));  // the host table goes out of scope
  return DCG_OK;
}

// y = exact local solves of f - Z z on every box (z null: of f; in 3D z is null)
int ras_fix_solve(dcg_problem* p, const Level& L, const double* f, const double* z, cudaStream_t s) {
  FixArgs a{};
  a.work = L.d_work;
  a.class_patches = L.d_class_patches;
  a.classes = L.d_classes;
  a.origin = L.d_origin;
  a.item_off = L.d_item_off;
  a.tab = L.d_fix;
  a.m = L.m;
  a.sc = ras_fix_scale(L, !z);
  const int LM = fx_lm(p->dim, L.fdm_lmax);
  if (p->dim == 3) {
    if (LM == 4) fx_launch<3, 4>(L, a, f, z, s);
    else fx_launch<3, 6>(L, a, f, z, s);
  } else {
    switch (LM) {
      case 4: fx_launch<2, 4>(L, a, f, z, s); break;
      case 6: fx_launch<2, 6>(L, a, f, z, s); break;
      case 8: fx_launch<2, 8>(L, a, f, z, s); break;
      case 10: fx_launch<2, 10>(L, a, f, z, s); break;
      case 12: fx_launch<2, 12>(L, a, f, z, s); break;
      default: fx_launch<2, 16>(L, a, f, z, s);
    }
  }
  DCG_LAUNCH_CHECK();
  return DCG_OK;
}

}  // namespace dcg
