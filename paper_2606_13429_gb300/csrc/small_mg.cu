// Algorithm 3 on small 2D hierarchies as one kernel (FP64).
//
// What bounds a small inner solve is not its work but the chain of dependent
// launches: a W-cycle of four levels at 96^2 is 95 kernels of 2 to 5 us of
// which each does a fraction of a microsecond of arithmetic (406 us per
// cycle, and a host round trip per cycle in the host-driven loop). Here a
// cluster of 16 CTAs runs the whole solve: the inner residual and its norm,
// the convergence test, every level visit of the W-cycle and the update of
// the iterate, one phase after the other with a cluster barrier (hardware, no
// polling) between dependent phases. The vectors stay in L2; values another
// CTA wrote are read past L1 (ld.global.cg). What does not change during the
// solve (transform tables, box descriptors, the indices of the weighted sums,
// the coarsest sine matrix) is copied to shared memory once, because the
// barrier's acquire empties L1 and every dependent global load then costs an
// L2 round trip (with them in global memory a phase took 3.1 us).
//
// The smoother is the box solve of ras_fix.cuh, a warp per box, with the work
// items, tables and box results of the level's own kernels; residuals, transfers
// and weighted sums use the same expressions. A step agrees with the kernels of
// mg.cu to rounding: lines of the largest extent are eliminated from both ends,
// there only in boxes that have it along every axis, here in every such line,
// and in groups of boxes from a zero iterate in none. The coarsest level is
// solved by dense sine passes around Thomas line solves, its rows and lines
// spread over the CTAs.
//
// Measured per inner solve (relative tolerance 1e-10, about 5 cycles), level-by-level
// kernels with the FP64 smoother against this form: four levels, 4 x 4
// cores: 96^2 2,782 -> 1,130 us, 32^2 2,095 -> 665 us; two levels, 8 x 8 cores,
// 96^2 937 -> 455 us (the level-by-level kernels of today: 1,665, 1,495, 615).
#include "ras_fix.cuh"

#include <algorithm>
#include <cmath>
#include <new>

namespace dcg {
namespace {

constexpr int kSmCtas = 16;     // CTAs of the cluster
constexpr int kSmLevels = 8;
constexpr int kSmThreads = 512;
// shared memory of one box: z with its halo, and two copies of the box values
constexpr int sm_box_words(int LM) { return (LM + 2) * (LM + 2) + 2 * LM * (LM | 1); }

enum SmOp { SM_RAS_ZERO = 0, SM_RAS = 1, SM_RES = 2, SM_COARSE = 3, SM_PRO = 4, SM_ZERO = 5, SM_SOLO = 6 };

struct SmLevel {
  int m, nn, nbox;
  const int* boxes;        // [nbox * 2]: work item (-1: none), box of the item
  const int* work;
  const int* class_patches;
  const RasClass* classes;
  const int4* origin;
  const long long* item_off;
  const int2* tab;
  const int* ysrc;
  double *f, *z, *y;
  double c0, c1;  // Z z = c0 z + c1 (3 x 3 box sum)
  FxScale sc, sc0;
  // shared-memory copies (byte offsets; -1: read the global arrays)
  int ntab, o_tab, o_desc, o_cls, o_ysrc;
  int nclass, rounds, bpw; // rounds of bpw boxes of one class per warp
  int o_f, o_z;            // solo levels: the vectors in shared memory
};

// the vectors of a level in the phases: global memory, or shared (solo levels)
struct SmVec {
  double *f, *z, *y;
};

struct SmArgs {
  SmLevel lev[kSmLevels];  // index 0 = coarsest
  int nlev, nops, nsolo, restricted;
  int solo;                // levels up to this index run in CTA 0's shared memory (-1: none)
  int o_y;                 // solo levels: box results
  int o_S, o_work;         // coarsest sine matrix (-1: global) and the phases' work area
  const int* ops;          // op | level index << 8: nops of the cluster, then nsolo of the solo levels
  // coarsest level
  const double *S, *tl, *tw, *te;
  // per call
  const double* g;
  double* z;
  int fixed;               // exactly nmax cycles, no test
  double tol;              // relative tolerance
  const double* tol_dev;   // read instead of tol when set
  int nmax;
  int* ncyc;               // cycles done
  int *total, *iter;       // counters to add them to (may be null)
  const int* in_iter;      // add to `iter` too when set and nonzero
  double* red;             // [2 * kSmCtas]
};

// Phases run on the cluster's CTAs (SOLO = false: vectors in global memory,
// read past L1, cluster barriers) or in one CTA (SOLO: vectors in its shared
// memory, block barriers).
template <bool SOLO>
__device__ __forceinline__ void sm_barrier(int ctas) {
  if (SOLO || ctas == 1) __syncthreads();
  else
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
template <bool SOLO>
__device__ __forceinline__ double sm_ld(const double* p) {
  return SOLO ? *p : __ldcg(p);
}
template <bool SOLO>
__device__ __forceinline__ void sm_st(double* p, double v) {
  if (SOLO) *p = v;
  else __stcg(p, v);
}

// residual of one node, the expressions of the box-sum kernels of mg.cu
template <bool SOLO>
__device__ __forceinline__ double sm_row(const double* z, int x, int y, int m, double& centre) {
  centre = 0.0;
  if (y < 0 || y >= m) return 0.0;
  const double* row = z + m * y;
  centre = sm_ld<SOLO>(row + x);
  double s = centre;
  if (x > 0) s = sm_ld<SOLO>(row + x - 1) + s;
  if (x + 1 < m) s = s + sm_ld<SOLO>(row + x + 1);
  return s;
}
template <bool SOLO>
__device__ __forceinline__ double sm_residual(double c0, double c1, double fv, const double* z, int x, int y, int m) {
  double c, d;
  const double sm = sm_row<SOLO>(z, x, y - 1, m, d), s0 = sm_row<SOLO>(z, x, y, m, c),
               sp = sm_row<SOLO>(z, x, y + 1, m, d);
  const double box = (sm + s0) + sp;
  return fma(-c1, box, fma(-c0, c, fv));
}

// Copies what a level's phases read over and over to shared memory. A box
// descriptor holds the origin, the extents and the class (all zero: no box)
// and the offset of the box's results in y.
template <int LM>
__device__ __forceinline__ void sm_stage(const SmLevel& L, int rank, int ctas, unsigned char* smem) {
  constexpr int NT = kSmThreads, NW = NT / 32;
  if (L.o_tab >= 0)
    for (int t = threadIdx.x; t < L.ntab; t += NT) reinterpret_cast<int2*>(smem + L.o_tab)[t] = __ldg(L.tab + t);
  for (int t = threadIdx.x; t < L.nclass; t += NT) {
    const RasClass& C = L.classes[t];
    reinterpret_cast<int4*>(smem + L.o_cls)[t] = make_int4(C.fx_f[0], C.fx_b[0], C.fx_tri, 0);
  }
  for (int t = threadIdx.x; t < L.rounds * NW * L.bpw; t += NT) {
    const int g = t / L.bpw, c = (rank + ctas * g) * L.bpw + t - g * L.bpw;
    int4 d = make_int4(0, 0, 0, 0);
    if (c < L.nbox && L.boxes[2 * c] >= 0) {
      const int w = L.boxes[2 * c], b = L.boxes[2 * c + 1], cls = L.work[3 * w];
      const RasClass& C = L.classes[cls];
      const int4 og = L.origin[L.class_patches[L.work[3 * w + 1] + b]];
      d = make_int4(og.x | og.y << 16, C.len[0] | C.len[1] << 8, cls, (int)L.item_off[w] + b * C.np);
    }
    reinterpret_cast<int4*>(smem + L.o_desc)[t] = d;
  }
  if (L.o_ysrc >= 0)
    for (int a = rank * NT + threadIdx.x, k = threadIdx.x; a < L.nn; a += ctas * NT, k += NT)
      reinterpret_cast<int4*>(smem + L.o_ysrc)[k] = __ldg(reinterpret_cast<const int4*>(L.ysrc) + a);
}

// Exact solve on one box by one warp: the arithmetic of fx_solve_2d, with the
// entries of every stage spread over the 32 lanes. A lone warp is latency bound, about six clocks per
// instruction, so the count per lane is what a small level costs: with a lane
// per column a step's solve took 5,700 clocks whatever the level's size.
template <int LM, bool SOLO>
__device__ __forceinline__ void sm_box(const FxScale& sc, bool zzero, int lx, int ly, int ox, int oy, int m,
                                       const double* z, const double* f, double* y, const int2* tf, const int2* tb,
                                       const int2* tri, long long* Z) {
  constexpr int HM = (LM + 1) / 2, HP = fx_hm(LM);
  constexpr int NZ = ((LM + 2) * (LM + 2) + 31) / 32, NF = (LM * LM + 31) / 32;
  const int lane = threadIdx.x & 31;
  const int wp = lx | 1, hx = lx + 2, nz = hx * (ly + 2), nf = lx * ly;
  long long* W = Z + (LM + 2) * (LM + 2);
  long long* W2 = W + LM * (LM | 1);
  // entry t of rows of length len: t / len by a 16-bit reciprocal (t < 400)
  const int ihx = (65536 + hx - 1) / hx, ilx = (65536 + lx - 1) / lx;
  long long zv[NZ], fv[NF];
  unsigned mag = 0;
#pragma unroll
  for (int i = 0; i < NF; ++i) {
    const int t = lane + 32 * i, q = (t * ilx) >> 16;
    fv[i] = t < nf ? __double_as_longlong(sm_ld<SOLO>(f + ox + t - q * lx + m * (oy + q))) : 0;
    mag = max(mag, fx_mag(fv[i]));
  }
  if (!zzero) {
#pragma unroll
    for (int i = 0; i < NZ; ++i) {
      const int t = lane + 32 * i, q = (t * ihx) >> 16, gx = ox - 1 + t - q * hx, gy = oy - 1 + q;
      const bool in = t < nz && gx >= 0 && gx < m && gy >= 0 && gy < m;
      zv[i] = in ? __double_as_longlong(sm_ld<SOLO>(z + gx + m * gy)) : 0;
      mag = max(mag, fx_mag(zv[i]));
    }
  }
  mag = __reduce_max_sync(0xffffffffu, mag);
  const int e = max((int)(mag >> 20), kFxLowest);
  int e0 = e + 63 + sc.kout;
  if (zzero) {
    const int sh0 = 63 - sc.bits + e;
    e0 -= sc.bits;
#pragma unroll
    for (int i = 0; i < NF; ++i) {
      const int t = lane + 32 * i, q = (t * ilx) >> 16;
      if (t < nf) W[q * wp + t - q * lx] = fx_near(fv[i], sh0);
    }
  } else {
    const int sh0 = 63 - kFxZBits + e;
#pragma unroll
    for (int i = 0; i < NZ; ++i) {
      const int t = lane + 32 * i;
      if (t < nz) Z[t] = fx_near(zv[i], sh0);
    }
    __syncwarp();
    unsigned long long any = 0;
#pragma unroll
    for (int i = 0; i < NF; ++i) {
      const int t = lane + 32 * i, q = (t * ilx) >> 16, x = t - q * lx;
      if (t < nf) {
        const long long* p = Z + q * hx + x;
        const long long c = p[hx + 1];
        fv[i] = ((p[0] + p[1] + p[2]) + (p[hx] + c + p[hx + 2]) + (p[2 * hx] + p[2 * hx + 1] + p[2 * hx + 2])) -
                (c << 3) - c + fx_near(fv[i], sh0) * 6;
        any |= fx_abs1(fv[i]);
      }
    }
    const int len = __reduce_max_sync(0xffffffffu, any ? fx_length(any) : 0);
    const int shift = len ? sc.bits + 2 - len : 0;
    e0 -= kFxZBits + shift;
#pragma unroll
    for (int i = 0; i < NF; ++i) {
      const int t = lane + 32 * i, q = (t * ilx) >> 16;
      if (t < nf) W[q * wp + t - q * lx] = fx_res(fv[i], shift, sc.sixth);
    }
  }
  __syncwarp();
  const int h = ly >> 1, hc = (ly + 1) >> 1;
#pragma unroll
  for (int i = 0; i < NF; ++i) {
    const int t = lane + 32 * i, j = (t * ilx) >> 16, x = t - j * lx;
    if (t < nf) {
      FxAcc acc = fx_zero();
#pragma unroll
      for (int k = 0; k < HM; ++k) {
        const long long a = k < hc ? W[k * wp + x] : 0, b = k < h ? W[(ly - 1 - k) * wp + x] : 0;
        const int2 c = tf[j * HP + k];
        fx_mac(acc, fx_split((j & 1) ? a - b : a + b), c.x, c.y);
      }
      W2[j * wp + x] = fx_value(acc);
    }
  }
  __syncwarp();
  if (lane < ly) {
    if (lx == LM) fx_line_solve<LM, true>(W2 + lane * wp, lx, tri + lane, ly);
    else fx_line_solve<LM, false>(W2 + lane * wp, lx, tri + lane, ly);
  }
  __syncwarp();
#pragma unroll
  for (int i = 0; i < (HM * LM + 31) / 32; ++i) {
    const int t = lane + 32 * i, q = (t * ilx) >> 16, x = t - q * lx;
    if (t < hc * lx) {
      FxAcc ev = fx_zero(), od = fx_zero();
#pragma unroll
      for (int k = 0; k < HM; ++k) {
        const int2 ce = tb[(2 * q) * HP + k], co = tb[(2 * q + 1) * HP + k];
        fx_mac(ev, fx_split(2 * k < ly ? W2[(2 * k) * wp + x] : 0), ce.x, ce.y);
        fx_mac(od, fx_split(2 * k + 1 < ly ? W2[(2 * k + 1) * wp + x] : 0), co.x, co.y);
      }
      const long long E = fx_value(ev), O = fx_value(od);
      sm_st<SOLO>(y + q * lx + x, mag < kFxNonFinite ? fx_to_double(E + O, e0) : fx_nan());
      if (q < h)
        sm_st<SOLO>(y + (ly - 1 - q) * lx + x, mag < kFxNonFinite ? fx_to_double(E - O, e0) : fx_nan());
    }
  }
  __syncwarp();  // the next box overwrites the shared values
}

// one smoothing step on the level: box solves, barrier, weighted sums, barrier
template <int LM, bool SOLO>
__device__ __forceinline__ void sm_ras(const SmLevel& L, const SmVec& V, bool zzero, int restricted, int rank, int ctas,
                                       unsigned char* smem, int o_work) {
  constexpr int NT = kSmThreads, NW = NT / 32;
  const int warp = threadIdx.x >> 5;
  const int4* desc = reinterpret_cast<const int4*>(smem + L.o_desc);
  const int2* tab = L.o_tab >= 0 ? reinterpret_cast<const int2*>(smem + L.o_tab) : L.tab;
  const FxScale& sc = zzero ? L.sc0 : L.sc;
  if (L.bpw > 1) {
    // more boxes than warps: a lane per column, as in k_ras_fix
    constexpr int G = fx_group(LM), BPW = 32 / G;
    const int lane = threadIdx.x & (G - 1), sub = (threadIdx.x & 31) / G, x = lane - 1, m = L.m;
    for (int it = 0; it < L.rounds; ++it) {
      const int4 d0 = desc[(it * NW + warp) * BPW], d = desc[(it * NW + warp) * BPW + sub];
      if (d0.y == 0) break;
      const int lx = d0.y & 255, ly = d0.y >> 8, ox = d.x & 0xffff, oy = d.x >> 16;
      const bool live = d.y != 0, own = live && x >= 0 && x < lx;
      long long zv[LM + 2], fv[LM];
      const int gx = ox + x, base = gx + m * (oy - 1);
      const bool col = live && !zzero && x <= lx && gx >= 0 && gx < m;
#pragma unroll
      for (int q = 0; q < LM + 2; ++q) {
        const int gy = oy - 1 + q;
        zv[q] = (col && q <= ly + 1 && gy >= 0 && gy < m) ? __double_as_longlong(sm_ld<SOLO>(V.z + base + q * m)) : 0;
      }
#pragma unroll
      for (int q = 0; q < LM; ++q)
        fv[q] = (own && q < ly) ? __double_as_longlong(sm_ld<SOLO>(V.f + base + (q + 1) * m)) : 0;
      const int4 cls = reinterpret_cast<const int4*>(smem + L.o_cls)[d0.z];
      double* yb = V.y + d.w + x;
      long long* W = reinterpret_cast<long long*>(smem + o_work) + (warp * BPW + sub) * (LM * (LM | 1));
      auto out = [&](int q, double v) { sm_st<SOLO>(yb + q * lx, v); };
      if (zzero)
        fx_solve_2d<LM, true, false, false>(sc, lx, ly, live, zv, fv, W, tab + cls.x, tab + cls.y, tab + cls.z, out);
      else if (lx == LM && ly == LM)
        fx_solve_2d<LM, false, true, false>(sc, LM, LM, live, zv, fv, W, tab + cls.x, tab + cls.y, tab + cls.z, out);
      else
        fx_solve_2d<LM, false, false, false>(sc, lx, ly, live, zv, fv, W, tab + cls.x, tab + cls.y, tab + cls.z, out);
      __syncwarp();
    }
  } else
  for (int it = 0; it < L.rounds; ++it) {
    const int4 d = desc[it * NW + warp];
    if (d.y == 0) break;  // boxes are dealt out in order
    const int4 cls = reinterpret_cast<const int4*>(smem + L.o_cls)[d.z];
    sm_box<LM, SOLO>(sc, zzero, d.y & 255, d.y >> 8, d.x & 0xffff, d.x >> 16, L.m, V.z, V.f, V.y + d.w, tab + cls.x,
                     tab + cls.y, tab + cls.z,
                     reinterpret_cast<long long*>(smem + o_work) + warp * sm_box_words(LM));
  }
  sm_barrier<SOLO>(ctas);
  for (int a = rank * NT + threadIdx.x, k = threadIdx.x; a < L.nn; a += ctas * NT, k += NT) {
    const int4 id = L.o_ysrc >= 0 ? reinterpret_cast<const int4*>(smem + L.o_ysrc)[k]
                                  : __ldg(reinterpret_cast<const int4*>(L.ysrc) + a);
    const bool h1 = !restricted && id.y >= 0, h2 = !restricted && id.z >= 0, h3 = !restricted && id.w >= 0;
    const double zo = zzero ? 0.0 : sm_ld<SOLO>(V.z + a);
    double s = sm_ld<SOLO>(V.y + id.x);
    const double s1 = h1 ? sm_ld<SOLO>(V.y + id.y) : 0.0, s2 = h2 ? sm_ld<SOLO>(V.y + id.z) : 0.0,
                 s3 = h3 ? sm_ld<SOLO>(V.y + id.w) : 0.0;
    int mult = 1;
    if (h1) { s += s1; ++mult; }
    if (h2) { s += s2; ++mult; }
    if (h3) { s += s3; ++mult; }
    const double inv = mult == 1 ? 1.0 : mult == 2 ? 0.5 : 0.25;
    sm_st<SOLO>(V.z + a, fma(s, inv, zo));
  }
  sm_barrier<SOLO>(ctas);
}

// coarse f = R (f - Z z): a CTA takes a block of coarse rows, the fine
// residual rows it needs go to shared memory. The coarse vector is global
// unless the fine level is a solo level too.
template <bool SOLO, int NT>
__device__ __forceinline__ void sm_restrict(const SmLevel& L, const SmVec& V, int mc, double* fc, int rank, int ctas,
                                            double* work) {
  const int m = L.m, rows = (mc + ctas - 1) / ctas;
  const int r0 = rank * rows, r1 = min(mc, r0 + rows);
  if (r0 < r1) {
    const int y0 = 2 * r0, ny = 2 * (r1 - r0) + 1;  // fine rows y0 .. y0 + ny - 1
    for (int t = threadIdx.x; t < ny * m; t += NT) {
      const int q = t / m, x = t - q * m, y = y0 + q;
      work[t] = sm_residual<SOLO>(L.c0, L.c1, sm_ld<SOLO>(V.f + x + m * y), V.z, x, y, m);
    }
    __syncthreads();
    for (int t = threadIdx.x; t < (r1 - r0) * mc; t += NT) {
      const int q = t / mc, X = t - q * mc;
      double row[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const double* f = work + (2 * q + k) * m + 2 * X + 1;
        row[k] = fma(0.5, f[-1] + f[1], f[0]);
      }
      sm_st<SOLO>(fc + X + mc * (r0 + q), fma(0.5, row[0] + row[2], row[1]));
    }
  }
  sm_barrier<SOLO>(ctas);
}

// z += P (coarse z)
template <bool SOLO, int NT>
__device__ __forceinline__ void sm_prolong(const SmLevel& L, const SmVec& V, int mc, const double* zc, int rank,
                                           int ctas) {
  const int m = L.m;
  for (int a = rank * NT + threadIdx.x; a < L.nn; a += ctas * NT) {
    const int y = a / m, x = a - y * m;
    const bool ey = (y & 1) == 0, ex = (x & 1) == 0;
    const int r2 = y >> 1, r1 = ey ? r2 - 1 : r2, i = x >> 1;  // coarse rows r1 (r2), columns i - 1 (even x), i
    auto cv = [&](int r, int c) {
      return (r >= 0 && r < mc && c >= 0 && c < mc) ? sm_ld<SOLO>(zc + r * mc + c) : 0.0;
    };
    double b = cv(r1, i);
    if (ey) b += cv(r2, i);
    const double wr = ey ? 0.5 : 1.0;
    double v = sm_ld<SOLO>(V.z + a);
    if (ex) {
      double c = cv(r1, i - 1);
      if (ey) c += cv(r2, i - 1);
      v = fma(0.5 * wr, c + b, v);
    } else {
      v = fma(wr, b, v);
    }
    sm_st<SOLO>(V.z + a, v);
  }
  sm_barrier<SOLO>(ctas);
}

// rows of out = rows of in times S (symmetric), rows spread over the CTAs;
// each row is folded by S[m-1-k][i] = (-1)^i S[k][i], half the FP64 operations
template <bool SOLO, int NT>
__device__ __forceinline__ void sm_sine_rows(int m, const double* S, const double* in, double* out, int rank, int ctas,
                                             double* work) {
  const int rows = (m + ctas - 1) / ctas, h = m >> 1, hc = (m + 1) >> 1;
  const int r0 = rank * rows, nr = max(0, min(m, r0 + rows) - r0);
  for (int t = threadIdx.x; t < nr * hc; t += NT) {
    const int q = t / hc, k = t - q * hc;
    const double* row = in + (r0 + q) * m;
    const double a = sm_ld<SOLO>(row + k), b = k < h ? sm_ld<SOLO>(row + m - 1 - k) : 0.0;
    work[q * m + k] = a + b;
    if (k < h) work[q * m + hc + k] = a - b;
  }
  __syncthreads();
  for (int t = threadIdx.x; t < nr * m; t += NT) {
    const int q = t / m, i = t - q * m, cnt = (i & 1) ? h : hc;
    const double* v = work + q * m + ((i & 1) ? hc : 0);
    double a0 = 0.0, a1 = 0.0;
    int k = 0;
    for (; k + 1 < cnt; k += 2) {
      a0 = fma(S[k * m + i], v[k], a0);
      a1 = fma(S[(k + 1) * m + i], v[k + 1], a1);
    }
    if (k < cnt) a0 = fma(S[k * m + i], v[k], a0);
    sm_st<SOLO>(out + r0 * m + t, a0 + a1);
  }
  sm_barrier<SOLO>(ctas);
}

// exact coarsest solve z = Z_1^-1 f: sine transform along x (into z), Thomas
// solves along y of the transformed lines, transform back
template <bool SOLO, int NT>
__device__ __forceinline__ void sm_coarse(const SmArgs& A, const double* S, const double* f, double* z, int rank,
                                          int ctas, double* work) {
  const int m = A.lev[0].m, cols = (m + ctas - 1) / ctas;
  sm_sine_rows<SOLO, NT>(m, S, f, z, rank, ctas, work);
  const int j0 = rank * cols, nc = max(0, min(m, j0 + cols) - j0);
  for (int t = threadIdx.x; t < nc * m; t += NT) {
    const int y = t / nc, o = y * m + j0 + t - y * nc;
    work[t] = sm_ld<SOLO>(z + o);
    work[nc * m + t] = __ldg(A.tl + o);
    work[2 * nc * m + t] = __ldg(A.tw + o);
  }
  __syncthreads();
  if (threadIdx.x < nc) {
    const double *sl = work + nc * m, *sw = work + 2 * nc * m;
    const double e = __ldg(A.te + j0 + threadIdx.x);
    double prev = 0.0;
    for (int t = threadIdx.x; t < nc * m; t += nc) {
      prev = fma(-sl[t], prev, work[t]);
      work[t] = prev;
    }
    double xn = 0.0;
    for (int t = (m - 1) * nc + threadIdx.x; t >= 0; t -= nc) {
      xn = fma(-(e * sw[t]), xn, work[t] * sw[t]);
      work[t] = xn;
    }
  }
  __syncthreads();
  for (int t = threadIdx.x; t < nc * m; t += NT) {
    const int y = t / nc;
    sm_st<SOLO>(z + y * m + j0 + t - y * nc, work[t]);
  }
  sm_barrier<SOLO>(ctas);
  sm_sine_rows<SOLO, NT>(m, S, z, z, rank, ctas, work);
}

template <int LM, bool SOLO>
__device__ __forceinline__ void sm_run(const SmArgs& A, int op, const double* S, int rank, int ctas,
                                       unsigned char* smem) {
  constexpr int NT = kSmThreads;
  const int kind = op & 255, k = op >> 8;
  const SmLevel& L = A.lev[k];
  double* work = reinterpret_cast<double*>(smem + A.o_work);
  auto vec = [&](int q) {
    const SmLevel& l = A.lev[q];
    return SOLO ? SmVec{reinterpret_cast<double*>(smem + l.o_f), reinterpret_cast<double*>(smem + l.o_z),
                        reinterpret_cast<double*>(smem + A.o_y)}
                : SmVec{l.f, l.z, l.y};
  };
  const SmVec V = vec(k);
  switch (kind) {
    case SM_RAS_ZERO:
    case SM_RAS: sm_ras<LM, SOLO>(L, V, kind == SM_RAS_ZERO, A.restricted, rank, ctas, smem, A.o_work); break;
    case SM_RES: sm_restrict<SOLO, NT>(L, V, A.lev[k - 1].m, vec(k - 1).f, rank, ctas, work); break;
    case SM_COARSE: sm_coarse<SOLO, NT>(A, S, V.f, V.z, rank, ctas, work); break;
    case SM_PRO: sm_prolong<SOLO, NT>(L, V, A.lev[k - 1].m, vec(k - 1).z, rank, ctas); break;
    default:
      for (int a = rank * NT + threadIdx.x; a < L.nn; a += ctas * NT) sm_st<SOLO>(V.z + a, 0.0);
      sm_barrier<SOLO>(ctas);
  }
}

// A cycle whose residual has a norm beyond 2^+-300 starts from the residual
// scaled to a largest entry in [1, 2), so that its boxes hold nothing near the
// ends of the FP64 range (the box solves of a cycle leave out what lies below
// 2^-831); the power of two that is returned (1 where it is zero or not finite)
// comes off its correction.
template <int NT>
__device__ __noinline__ double sm_to_one(double* f, int nn, double* red, int rank, int ctas, double* s_red) {
  unsigned mag = 0;
  for (int a = rank * NT + threadIdx.x; a < nn; a += ctas * NT) mag = max(mag, fx_mag(__double_as_longlong(__ldcg(f + a))));
  mag = __reduce_max_sync(0xffffffffu, mag);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = (double)mag;
  __syncthreads();
  double m = 0.0;
  for (int k = 0; k < NT / 32; ++k) m = max(m, s_red[k]);
  sm_barrier<false>(ctas);  // the norms in `red` have been read
  if (threadIdx.x == 0) __stcg(red + 2 * rank, m);
  sm_barrier<false>(ctas);
  for (int k = 0; k < ctas; ++k) m = max(m, __ldcg(red + 2 * k));
  mag = (unsigned)m;
  if (mag == 0 || mag >= kFxNonFinite) return 1.0;
  // 2^1023 / 2^(field): a subnormal number for the largest field
  const int e = 2046 - max((int)(mag >> 20), 1);
  const double s = e > 0 ? __longlong_as_double((long long)e << 52) : __longlong_as_double(1LL << 51);
  for (int a = rank * NT + threadIdx.x; a < nn; a += ctas * NT) __stcg(f + a, __ldcg(f + a) * s);
  sm_barrier<false>(ctas);
  return s;
}

template <int LM>
__global__ void __launch_bounds__(kSmThreads, 1) k_small_mg(const __grid_constant__ SmArgs A) {
  constexpr int NT = kSmThreads;
  extern __shared__ __align__(16) unsigned char sm_smem[];
  __shared__ double s_red[64];
  const int rank = blockIdx.x, ctas = gridDim.x;  // one cluster, or one CTA
  for (int k = 1; k < A.nlev; ++k) {
    if (k > A.solo) sm_stage<LM>(A.lev[k], rank, ctas, sm_smem);
    else if (rank == 0) sm_stage<LM>(A.lev[k], 0, 1, sm_smem);
  }
  const double* S = A.S;
  if (A.o_S >= 0) {
    double* c = reinterpret_cast<double*>(sm_smem + A.o_S);
    const int m0 = A.lev[0].m;
    for (int t = threadIdx.x; t < m0 * m0; t += NT) c[t] = __ldg(A.S + t);
    S = c;
  }
  __syncthreads();
  const SmLevel& T = A.lev[A.nlev - 1];
  const double tol = A.tol_dev ? __ldcg(A.tol_dev) : A.tol;
  double gn = 0.0;
  int n = 0;
  for (;;) {
    // inner residual r = g - Z z into the top level's right-hand side
    double part[2] = {0.0, 0.0};
    for (int a = rank * NT + threadIdx.x; a < T.nn; a += ctas * NT) {
      const int y = a / T.m, x = a - y * T.m;
      const double ga = __ldg(A.g + a);
      const double r = sm_residual<false>(T.c0, T.c1, ga, A.z, x, y, T.m);
      __stcg(T.f + a, r);
      part[0] = fma(r, r, part[0]);
      part[1] = fma(ga, ga, part[1]);
    }
    block_sum<2>(part, s_red);
    if (threadIdx.x == 0) {
      __stcg(A.red + 2 * rank, part[0]);
      __stcg(A.red + 2 * rank + 1, part[1]);
    }
    sm_barrier<false>(ctas);
    double rr = 0.0, gg = 0.0;
    for (int k = 0; k < ctas; ++k) {
      rr += __ldcg(A.red + 2 * k);
      gg += __ldcg(A.red + 2 * k + 1);
    }
    // Algorithm 3's test, the same decision in every thread
    if (!A.fixed) {
      const double rn = sqrt(rr);
      if (n == 0) gn = sqrt(gg);
      if (!(gn > 0.0) || !(rn / gn > tol)) break;
    }
    if (n >= A.nmax) break;
    double scale = 1.0;
    if (!(rr >= 0x1p-600 && rr <= 0x1p600)) scale = sm_to_one<NT>(T.f, T.nn, A.red, rank, ctas, s_red);
    for (int k = 0; k < A.nops; ++k) {
      const int op = __ldg(A.ops + k);
      if ((op & 255) != SM_SOLO) {
        sm_run<LM, false>(A, op, S, rank, ctas, sm_smem);
        continue;
      }
      // the W-cycle of the solo levels (both recursive calls of Algorithm 4)
      if (rank == 0) {
        const SmLevel& L = A.lev[A.solo];
        double* f = reinterpret_cast<double*>(sm_smem + L.o_f);
        const double* z = reinterpret_cast<const double*>(sm_smem + L.o_z);
        for (int a = threadIdx.x; a < L.nn; a += NT) f[a] = __ldcg(L.f + a);
        __syncthreads();
        for (int q = 0; q < A.nsolo; ++q) sm_run<LM, true>(A, __ldg(A.ops + A.nops + q), S, 0, 1, sm_smem);
        for (int a = threadIdx.x; a < L.nn; a += NT) __stcg(L.z + a, z[a]);
      }
      sm_barrier<false>(ctas);
    }
    for (int a = rank * NT + threadIdx.x; a < T.nn; a += ctas * NT)
      __stcg(A.z + a, __ldcg(A.z + a) + (scale == 1.0 ? __ldcg(T.z + a) : __ldcg(T.z + a) / scale));
    sm_barrier<false>(ctas);
    ++n;
  }
  if (rank == 0 && threadIdx.x == 0) {
    *A.ncyc = n;
    if (A.total) *A.total += n;
    if (A.iter && A.in_iter && *A.in_iter) *A.iter += n;
  }
}

// Thomas factors of the coarsest level's transformed lines (the closed form of
// mg.cu's k_tri_setup in 2D), for hierarchies whose own tables are the
// cyclic-reduction ones
__global__ void k_small_tri(int m, double* __restrict__ fl, double* __restrict__ fw, double* __restrict__ fe) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= m) return;
  const double h = 1.0 / (m + 1), th = M_PI * (j + 1) / (m + 1);
  const double a = (2.0 / h) * (1.0 - cos(th)) / 2.0, b = (h / 3.0) * (2.0 + cos(th)) / 2.0;
  const double dg = a * (2.0 * h / 3.0) + b * (2.0 / h), e = a * (h / 6.0) - b / h;
  double w = dg;
  fl[j] = 0.0;
  fw[j] = 1.0 / w;
  for (int y = 1; y < m; ++y) {
    const double l = e / w;
    w = dg - l * e;
    fl[j + m * y] = l;
    fw[j + m * y] = 1.0 / w;
  }
  fe[j] = e;
}

struct SmallState {
  SmArgs args{};
  int lm = 0, ctas = kSmCtas;
  size_t smem = 0;
  double* buf = nullptr;   // tri [2 m^2 + m], red [2 * kSmCtas], then the integers
  std::vector<int> host;   // ops, boxes ([2] per box of every smoothed level), ncyc
};

// Algorithm 4 on level index k (0 = coarsest); levels up to `solo` are one
// operation (its own list is made with solo = -1)
void sm_cycle(std::vector<int>& ops, const dcg_options& o, int k, bool zero, int solo) {
  if (k == solo) {
    ops.push_back(SM_SOLO | k << 8);
    return;
  }
  if (k == 0) {
    ops.push_back(SM_COARSE);
    return;
  }
  if (zero && o.m1 == 0) ops.push_back(SM_ZERO | k << 8);
  for (int i = 0; i < o.m1; ++i) ops.push_back((zero && i == 0 ? SM_RAS_ZERO : SM_RAS) | k << 8);
  ops.push_back(SM_RES | k << 8);
  sm_cycle(ops, o, k - 1, true, solo);
  if (k - 1 > 0 && k - 1 != solo) sm_cycle(ops, o, k - 1, false, solo);
  ops.push_back(SM_PRO | k << 8);
  for (int i = 0; i < o.m2; ++i) ops.push_back(SM_RAS | k << 8);
}

// launch configuration of one cluster
void sm_config(int ctas, int threads, size_t smem, cudaStream_t s, cudaLaunchConfig_t* cfg, cudaLaunchAttribute* at) {
  *cfg = cudaLaunchConfig_t{};
  cfg->gridDim = dim3(ctas);
  cfg->blockDim = dim3(threads);
  cfg->dynamicSmemBytes = smem;
  cfg->stream = s;
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = ctas;
  at->val.clusterDim.y = 1;
  at->val.clusterDim.z = 1;
  cfg->attrs = at;
  cfg->numAttrs = 1;
}

// shared memory a problem may plan for (227 KB less the kernel's static part)
constexpr size_t kSmRoom = 216 * 1024;

// *fits: the device can hold one such cluster. The limit on the dynamic shared
// memory belongs to the kernel, not to a problem: every problem sets the same
// constant, and a launch asks for what its own plan takes.
template <int LM>
int sm_attr(int ctas, size_t smem, bool* fits) {
  DCG_CUDA(cudaFuncSetAttribute(k_small_mg<LM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmRoom));
  DCG_CUDA(cudaFuncSetAttribute(k_small_mg<LM>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at[1];
  sm_config(ctas, kSmThreads, smem, nullptr, &cfg, at);
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, k_small_mg<LM>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    n = 0;
  }
  *fits = n > 0;
  return DCG_OK;
}

template <int LM>
cudaError_t sm_start(const SmArgs& a, int ctas, size_t smem, cudaStream_t s) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at[1];
  sm_config(ctas, kSmThreads, smem, s, &cfg, at);
  return cudaLaunchKernelEx(&cfg, k_small_mg<LM>, a);
}

int sm_dispatch(const SmallState& S, const SmArgs& a, cudaStream_t s) {
  cudaError_t e;
  switch (S.lm) {
    case 4: e = sm_start<4>(a, S.ctas, S.smem, s); break;
    case 6: e = sm_start<6>(a, S.ctas, S.smem, s); break;
    case 8: e = sm_start<8>(a, S.ctas, S.smem, s); break;
    case 10: e = sm_start<10>(a, S.ctas, S.smem, s); break;
    case 12: e = sm_start<12>(a, S.ctas, S.smem, s); break;
    default: e = sm_start<16>(a, S.ctas, S.smem, s);
  }
  if (e != cudaSuccess) {
    cudaGetLastError();  // reported here, not by the next launch check
    set_error("small multigrid solve (cluster launch)", e);
    return DCG_ERR_CUDA;
  }
  DCG_LAUNCH_CHECK();
  return DCG_OK;
}

}  // namespace

// The one-kernel solve serves FP64 2D hierarchies of at least two levels whose
// smoothed levels are box-sum levels with fixed-point local solves, with at
// most kSmallNodes nodes on the finest level (two levels: kSmallNodes2) and 80
// per axis on the coarsest (its dense passes grow with the cube). Per inner
// solve against the level-by-level kernels with fixed-point smoother, us: four
// levels, 4 x 4 cores, 112^2 1,171 / 1,664, 160^2 1,428 / 1,733; two levels, 4 x 4
// cores, 64^2 324 / 428, 112^2 428 / 503, 128^2 503 / 467, 160^2 630 / 569; 8 x 8
// cores, 128^2 543 / 568, 160^2 675 / 679. Above these sizes a phase no longer is
// the latency of one round, with two levels sooner (fewer phases per cycle,
// more work in each): whole captured solves of two levels, 4 x 4 cores, take
// 8.18 against 6.64 ms at 128^2 and 12.22 against 10.02 at 160^2, so two levels
// stop at kSmallNodes2. Deeper hierarchies stop at the largest size measured;
// their crossing lies above it.
// A solve holds 16 SMs, so about nine run at a time, the level kernels of a
// batch more; batches gain all the same (ms, one kernel / level kernels): 64
// problems, two levels 32^2 67 / 103, 112^2 77 / 114, four levels 32^2 152 / 408,
// 112^2 197 / 357; 8 problems, two levels 112^2 10.0 / 14.3.
constexpr long long kSmallNodes = 26000, kSmallNodes2 = 13000;
bool small_mg_supported(const dcg_problem* p) {
  const int J = (int)p->levels.size();
  if (p->dim != 2 || p->mg.fp32 || J < 2 || J > kSmLevels || p->coarse.m > 80 ||
      p->levels.back().nn > (J > 2 ? kSmallNodes : kSmallNodes2))
    return false;
  for (int k = 1; k < J; ++k)
    if (!p->levels[k].fdm || !p->levels[k].box) return false;
  return true;
}

void small_mg_free(dcg_problem* p) {
  SmallState* S = static_cast<SmallState*>(p->mg.small);
  if (!S) return;
  cudaFree(S->buf);
  delete S;
  p->mg.small = nullptr;
}

int small_mg_setup(dcg_problem* p, cudaStream_t s) {
  small_mg_free(p);
  if (!small_mg_supported(p)) return DCG_OK;
  SmallState* S = new (std::nothrow) SmallState();
  if (!S) return DCG_ERR_OOM;
  p->mg.small = S;
  SmArgs& a = S->args;
  const int J = (int)p->levels.size(), m0 = p->coarse.m;
  S->lm = ras_fix_lm(2, p->levels.back().fdm_lmax);
  a.nlev = J;
  a.restricted = p->opts.ras_weights == DCG_RAS_RESTRICTED;
  const int nt = kSmThreads, warps = nt / 32;
  // The levels' boxes in the order of their work items: one per warp where the
  // cluster has a warp for each, else in groups of one class (a lane per
  // column; 95^2: 11,000 clocks per step against 18,300 in three rounds).
  const int group = S->lm + 2 <= 8 ? 8 : S->lm + 2 <= 16 ? 16 : 32;
  std::vector<int> boxes, bpw(J, 1);
  std::vector<size_t> box_end(J, 0);
  for (int k = 1; k < J; ++k) {
    const Level& L = p->levels[k];
    bpw[k] = L.npatch <= kSmCtas * warps ? 1 : 32 / group;
    for (int w = 0; w < L.nwork; ++w) {
      const int cnt = L.item_count[w];
      for (int b = 0; b < (cnt + bpw[k] - 1) / bpw[k] * bpw[k]; ++b) {
        boxes.push_back(b < cnt ? w : -1);
        boxes.push_back(b);
      }
    }
    box_end[k] = boxes.size();
  }
  // solo levels: at most one box per warp of a CTA (a step takes 5,300 clocks
  // against 9,100 with cluster barriers; 15,000 in three rounds), and a coarsest
  // level of at most 15 per axis; with all levels solo one CTA does the solve
  a.solo = -1;
  if (m0 <= 15)
    for (int k = 0; k < J; ++k)
      if (k == 0 || p->levels[k].npatch <= warps) a.solo = k;
      else break;
  S->ctas = a.solo == J - 1 ? 1 : kSmCtas;
  auto ctas_of = [&](int k) { return k <= a.solo ? 1 : S->ctas; };
  // work area: box values per warp, fine residual rows of a restriction, or a
  // share of the coarsest solve; then the copies, as far as they fit
  size_t work = sizeof(long long) * warps * std::max(sm_box_words(S->lm), 32 / group * S->lm * (S->lm | 1));
  work = std::max(work, sizeof(double) * 3 * m0 * ((m0 + ctas_of(0) - 1) / ctas_of(0)));
  for (int k = 1; k < J; ++k)
    work = std::max(work, sizeof(double) * p->levels[k].m *
                              (2 * ((p->levels[k - 1].m + ctas_of(k) - 1) / ctas_of(k)) + 1));
  size_t used = 0, ymax = 0;
  auto take = [&](size_t bytes) {
    const size_t at = used;
    used += (bytes + 15) / 16 * 16;
    return (int)at;
  };
  a.o_work = take(work);
  for (int k = 0; k < J; ++k) {
    const Level& L = p->levels[k];
    SmLevel& l = a.lev[k];
    l.m = L.m;
    l.nn = (int)L.nn;
    l.f = (double*)L.f;
    l.z = (double*)L.z;
    if (k <= a.solo) {
      l.o_f = take(sizeof(double) * L.nn);
      l.o_z = take(sizeof(double) * L.nn);
    }
    if (k == 0) continue;
    if (k <= a.solo) ymax = std::max(ymax, sizeof(double) * (size_t)L.ylen);
    l.work = L.d_work;
    l.class_patches = L.d_class_patches;
    l.classes = L.d_classes;
    l.origin = L.d_origin;
    l.item_off = L.d_item_off;
    l.tab = L.d_fix;
    l.ysrc = L.d_ysrc;
    l.y = (double*)L.y;
    l.c0 = L.box_c0;
    l.c1 = L.box_c1;
    l.sc = ras_fix_scale(L, false);
    l.sc0 = ras_fix_scale(L, true);
    l.ntab = L.fx_ntab;
    l.nclass = L.nclass;
    const int each = ctas_of(k) * warps;
    l.nbox = (int)(box_end[k] - box_end[k - 1]) / 2;
    l.bpw = bpw[k];
    l.rounds = (l.nbox / l.bpw + each - 1) / each;
    l.o_desc = take(sizeof(int4) * l.rounds * warps * l.bpw);
    l.o_cls = take(sizeof(int4) * L.nclass);
  }
  a.o_y = take(ymax);
  if (used > kSmRoom) {  // no room for the solo levels' vectors
    small_mg_free(p);
    return DCG_OK;
  }
  // the coarser a level, the more often a W-cycle visits it
  a.o_S = used + sizeof(double) * m0 * m0 <= kSmRoom ? take(sizeof(double) * m0 * m0) : -1;
  for (int k = 1; k < J; ++k) {
    SmLevel& l = a.lev[k];
    const int share = ctas_of(k) * nt;
    const size_t tb = sizeof(int2) * l.ntab, yb = sizeof(int4) * nt * ((l.nn + share - 1) / share);
    l.o_tab = used + tb <= kSmRoom ? take(tb) : -1;
    l.o_ysrc = used + yb <= kSmRoom ? take(yb) : -1;
  }
  const size_t smem = used;
  S->smem = smem;
  std::vector<int> ops;
  sm_cycle(ops, p->opts, J - 1, true, a.solo);
  a.nops = (int)ops.size();
  if (a.solo >= 0) {
    sm_cycle(ops, p->opts, a.solo, true, -1);
    if (a.solo > 0 && a.solo < J - 1) sm_cycle(ops, p->opts, a.solo, false, -1);
  }
  a.nsolo = (int)ops.size() - a.nops;
  bool fits = false;
  switch (S->lm) {
    case 4: DCG_TRY(sm_attr<4>(S->ctas, smem, &fits)); break;
    case 6: DCG_TRY(sm_attr<6>(S->ctas, smem, &fits)); break;
    case 8: DCG_TRY(sm_attr<8>(S->ctas, smem, &fits)); break;
    case 10: DCG_TRY(sm_attr<10>(S->ctas, smem, &fits)); break;
    case 12: DCG_TRY(sm_attr<12>(S->ctas, smem, &fits)); break;
    default: DCG_TRY(sm_attr<16>(S->ctas, smem, &fits));
  }
  if (!fits) {  // the level-by-level kernels serve
    small_mg_free(p);
    return DCG_OK;
  }
  // one buffer; the state keeps the host's copy of the integers, so the copy
  // to the device needs no wait
  const size_t ntri = 2 * (size_t)m0 * m0 + m0, ndbl = ntri + 2 * kSmCtas;
  S->host = ops;
  S->host.insert(S->host.end(), boxes.begin(), boxes.end());
  S->host.push_back(0);
  DCG_CUDA(cudaMalloc(&S->buf, sizeof(double) * ndbl + sizeof(int) * S->host.size()));
  int* ints = reinterpret_cast<int*>(S->buf + ndbl);
  DCG_CUDA(cudaMemcpyAsync(ints, S->host.data(), sizeof(int) * S->host.size(), cudaMemcpyHostToDevice, s));
  k_small_tri<<<(m0 + 63) / 64, 64, 0, s>>>(m0, S->buf, S->buf + (size_t)m0 * m0, S->buf + 2 * (size_t)m0 * m0);
  DCG_LAUNCH_CHECK();
  a.ops = ints;
  for (int k = 1; k < J; ++k) a.lev[k].boxes = ints + ops.size() + box_end[k - 1];
  a.S = p->coarse.S64;
  a.tl = S->buf;
  a.tw = S->buf + (size_t)m0 * m0;
  a.te = S->buf + 2 * (size_t)m0 * m0;
  a.red = S->buf + ntri;
  a.ncyc = ints + ops.size() + boxes.size();
  return DCG_OK;
}

// Algorithm 3 on g from the iterate z: until ||g - Z z|| <= tol ||g|| or nmax
// cycles (fixed: exactly nmax); the cycle count is left on the device.
// tol_dev, total, iter, in_iter: device operands of the captured solve.
int small_mg_launch(dcg_problem* p, const double* g, double* z, bool fixed, double tol, int nmax, const double* tol_dev,
                    int* total, int* iter, const int* in_iter, cudaStream_t s) {
  SmallState* S = static_cast<SmallState*>(p->mg.small);
  SmArgs a = S->args;
  a.g = g;
  a.z = z;
  a.fixed = fixed;
  a.tol = tol;
  a.tol_dev = tol_dev;
  a.nmax = nmax;
  a.total = total;
  a.iter = iter;
  a.in_iter = in_iter;
  return sm_dispatch(*S, a, s);
}

int small_mg_cycles_done(dcg_problem* p, int* ncyc, cudaStream_t s) {
  SmallState* S = static_cast<SmallState*>(p->mg.small);
  int* host = reinterpret_cast<int*>(p->scal_host + S_COUNT - 1);  // pinned, unused slot
  DCG_CUDA(cudaMemcpyAsync(host, S->args.ncyc, sizeof(int), cudaMemcpyDeviceToHost, s));
  DCG_CUDA(cudaStreamSynchronize(s));
  *ncyc = *host;
  return DCG_OK;
}

}  // namespace dcg
