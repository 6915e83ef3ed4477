// FP64 product with the pseudo-stress operator A = (1/dt) M_dev + K_div on the
// uniform Q1 mesh, for assembled and matrix-free problems alike.
//
// A block of A couples nodes a and a + o as (1/dt) mt(a, o) D_d + kron(I_d,
// G(o)) (Section 3.1; forms of Section 3.2.1): of its 16 (2D) or 81 (3D)
// entries only the scalar mt(a, o) = sum_e nu_e^-1 int_e phi_a phi_{a+o}
// depends on a, and it comes from the 1/nu of the 4 or 8 elements around a.
// G(o) is a product of 1D factors,
//   G_pp = K along p, M along the other axes,
//   G_pq = -C along p and q (p != q), M along the third,
// K = (-1, 2, -1)/h, M = (h/6)(1, 4, 1), C = (-1, 0, 1)/2. So the product reads
// x and 1/nu, writes y, and applies 1D factors one axis after the other.
//
// What bounds it. Reading the stored blocks takes 1,256 B per node in 2D and
// 17.75 KB in 3D and was HBM bound (258 us at 1024^2; 1,216 us at 80^3); this
// form moves 72 B and 152 B and is bound by FP64 issue (2 lanes per clock per
// SM; the FP64 pipe is 82-85% busy), so its FP64 operations are what counts:
// 46 per node in 2D (68 with a viscosity per element) against 94 of the stored
// blocks, about 185 in 3D (310) against 890, and against 750 of the
// matrix-free product's unfactored 27-point stencils. Measured: 107 us at
// 1024^2, 229 us at 80^3, and with a viscosity per element 3,514 -> 1,881 us
// at 129^3 (matrix-free).
//
// Mapping, 2D: a thread walks `seg` rows of one column; the row quantities
// (sums and differences along x of the four components) slide along y.
// 3D: a warp owns 30 columns of one row of nodes (32 lanes with the halo),
// marches along z, forms the y factors from the three rows it loads, the x
// factors by shuffles (free beside the FP64 issue), and adds each plane's
// contribution to the three output planes it meets in two accumulators per
// component. M_dev V = 0 holds: the deviatoric part of equal diagonal entries
// is formed first.
#include "common.cuh"

#include <algorithm>
#include <cmath>

namespace dcg {
namespace {

enum OpX { OX_X = 0, OX_X_MINUS_VZ = 1, OX_VZ = 2 };
enum OpO { OO_Y = 0, OO_FMY = 1, OO_VT = 2, OO_YVT = 3, OO_RHS = 4 };
enum OpPart { OP_FULL = 0, OP_MASS = 1, OP_DIV = 2 };  // A, (1/dt) M_dev or K_div alone

struct OpArgs {
  const double* x;
  const double* zh;
  const double* f;       // OO_FMY: f - y; OO_RHS: y + f (+ f0)
  const double* f0;
  double* y;
  double* g;             // V^T y for OO_YVT
  const double* dvec;    // dot(dvec, y) for OO_Y
  const double* inv_nu;  // per element, or null: cmass holds the uniform value
  double cmass;          // 2D: h^2 / (36 dt) (/ nu); 3D: (h^3 / (216 dt) (/ nu)) / (h / 36)
  double scale;          // 3D: +-h / 36
  double kx, ky;         // 2D: factors of K_div, +-1/6 and +-1/4
  double isd;            // 1/sqrt(d)
  int m, n;
  int gx, gy, seg;       // 2D: column blocks, -, rows per warp; 3D: column and row blocks, planes per CTA
  int vec;               // x, f, f0, y, dvec 16-byte aligned (2D)
  Reduce red;
};

// ---------------------------------------------------------------------------
// 2D
// ---------------------------------------------------------------------------
constexpr int kOp2Threads = 128;

__device__ __forceinline__ void op_load4(const double* p, bool vec, double (&v)[4]) {
  if (vec) {
    const double2 a = __ldg(reinterpret_cast<const double2*>(p)), b = __ldg(reinterpret_cast<const double2*>(p) + 1);
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
  } else {
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = __ldg(p + c);
  }
}

template <int XM>
__device__ __forceinline__ void op_operand2(const OpArgs& A, bool in, int a, double (&v)[4]) {
  v[0] = v[1] = v[2] = v[3] = 0.0;
  if (!in) return;
  if (XM != OX_VZ) op_load4(A.x + 4LL * a, A.vec, v);
  if (XM != OX_X) {
    const double q = __dmul_rn(A.isd, __ldg(A.zh + a));
    if (XM == OX_VZ) {
      v[0] = q;
      v[3] = q;
    } else {
      v[0] = __dsub_rn(v[0], q);
      v[3] = __dsub_rn(v[3], q);
    }
  }
}

// row quantities of one column: stiffness k, mass m and difference c along x
// of the components (0, 1, 2, 3 = xx, xy, yx, yy), and those of the mass part:
// uniform viscosity M1 of e = x_0 - x_3 and component 2 (component 1's is m1);
// per element the left and right element sums l + 2c, r + 2c of e/2, 1 and 2
template <bool VAR>
struct OpRow2 {
  double k0, c0, m1, c1, k2, c2, m3, c3;
  double q[VAR ? 6 : 2];
};

template <int XM, bool VAR>
__device__ __forceinline__ void op_row2(const OpArgs& A, int x, int y, OpRow2<VAR>& R) {
  const int m = A.m;
  const bool in = y >= 0 && y < m && x < m;
  double l[4], c[4], r[4];
  const int a = x + m * y;
  op_operand2<XM>(A, in && x > 0, a - 1, l);
  op_operand2<XM>(A, in, a, c);
  op_operand2<XM>(A, in && x + 1 < m, a + 1, r);
  const double u0 = l[0] + r[0], u1 = l[1] + r[1], u2 = l[2] + r[2], u3 = l[3] + r[3];
  R.k0 = fma(2.0, c[0], -u0);
  R.c0 = r[0] - l[0];
  R.m1 = fma(4.0, c[1], u1);
  R.c1 = r[1] - l[1];
  R.k2 = fma(2.0, c[2], -u2);
  R.c2 = r[2] - l[2];
  R.m3 = fma(4.0, c[3], u3);
  R.c3 = r[3] - l[3];
  const double ec = c[0] - c[3];
  if (VAR) {
    const double el = l[0] - l[3], er = r[0] - r[3];
    R.q[0] = fma(0.5, el, ec);  // halves of e: (l + 2c) / 2
    R.q[1] = fma(0.5, er, ec);
    R.q[2] = fma(2.0, c[1], l[1]);
    R.q[3] = fma(2.0, c[1], r[1]);
    R.q[4] = fma(2.0, c[2], l[2]);
    R.q[5] = fma(2.0, c[2], r[2]);
  } else {
    // deviatoric entries first: exactly zero when x_0 = x_3
    R.q[0] = fma(4.0, ec, (l[0] - l[3]) + (r[0] - r[3]));
    R.q[1] = fma(4.0, c[2], u2);
  }
}

template <int XM, int OM, bool DOT, bool VAR, int PART = OP_FULL>
__global__ void __launch_bounds__(kOp2Threads) k_op2(OpArgs A) {
  constexpr bool MASS = XM != OX_VZ && OM != OO_VT && PART != OP_DIV;  // M_dev V = 0 and V^T M_dev = 0
  double part[1] = {0.0};
  const int w = blockIdx.x * (kOp2Threads / 32) + (threadIdx.x >> 5);  // warp: 32 columns x seg rows
  const int wy = w / A.gx;
  const int x = (w - wy * A.gx) * 32 + (threadIdx.x & 31);
  const int m = A.m;
  const int y0 = wy * A.seg, y1 = min(y0 + A.seg, m);
  if (x < m && y0 < m) {
    OpRow2<VAR> P, Q, N;  // rows y - 1, y, y + 1
    op_row2<XM, VAR>(A, x, y0 - 1, P);
    op_row2<XM, VAR>(A, x, y0, Q);
    double wl = 0.0, wr = 0.0;  // weights of the two elements below row y
    if (MASS && VAR) {
      const double* e = A.inv_nu + x + A.n * y0;
      wl = A.cmass * __ldg(e);
      wr = A.cmass * __ldg(e + 1);
    }
    const double axx = OM == OO_RHS ? A.kx : 1.0 / 6.0, axy = OM == OO_RHS ? A.ky : 0.25;
    for (int y = y0; y < y1; ++y) {
      op_row2<XM, VAR>(A, x, y + 1, N);
      double o[4] = {0.0, 0.0, 0.0, 0.0};
      if (PART != OP_MASS) {
        o[0] = fma(axy, P.c1 - N.c1, axx * fma(4.0, Q.k0, P.k0 + N.k0));
        o[1] = fma(axy, P.c0 - N.c0, axx * fma(2.0, Q.m1, -(P.m1 + N.m1)));
        o[2] = fma(axy, P.c3 - N.c3, axx * fma(4.0, Q.k2, P.k2 + N.k2));
        o[3] = fma(axy, P.c2 - N.c2, axx * fma(2.0, Q.m3, -(P.m3 + N.m3)));
      }
      // (1/dt) M_dev
      if (MASS && VAR) {
        const double* e = A.inv_nu + x + A.n * (y + 1);
        const double vl = A.cmass * __ldg(e), vr = A.cmass * __ldg(e + 1);
        const double cl = wl + vl, cr = wr + vr;
        const double dl = cl + cl, dr = cr + cr;  // exact doubling
        double M[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          double s = wl * P.q[2 * k];
          s = fma(wr, P.q[2 * k + 1], s);
          s = fma(dl, Q.q[2 * k], s);
          s = fma(dr, Q.q[2 * k + 1], s);
          s = fma(vl, N.q[2 * k], s);
          M[k] = fma(vr, N.q[2 * k + 1], s);
        }
        o[0] += M[0];
        o[3] -= M[0];
        o[1] += M[1];
        o[2] += M[2];
        wl = vl;
        wr = vr;
      } else if (MASS) {
        const double ch = 0.5 * A.cmass;
        const double Me = fma(4.0, Q.q[0], P.q[0] + N.q[0]);
        o[0] = fma(ch, Me, o[0]);
        o[3] = fma(-ch, Me, o[3]);
        o[1] = fma(A.cmass, fma(4.0, Q.m1, P.m1 + N.m1), o[1]);
        o[2] = fma(A.cmass, fma(4.0, Q.q[1], P.q[1] + N.q[1]), o[2]);
      }
      const int a = x + m * y;
      if (OM == OO_VT) {
        const double g = (o[0] + o[3]) * A.isd;
        A.y[a] = g;
        if (DOT) part[0] = fma(g, g, part[0]);
      } else {
        if (OM == OO_FMY) {
          double fv[4];
          op_load4(A.f + 4LL * a, A.vec, fv);
#pragma unroll
          for (int c = 0; c < 4; ++c) o[c] = fv[c] - o[c];
        }
        if (OM == OO_RHS) {
          double fv[4];
          op_load4(A.f + 4LL * a, A.vec, fv);
#pragma unroll
          for (int c = 0; c < 4; ++c) o[c] += fv[c];
          if (A.f0) {
            op_load4(A.f0 + 4LL * a, A.vec, fv);
#pragma unroll
            for (int c = 0; c < 4; ++c) o[c] += fv[c];
          }
        }
        double* yp = A.y + 4LL * a;
        if (A.vec) {
          reinterpret_cast<double2*>(yp)[0] = make_double2(o[0], o[1]);
          reinterpret_cast<double2*>(yp)[1] = make_double2(o[2], o[3]);
        } else {
#pragma unroll
          for (int c = 0; c < 4; ++c) yp[c] = o[c];
        }
        if (OM == OO_YVT) {
          const double g = (o[0] + o[3]) * A.isd;
          A.g[a] = g;
          if (DOT) part[0] = fma(g, g, part[0]);
        } else if (DOT) {
          double dv[4];
          if (OM == OO_FMY) {
#pragma unroll
            for (int c = 0; c < 4; ++c) dv[c] = o[c];
          } else {
            op_load4(A.dvec + 4LL * a, A.vec, dv);
          }
#pragma unroll
          for (int c = 0; c < 4; ++c) part[0] = fma(dv[c], o[c], part[0]);
        }
      }
      P = Q;
      Q = N;
    }
  }
  if (DOT) grid_reduce<1>(part, A.red);
}

// ---------------------------------------------------------------------------
// 3D
// ---------------------------------------------------------------------------
constexpr int kOp3Rows = 4;            // rows of nodes (warps) per CTA
constexpr int kOp3Threads = 32 * kOp3Rows;

template <int XM>
__device__ __forceinline__ double op_operand3(const OpArgs& A, bool in, long long a, int c) {
  if (!in) return 0.0;
  const bool diag = (c & 3) == 0;
  if (XM == OX_X) return __ldg(A.x + a * 9 + c);
  if (XM == OX_VZ) return diag ? A.isd * __ldg(A.zh + a) : 0.0;
  const double v = __ldg(A.x + a * 9 + c);
  return diag ? v - A.isd * __ldg(A.zh + a) : v;
}

__device__ __forceinline__ double lane_l(double v) { return __shfl_up_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ double lane_r(double v) { return __shfl_down_sync(0xffffffffu, v, 1); }

// The rows k in [K0, K1) of the tensor (components k*3 .. k*3 + 2) of one
// block's nodes. All three: the uniform-viscosity mass part of the diagonal
// components is made deviatoric after its y and x factors; one alone (or with
// a viscosity per element): the deviatoric operand is formed first.
template <int XM, int OM, bool DOT, bool VAR, int K0, int K1, int PART>
__device__ __forceinline__ double op3_rows(const OpArgs& A, int block) {
  constexpr bool RAW = VAR || K1 - K0 < 3;  // deviatoric operand first
  constexpr bool MASS = XM != OX_VZ && OM != OO_VT && PART != OP_DIV;  // M_dev V = 0 and V^T M_dev = 0
  constexpr bool DIV = PART != OP_MASS;
  constexpr double third = 1.0 / 3.0;
  double part[1] = {0.0};
  const int lane = threadIdx.x & 31, row = threadIdx.x >> 5;
  const int m = A.m;
  int b = block;
  const int bx = b % A.gx;
  b /= A.gx;
  const int by = b % A.gy, bz = b / A.gy;
  const int x = bx * 30 + lane - 1, y = by * kOp3Rows + row;
  const int z0 = bz * A.seg, z1 = min(m, z0 + A.seg);
  const bool colin = x >= 0 && x < m;
  const bool own = colin && y < m && lane >= 1 && lane <= 30;
  const long long mm = (long long)m * m;
  // first[c], next[c]: what the planes so far give the outputs z - 1 and z
  double first[9], next[9];
#pragma unroll
  for (int c = 0; c < 9; ++c) first[c] = next[c] = 0.0;
  // weights of the elements between node planes z - 1 and z (index sx + 2 sy),
  // zero-padded rows and planes take any valid element
  const int ex0 = min(max(x, 0), m - 1), ey0 = min(y, m - 1);
  auto weights = [&](int z, double (&w)[4]) {
    const long long e = ex0 + (long long)A.n * (ey0 + (long long)A.n * min(max(z, 0), m));
    w[0] = A.cmass * __ldg(A.inv_nu + e);
    w[1] = A.cmass * __ldg(A.inv_nu + e + 1);
    w[2] = A.cmass * __ldg(A.inv_nu + e + A.n);
    w[3] = A.cmass * __ldg(A.inv_nu + e + A.n + 1);
  };
  double wlo[4], whi[4];
  if (VAR && MASS) weights(z0 - 1, wlo);
  for (int z = z0 - 1; z <= z1; ++z) {
    const bool zin = z >= 0 && z < m;
    const long long a = x + (long long)m * y + mm * z;
    const bool in0 = zin && colin && y < m, inm = zin && colin && y > 0 && y - 1 < m, inp = zin && colin && y + 1 < m;
    const bool done = z > z0 && own;  // output z - 1 is completed by this plane
    const long long ao = a - mm;
    if (VAR && MASS) weights(z + 1, whi);
    // deviatoric diagonal entries of the three rows, exactly zero where the
    // diagonal entries agree
    double dev[3][3];
    if (RAW && MASS) {
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        const bool in = r == 0 ? inm : r == 1 ? in0 : inp;
        const long long ar = a + (r - 1) * m;
        const double v0 = op_operand3<XM>(A, in, ar, 0), v4 = op_operand3<XM>(A, in, ar, 4),
                     v8 = op_operand3<XM>(A, in, ar, 8);
        dev[r][0] = third * fma(2.0, v0, -(v4 + v8));
        dev[r][1] = third * fma(2.0, v4, -(v0 + v8));
        dev[r][2] = -(dev[r][0] + dev[r][1]);
      }
    }
    double od[3] = {0.0, 0.0, 0.0};  // completed diagonal components
    // plane z adds t1 to output z - 1, t0 to z and t2 to z + 1
    auto finish = [&](int c, double t1, double t0, double t2) {
      const double o = A.scale * (first[c] + t1);
      first[c] = next[c] + t0;
      next[c] = t2;
      if ((c & 3) == 0) od[c >> 2] = o;
      if (OM == OO_VT || !done) return;
      double v = o;
      if (OM == OO_FMY) v = A.f[ao * 9 + c] - v;
      if (OM == OO_RHS) {
        v += A.f[ao * 9 + c];
        if (A.f0) v += A.f0[ao * 9 + c];
      }
      A.y[ao * 9 + c] = v;
      if (DOT && OM != OO_YVT) part[0] = OM == OO_FMY ? fma(v, v, part[0]) : fma(A.dvec[ao * 9 + c], v, part[0]);
    };
    // uniform viscosity: 36 M M of the diagonal components in the plane and
    // their K_div contributions, completed after the loop over k
    double F[3], d1[3], d0[3], d2[3];
#pragma unroll
    for (int k = K0; k < K1; ++k) {
      double vd[3], vc[3], vu[3];
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        vd[q] = op_operand3<XM>(A, inm, a - m, k * 3 + q);
        vc[q] = op_operand3<XM>(A, in0, a, k * 3 + q);
        vu[q] = op_operand3<XM>(A, inp, a + m, k * 3 + q);
      }
      // factors along y (C as lower - upper)
      const double s0 = vd[0] + vu[0], s1 = vd[1] + vu[1], s2 = vd[2] + vu[2];
      const double Ma = fma(4.0, vc[0], s0), Ca = vd[0] - vu[0];
      const double Kb = fma(2.0, vc[1], -s1), Cb = vd[1] - vu[1];
      const double Mc = fma(4.0, vc[2], s2), Cc = vd[2] - vu[2];
      // factors along x (C as upper - lower)
      const double Mal = lane_l(Ma), Mar = lane_r(Ma), uMa = Mal + Mar;
      const double Cbl = lane_l(Cb), Cbr = lane_r(Cb);
      const double Mcl = lane_l(Mc), Mcr = lane_r(Mc), uMc = Mcl + Mcr;
      double Ax = DIV ? fma(1.5, Cbr - Cbl, fma(2.0, Ma, -uMa)) : 0.0;
      const double Bx = Mcr - Mcl;
      double Ay = DIV ? fma(1.5, lane_r(Ca) - lane_l(Ca), fma(4.0, Kb, lane_l(Kb) + lane_r(Kb))) : 0.0;
      const double By = fma(4.0, Cc, lane_l(Cc) + lane_r(Cc));
      const double Dz = fma(4.0, Mc, uMc);
      const double Bz = (Mar - Mal) - fma(4.0, Cb, Cbl + Cbr);
      // Factors along z. In the component (k, p) with p = x, y the z
      // difference is upper - lower, in (k, z) lower - upper; plane z is the
      // upper one for output z - 1 and the lower one for output z + 1.
      if (MASS && !VAR) {
        const double Mb = fma(4.0, vc[1], s1);
        const double Fa = fma(4.0, Ma, uMa), Fb = fma(4.0, Mb, lane_l(Mb) + lane_r(Mb));
        if (RAW) {
          const double Md = fma(4.0, dev[1][k], dev[0][k] + dev[2][k]);
          F[k] = fma(4.0, Md, lane_l(Md) + lane_r(Md));
        } else {
          F[k] = k == 0 ? Fa : k == 1 ? Fb : Dz;
        }
        if (k != 0 || RAW) Ax = fma(A.cmass, k == 0 ? F[k] : Fa, Ax);
        if (k != 1 || RAW) Ay = fma(A.cmass, k == 1 ? F[k] : Fb, Ay);
      }
      double t1[3], t0[3], t2[3];
      t1[0] = DIV ? fma(-1.5, Bx, Ax) : Ax;
      t2[0] = DIV ? fma(1.5, Bx, Ax) : Ax;
      t0[0] = 4.0 * Ax;
      t1[1] = DIV ? fma(1.5, By, Ay) : Ay;
      t2[1] = DIV ? fma(-1.5, By, Ay) : Ay;
      t0[1] = 4.0 * Ay;
      t1[2] = DIV ? fma(-1.5, Bz, -Dz) : 0.0;
      t2[2] = DIV ? fma(1.5, Bz, -Dz) : 0.0;
      t0[2] = DIV ? Dz + Dz : 0.0;
      if (MASS && !VAR && (k != 2 || RAW)) {
        const double v = A.cmass * (k == 2 ? F[k] : Dz);
        t1[2] += v;
        t0[2] = fma(4.0, v, t0[2]);
        t2[2] += v;
      }
      if (MASS && VAR) {
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const double cd = q == k ? dev[0][k] : vd[q], cc = q == k ? dev[1][k] : vc[q],
                       cu = q == k ? dev[2][k] : vu[q];
          const double lo = fma(2.0, cc, cd), up = fma(2.0, cc, cu);  // element rows below and above
          const double ll = fma(2.0, lo, lane_l(lo)), lr = fma(2.0, lo, lane_r(lo));
          const double ul = fma(2.0, up, lane_l(up)), ur = fma(2.0, up, lane_r(up));
          const double G1 = fma(wlo[3], ur, fma(wlo[2], ul, fma(wlo[1], lr, wlo[0] * ll)));
          const double G2 = fma(whi[3], ur, fma(whi[2], ul, fma(whi[1], lr, whi[0] * ll)));
          t1[q] += G1;
          t0[q] = fma(2.0, G1 + G2, t0[q]);
          t2[q] += G2;
        }
      }
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        if (MASS && !RAW && q == k) {
          d1[k] = t1[q];
          d0[k] = t0[q];
          d2[k] = t2[q];
        } else {
          finish(k * 3 + q, t1[q], t0[q], t2[q]);
        }
      }
    }
    if (MASS && !RAW) {
      // the deviatoric part of the diagonal, exactly zero where F agrees
      const double cm3 = A.cmass * third;
      const double v0 = cm3 * fma(2.0, F[0], -(F[1] + F[2])), v1 = cm3 * fma(2.0, F[1], -(F[0] + F[2]));
      const double v[3] = {v0, v1, -(v0 + v1)};
#pragma unroll
      for (int k = 0; k < 3; ++k) finish(4 * k, d1[k] + v[k], fma(4.0, v[k], d0[k]), d2[k] + v[k]);
    }
    if ((OM == OO_VT || OM == OO_YVT) && done) {
      const double g = A.isd * (od[0] + od[1] + od[2]);
      if (OM == OO_VT) A.y[ao] = g;
      else A.g[ao] = g;
      if (DOT) part[0] = fma(g, g, part[0]);
    }
    if (VAR && MASS) {
#pragma unroll
      for (int s = 0; s < 4; ++s) wlo[s] = whi[s];
    }
  }
  return part[0];
}

template <int XM, int OM, bool DOT, bool VAR, int PART = OP_FULL>
__global__ void __launch_bounds__(kOp3Threads) k_op3(OpArgs A) {
  double part[1] = {op3_rows<XM, OM, DOT, VAR, 0, 3, PART>(A, blockIdx.x)};
  if (DOT) grid_reduce<1>(part, A.red);
}

// one row of the tensor per block: a third of the FP64 chain per warp, for
// grids too small to fill the GPU (outputs y and f - y only)
template <int XM, int OM, bool DOT, bool VAR, int PART = OP_FULL>
__global__ void __launch_bounds__(kOp3Threads) k_op3_split(OpArgs A) {
  const int b = blockIdx.x / 3;
  double part[1];
  switch (blockIdx.x - 3 * b) {
    case 0: part[0] = op3_rows<XM, OM, DOT, VAR, 0, 1, PART>(A, b); break;
    case 1: part[0] = op3_rows<XM, OM, DOT, VAR, 1, 2, PART>(A, b); break;
    default: part[0] = op3_rows<XM, OM, DOT, VAR, 2, 3, PART>(A, b);
  }
  if (DOT) grid_reduce<1>(part, A.red);
}

template <int XM, int OM, bool DOT, int PART = OP_FULL>
int op_launch(dcg_problem* p, OpArgs a, cudaStream_t s) {
  if (p->dim == 2) {
    a.gx = (a.m + 31) / 32;
    // rows per warp: a walk of s rows forms s + 2 rows' quantities (about 26
    // operations each, 33 with a viscosity per element) and s outputs (20, 35);
    // the warps share 608 schedulers, and one warp alone on a scheduler
    // leaves latency uncovered (taken as 1.3 times the time)
    double best = 1e300;
    for (int q = 1; q <= 32 && q <= a.m; ++q) {
      const long long per = ((long long)a.gx * ((a.m + q - 1) / q) + 607) / 608;
      const double t = (double)per * (a.inv_nu ? 33.0 * (q + 2) + 35.0 * q : 26.0 * (q + 2) + 20.0 * q) *
                       (per == 1 ? 1.3 : 1.0);
      if (t < best) {
        best = t;
        a.seg = q;
      }
    }
    constexpr int kWarps = kOp2Threads / 32;
    auto ctas = [&]() { return ((long long)a.gx * ((a.m + a.seg - 1) / a.seg) + kWarps - 1) / kWarps; };
    while (DOT && ctas() > kMaxRedCtas) a.seg *= 2;
    const unsigned g = (unsigned)ctas();
    if (a.inv_nu && PART != OP_DIV) k_op2<XM, OM, DOT, true, PART><<<g, kOp2Threads, 0, s>>>(a);
    else k_op2<XM, OM, DOT, false, PART><<<g, kOp2Threads, 0, s>>>(a);
  } else {
    a.gx = (a.m + 29) / 30;
    a.gy = (a.m + kOp3Rows - 1) / kOp3Rows;
    const long long cols = (long long)a.gx * a.gy;
    const long long cap = DOT ? (long long)kMaxRedCtas : (1LL << 31) - 1;
    if (cols > cap) {
      set_error_msg("operator product: grid too large for the fused reduction");
      return DCG_ERR_UNSUPPORTED;
    }
    // z chunks, and one row of the tensor per CTA or all three: a CTA's time is
    // its planes plus two halo planes (0.4 of it for one row), an SM's the sum
    // over its CTAs; a single CTA per SM leaves latency uncovered (taken as 1.3
    // times the time). Split at 19^3: 2 planes per CTA instead of 4.
    long long nz = 1;
    bool split = false;
    double best = 1e300;
    constexpr bool kSplit = OM == OO_Y || OM == OO_FMY || OM == OO_RHS;
    for (int sp = 0; sp < (kSplit ? 2 : 1); ++sp)
      for (long long q = 1; q <= a.m && cols * q * (sp ? 3 : 1) <= cap; ++q) {
        const long long per = (cols * q * (sp ? 3 : 1) + 151) / 152, seg = (a.m + q - 1) / q;
        const double t = (double)(per * (seg + 2)) * (per == 1 ? 1.3 : 1.0) * (sp ? 0.4 : 1.0);
        if (t < best) {
          best = t;
          nz = q;
          split = sp;
        }
      }
    a.seg = (int)((a.m + nz - 1) / nz);
    const unsigned g = (unsigned)(cols * ((a.m + a.seg - 1) / a.seg));
    if constexpr (kSplit) {
      if (split) {
        if (a.inv_nu && PART != OP_DIV) k_op3_split<XM, OM, DOT, true, PART><<<3 * g, kOp3Threads, 0, s>>>(a);
        else k_op3_split<XM, OM, DOT, false, PART><<<3 * g, kOp3Threads, 0, s>>>(a);
        DCG_LAUNCH_CHECK();
        return DCG_OK;
      }
    }
    if (a.inv_nu && PART != OP_DIV) k_op3<XM, OM, DOT, true, PART><<<g, kOp3Threads, 0, s>>>(a);
    else k_op3<XM, OM, DOT, false, PART><<<g, kOp3Threads, 0, s>>>(a);
  }
  DCG_LAUNCH_CHECK();
  return DCG_OK;
}

}  // namespace

namespace {
OpArgs op_args(dcg_problem* p, const OpCall& c) {
  OpArgs a{};
  a.x = c.x;
  a.zh = c.zh;
  a.f = c.f;
  a.y = c.y;
  a.g = c.g;
  a.dvec = c.dvec;
  a.inv_nu = p->inv_nu_elem;
  const double h = 1.0 / p->n, w = (a.inv_nu ? 1.0 : 1.0 / p->nu) / p->dt;
  a.cmass = p->dim == 2 ? h * h / 36.0 * w : h * h / 6.0 * w;
  a.scale = h / 36.0;
  a.kx = 1.0 / 6.0;
  a.ky = 0.25;
  a.isd = 1.0 / std::sqrt((double)p->dim);
  a.m = p->m;
  a.n = p->n;
  a.vec = (!c.x || aligned16(c.x)) && aligned16(c.y) && (!c.f || aligned16(c.f)) && (!c.dvec || aligned16(c.dvec));
  return a;
}
}  // namespace

// y = K_div x
int op_div(dcg_problem* p, const double* x, double* y, cudaStream_t s) {
  OpCall c;
  c.x = x;
  c.y = y;
  return op_launch<OX_X, OO_Y, false, OP_DIV>(p, op_args(p, c), s);
}

// y = (1/dt) M_dev w + f (+ f0), or with `minus_div` ((1/dt) M_dev - K_div) w +
// f (+ f0): one pass instead of the products A w and K_div w, their difference
// and the loads (700^2, Crank-Nicolson, a viscosity per element: 230 -> 84 us,
// and no scratch). w must not overlap y.
int op_time_rhs(dcg_problem* p, bool minus_div, const double* w, const double* f, const double* f0, double* y,
                cudaStream_t s) {
  OpCall c;
  c.x = w;
  c.f = f;
  c.y = y;
  OpArgs a = op_args(p, c);
  a.f0 = f0;
  a.vec = a.vec && (!f0 || aligned16(f0));
  if (!minus_div) return op_launch<OX_X, OO_RHS, false, OP_MASS>(p, a, s);
  a.kx = -a.kx;
  a.ky = -a.ky;
  a.scale = -a.scale;  // 3D: -(h/36) (K - mass)
  if (p->dim == 3) a.cmass = -a.cmass;
  return op_launch<OX_X, OO_RHS, false>(p, a, s);
}

// y = A x in FP64. Operand x (zh null), x - V zh, or V zh (x null, with f or vt);
// output y, f - y (f given), V^T y (vt), or y and g = V^T y (g given). slot: the sum
// of squares of the output (of g when it is formed), or with dvec (dvec, y);
// y = A x alone may go without (slot < 0).
int op_product(dcg_problem* p, const OpCall& c, cudaStream_t s) {
  OpArgs a = op_args(p, c);
  if (c.slot >= 0) a.red = make_reduce(p, c.slot);
  // algorithmic work: FP64 instructions of the factored form per node, each
  // counted as a multiply-add (V^T y forms the diagonal components alone),
  // and the vectors and 1/nu
  const double N = (double)p->N, nn = (double)p->n_nodes;
  const double ops = (p->dim == 2 ? (a.inv_nu ? 68.0 : 46.0) : (a.inv_nu ? 310.0 : 185.0)) *
                     (!c.vt ? 1.0 : p->dim == 2 ? 0.6 : 0.45);
  double bytes = 8.0 * ((c.x ? N : 0.0) + (c.zh ? nn : 0.0) + (c.vt ? nn : N) + (c.g ? nn : 0.0) + (c.f ? N : 0.0) +
                        (c.dvec && c.dvec != c.x ? N : 0.0) + (a.inv_nu ? nn : 0.0));
  const int prof = prof_begin(p, PC_SPMV, s);
  int st;
  if (c.x && !c.zh) {
    if (c.vt) st = op_launch<OX_X, OO_VT, true>(p, a, s);
    else if (c.g) st = op_launch<OX_X, OO_YVT, true>(p, a, s);
    else if (c.f) st = op_launch<OX_X, OO_FMY, true>(p, a, s);
    else if (c.slot >= 0) st = op_launch<OX_X, OO_Y, true>(p, a, s);
    else st = op_launch<OX_X, OO_Y, false>(p, a, s);
  } else if (c.x) {
    st = op_launch<OX_X_MINUS_VZ, OO_Y, true>(p, a, s);
  } else if (c.vt) {
    st = op_launch<OX_VZ, OO_VT, true>(p, a, s);
  } else {
    st = op_launch<OX_VZ, OO_FMY, true>(p, a, s);
  }
  DCG_TRY(st);
  prof_end(p, prof, s, 2.0 * ops * nn, bytes);
  return DCG_OK;
}

}  // namespace dcg
