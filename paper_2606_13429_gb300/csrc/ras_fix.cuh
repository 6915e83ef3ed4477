// Device part of the FP64 smoother's exact local solves in fixed point: the
// transforms and line solves of a box, and the whole 2D box solve. What bounds
// it, the scaling and the mapping are described in ras_fix.cu.
#pragma once

#include "common.cuh"
#include "fix64.cuh"

namespace dcg {
namespace {

constexpr int fx_group(int LM) { return LM + 2 <= 8 ? 8 : LM + 2 <= 16 ? 16 : 32; }  // lanes per box, 2D
constexpr int fx_batch(int D, int LM) { return D == 2 ? 128 / fx_group(LM) : 8; }
constexpr int fx_threads(int D, int LM) { return D == 2 ? 128 : 8 * LM * LM; }
// CTAs per SM the register allocation leaves room for (12: with 6 the step from
// an iterate spills, a cycle at 1024^2 takes 334.7 us instead of 331.7)
constexpr int fx_blocks(int D, int LM) { return D == 2 ? (LM <= 8 ? 7 : LM <= 10 ? 6 : LM <= 12 ? 5 : 4) : (LM <= 4 ? 6 : 2); }
// pitch of a line of table constants (pairs are read as 16-byte loads)
__host__ __device__ constexpr int fx_hm(int LM) { return ((LM + 1) / 2 + 1) / 2 * 2; }

// forward transform of one line in place; C[j][x], x < fx_hm(LM)
template <int LM>
__device__ __forceinline__ void fx_forward(long long* __restrict__ W, int stride, int l, const int2* __restrict__ C) {
  constexpr int HM = (LM + 1) / 2, HP = fx_hm(LM);
  const int h = l >> 1, hc = (l + 1) >> 1;
  FxVal p[HP], q[HP];
#pragma unroll
  for (int x = 0; x < HP; ++x) {
    const long long a = (x < HM && x < hc) ? W[x * stride] : 0;
    const long long b = (x < HM && x < h) ? W[(l - 1 - x) * stride] : 0;
    p[x] = fx_split(a + b);
    q[x] = fx_split(a - b);
  }
  // two outputs per turn of a rolled loop: unrolled, the table loads of many
  // outputs are hoisted together and take 250 registers
#pragma unroll 1
  for (int j = 0; j < l; j += 2) {
    FxAcc e = fx_zero(), o = fx_zero();
#pragma unroll
    for (int x = 0; x < HP; x += 2) {
      const int4 ce = *reinterpret_cast<const int4*>(C + j * HP + x);
      const int4 co = *reinterpret_cast<const int4*>(C + (j + 1) * HP + x);
      fx_mac(e, p[x], ce.x, ce.y);
      fx_mac(o, q[x], co.x, co.y);
      if (x + 1 < HM) {
        fx_mac(e, p[x + 1], ce.z, ce.w);
        fx_mac(o, q[x + 1], co.z, co.w);
      }
    }
    W[j * stride] = fx_value(e);
    if (j + 1 < l) W[(j + 1) * stride] = fx_value(o);
  }
}

// transform back: out_x = sum_j C_x[j] v_j; C[x][j], x < (LM+1)/2, j < LM
// (even j, then odd j, each padded to fx_hm(LM))
template <int LM>
__device__ __forceinline__ void fx_back(long long* __restrict__ W, int stride, int l, const int2* __restrict__ C) {
  constexpr int HM = (LM + 1) / 2, HP = fx_hm(LM);
  const int h = l >> 1, hc = (l + 1) >> 1;
  FxVal v[2 * HP];
#pragma unroll
  for (int j = 0; j < 2 * HP; ++j) v[j] = fx_split((j < LM && j < l) ? W[j * stride] : 0);
#pragma unroll 1
  for (int x = 0; x < hc; ++x) {
    FxAcc e = fx_zero(), o = fx_zero();
#pragma unroll
    for (int k = 0; k < HP; k += 2) {
      const int4 ce = *reinterpret_cast<const int4*>(C + (2 * x) * HP + k);
      const int4 co = *reinterpret_cast<const int4*>(C + (2 * x + 1) * HP + k);
      fx_mac(e, v[2 * k], ce.x, ce.y);
      fx_mac(o, v[2 * k + 1], co.x, co.y);
      if (k + 1 < HM) {
        fx_mac(e, v[2 * k + 2], ce.z, ce.w);
        fx_mac(o, v[2 * k + 3], co.z, co.w);
      }
    }
    const long long E = fx_value(e), O = fx_value(o);
    W[x * stride] = E + O;
    if (x < h) W[(l - 1 - x) * stride] = E - O;
  }
}

// line solve in place. t (global or shared memory): [4][n][nl] constants of this line with pitch nl:
// -l_i; winv_i 2^-K; -b winv_i; and, for the exact extent n = LM, in entry
// [3][0] the reciprocal pivot of the meeting row.
// General extents: y_i = g_i - l_i y_{i-1}; x_i = winv_i y_i - b winv_i x_{i+1}.
// n = LM: the line is Toeplitz, so it is eliminated from both ends with the
// same factors, the two chains meeting at rows LM/2 - 1 and LM/2 (half the
// dependent steps).
template <int LM, bool EX>
__device__ __forceinline__ void fx_line_solve(long long* __restrict__ W, int n, const int2* __restrict__ t, int nl) {
  long long g[LM];
#pragma unroll
  for (int i = 0; i < LM; ++i) g[i] = (EX || i < n) ? W[i] : 0;
  if constexpr (EX) {
    constexpr int H = LM / 2;
#pragma unroll
    for (int i = 1; i < H; ++i) {
      const int2 c = t[i * nl];
      FxAcc a = fx_zero(), d = fx_zero();
      fx_mac(a, fx_split(g[i - 1]), c.x, c.y);
      fx_mac(d, fx_split(g[LM - i]), c.x, c.y);
      g[i] += fx_value(a);
      g[LM - 1 - i] += fx_value(d);
    }
    // row H with the whole upper half eliminated
    long long xa, xb;
    {
      const int2 c = t[H * nl], cm = t[3 * LM * nl];
      FxAcc a = fx_zero(), d = fx_zero();
      fx_mac(a, fx_split(g[H - 1]), c.x, c.y);
      fx_mac(d, fx_split(g[H] + fx_value(a)), cm.x, cm.y);
      xb = fx_value(d);
      W[H] = xb;
    }
    {
      const int2 cw = t[(LM + H - 1) * nl], cb = t[(2 * LM + H - 1) * nl];
      FxAcc a = fx_zero();
      fx_mac(a, fx_split(g[H - 1]), cw.x, cw.y);
      fx_mac(a, fx_split(xb), cb.x, cb.y);
      xa = fx_value(a);
      W[H - 1] = xa;
    }
#pragma unroll
    for (int i = H - 2; i >= 0; --i) {
      const int2 cw = t[(LM + i) * nl], cb = t[(2 * LM + i) * nl];
      FxAcc a = fx_zero(), d = fx_zero();
      fx_mac(a, fx_split(g[i]), cw.x, cw.y);
      fx_mac(d, fx_split(g[LM - 1 - i]), cw.x, cw.y);
      fx_mac(a, fx_split(xa), cb.x, cb.y);
      fx_mac(d, fx_split(xb), cb.x, cb.y);
      xa = fx_value(a);
      xb = fx_value(d);
      W[i] = xa;
      W[LM - 1 - i] = xb;
    }
  } else {
#pragma unroll
    for (int i = 1; i < LM; ++i)
      if (i < n) {
        const int2 c = t[i * nl];
        FxAcc a = fx_zero();
        fx_mac(a, fx_split(g[i - 1]), c.x, c.y);
        g[i] += fx_value(a);
      }
    long long xn = 0;
#pragma unroll
    for (int i = LM - 1; i >= 0; --i)
      if (i < n) {
        const int2 cw = t[(n + i) * nl], cb = t[(2 * n + i) * nl];
        FxAcc a = fx_zero();
        fx_mac(a, fx_split(g[i]), cw.x, cw.y);
        fx_mac(a, fx_split(xn), cb.x, cb.y);
        xn = fx_value(a);
        W[i] = xn;
      }
  }
}

__device__ __forceinline__ double fx_nan() { return __longlong_as_double(0x7ff8000000000000ll); }
// result of a scaled box, or of one with a non-finite entry
__device__ __forceinline__ double fx_special(long long v, int e0, unsigned mag) {
  return mag < kFxNonFinite ? fx_to_double(v, e0) * fx_two320(-fx_lift(mag)) : fx_nan();
}

// scaling of a level's boxes
struct FxScale {
  int bits, sf, kout;  // bits of the quantised residual; powers of two of the right-hand side and the results
  int2 sixth;          // 1/6
};
inline FxScale ras_fix_scale(const Level& L, bool z_zero) {
  return FxScale{z_zero ? L.fx_gb : L.fx_rb, L.fx_sf, L.fx_kout, L.fx_sixth};
}

// The residual of a 2D step is formed exactly from z and f quantised to
// kFxZBits bits below the block's largest entry (entries within 2^5 of it lose
// nothing): 6 r = 6 f + T(z), T = (sum of the 3 x 3 box) - 9 z, an integer of at
// most 22 2^58 < 2^63. It then gets an exponent of its own: a shift that takes
// its largest entry to 2^(bits + 2) at most.
constexpr int kFxZBits = 58;
__device__ __forceinline__ unsigned long long fx_abs1(long long v) { return (unsigned long long)(v ^ (v >> 63)); }
__device__ __forceinline__ int fx_length(unsigned long long any) { return 64 - __clzll((long long)any); }
__device__ __forceinline__ long long fx_res(long long v, int shift, int2 c) {
  FxAcc a = fx_zero();
  fx_mac(a, fx_split(shift >= 0 ? v << shift : v >> -shift), c.x, c.y);
  return fx_value(a);
}

// Exact solve on one 2D box by a group of fx_group(LM) lanes, all lanes of the
// warp taking part: lane `x + 1` holds column x of z (rows -1 .. ly) and f (FP64
// bits, zero outside the box or grid). W: the box's shared memory [ly][lx | 1];
// tf, tb, tri: tables of the box's class; out(q, v) receives entry (x, q).
// EX: the box has extent LM along both axes. ANY: data of any size; else at
// least 2^-831 beside the values that count (what lies below vanishes).
template <int LM, bool ZZERO, bool EX, bool ANY, typename Out>
__device__ __forceinline__ void fx_solve_2d(const FxScale& A, int lx, int ly, bool live, long long (&zv)[LM + 2],
                                            long long (&fv)[LM], long long* __restrict__ W,
                                            const int2* __restrict__ tf, const int2* __restrict__ tb,
                                            const int2* __restrict__ tri, Out&& out) {
  constexpr int G = fx_group(LM);
  const int lane = threadIdx.x & (G - 1), x = lane - 1;
  const int wp = lx | 1;
  const bool own = live && x >= 0 && x < lx;
  unsigned mag = 0;
#pragma unroll
  for (int q = 0; q < LM; ++q) mag = max(mag, fx_mag(fv[q]));
  if (!ZZERO) {
#pragma unroll
    for (int q = 0; q < LM + 2; ++q) mag = max(mag, fx_mag(zv[q]));
  }
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) mag = max(mag, __shfl_xor_sync(0xffffffffu, mag, o, G));
  const bool odd = ANY ? fx_odd(mag) : mag >= kFxNonFinite;
  int e = ANY ? (int)(mag >> 20) : max((int)(mag >> 20), kFxLowest);
  if (ANY && odd) {
    const int lift = fx_lift(mag);
    const double up = fx_two320(lift);
    e = fx_odd_exponent(mag, lift);
#pragma unroll
    for (int q = 0; q < LM; ++q) fv[q] = fx_scaled(fv[q], up);
    if (!ZZERO) {
#pragma unroll
      for (int q = 0; q < LM + 2; ++q) zv[q] = fx_scaled(zv[q], up);
    }
  }
  int e0 = e + 63 + A.kout;  // of the results, less the bits of the residual
  if (ZZERO) {
    const int sh0 = 63 - A.bits + e;
    e0 -= A.bits;
#pragma unroll
    for (int q = 0; q < LM; ++q)
      if (own && q < ly) W[q * wp + x] = fx_near(fv[q], sh0);
  } else {
    const int sh0 = 63 - kFxZBits + e;
    long long s0 = 0, s1 = 0, zm = 0;
    unsigned long long any = 0;
#pragma unroll
    for (int q = 0; q < LM + 2; ++q) {
      const long long zc = fx_near(zv[q], sh0);
      const long long s2 = __shfl_up_sync(0xffffffffu, zc, 1, G) + zc + __shfl_down_sync(0xffffffffu, zc, 1, G);
      if (q >= 2) {
        const long long r6 = (s0 + s1 + s2) - (zm << 3) - zm + fx_near(fv[q - 2], sh0) * 6;
        fv[q - 2] = r6;
        if (own && q - 2 < ly) any |= fx_abs1(r6);
      }
      s0 = s1;
      s1 = s2;
      zm = zc;
    }
    int shift = any ? fx_length(any) : 0;  // bits of the largest |6 r|
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) shift = max(shift, __shfl_xor_sync(0xffffffffu, shift, o, G));
    shift = shift ? A.bits + 2 - shift : 0;
    e0 -= kFxZBits + shift;
#pragma unroll
    for (int q = 0; q < LM; ++q)
      if (own && q < ly) W[q * wp + x] = fx_res(fv[q], shift, A.sixth);
  }
  if (own) fx_forward<LM>(W + x, wp, ly, tf);
  __syncwarp();
  if (live && lane < ly) fx_line_solve<LM, EX>(W + lane * wp, lx, tri + lane, ly);
  __syncwarp();
  if (own) {
    fx_back<LM>(W + x, wp, ly, tb);
    if (!odd) {
#pragma unroll 4
      for (int q = 0; q < ly; ++q) out(q, fx_to_double(W[q * wp + x], e0));
    } else {
      for (int q = 0; q < ly; ++q) out(q, ANY ? fx_special(W[q * wp + x], e0, mag) : fx_nan());
    }
  }
}

}  // namespace
}  // namespace dcg
