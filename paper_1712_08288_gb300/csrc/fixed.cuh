// fixed.cuh -- the MRT collision of FP64 storage in 64-bit block fixed point.
//
// Why: the FP64 pipe of this GPU issues one warp instruction in 64 cycles per quarter of
// an SM (about 1.25 TFLOP/s in all), the integer pipe one in one or two.  A collision is
// some 200 additions, small integer multiples and two dozen products; in FP64 that work,
// not memory, bounds the sweep.  Here the Q deviations of a node are aligned to
// the exponent of the largest of them and held as 64-bit integers, so that an addition is
// two integer instructions and exact.  D3Q19, 32 nodes on one SM: 3413 cycles in FP64, 471
// here (1216 instructions, 19 of them conversions on the FP64 pipe); D2Q9 1364 and 212.
// The D3Q19 pipe at L = 128: 546 us a step in FP64, 164 with this collision alone.  Error
// of a step against extended precision, rms in half ulps of the node's largest deviation
// (rounding the result once is 0.28 to 0.33 of that), FP64 form with fused multiply-adds and
// here, at s_nu 0.5 to 1.9 and the workloads' other rates: D2Q9 0.45-0.77 and 0.34-0.36,
// D3Q15 0.41-0.61 and 0.37-0.40, D3Q19 0.68-0.73 and 0.38-0.44.  Where every rate is far below
// 1 the FP64 form subtracts little and rounds little: all rates 0.05, D3Q15 0.28 and 0.43.
//
// Number form.  With E the largest exponent among the node's deviations and the force,
// value = v 2^(E - top) with top = 56 (57 for D2Q9): the largest |v| is below 2^(top+1),
// one unit is 1/16 (1/32) of an ulp of the largest deviation.  Deviations within that
// factor of the largest are held exactly; the bits a smaller one loses are replaced by
// half a unit (the middle of what they could be), so that no sum is biased.  Sums and the
// back-transform are exact, a product is cut to one unit, centred, and the result is
// rounded once to FP64.  Mass and momentum change only by the roundings at the two ends:
// the rows of M are orthogonal in integers too.  The FP64 form rounds every partial sum.
//
// Range.  The bounds below hold for deviations under rho0/16 (and under 2^15, where a
// density cannot pass the runaway limit of 1e6); a node outside that range, with a
// non-finite entry, or with all entries under 2^-895 takes the FP64 form, so any input
// gives what it gave (values that all lie below 2^-1042 count as a node at rest), and so
// do contexts without a relaxed row (every s_k = 0), whose advection is exact.  With g the
// largest deviation, |j_a| <= 10 g and j_a j_b / rho0 <= 6.3 g (D2Q9: 6 g and 2.3 g), every
// sum given to fx_mul is below 45 g (D2Q9: 25 g) and every result below 55 g (D2Q9: 16 g):
// all within 64 bits.
#pragma once

#include <math.h>
#include <string.h>

#include "common.cuh"
#include "moments.cuh"

namespace lbm {

typedef long long i64;
typedef unsigned long long u64;

// bit position of the largest deviation's leading bit
template <class L>
constexpr int kFxTop = L::Q == 9 ? 57 : 56;
constexpr int kFxMinExp = 128;  // smallest biased exponent of a block

// right shifts whose amount may exceed 63 (result 0, or -1 for negative x); the hardware clamps
LBM_HD u64 fx_shr(u64 x, int n) {
#ifdef __CUDA_ARCH__
  u64 r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));
  return r;
#else
  return n > 63 ? 0 : x >> n;
#endif
}
LBM_HD i64 fx_sar(i64 x, int n) {
#ifdef __CUDA_ARCH__
  i64 r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));
  return r;
#else
  return n > 63 ? (x < 0 ? -1 : 0) : x >> n;
#endif
}
LBM_HD int fx_hi(double x) {
#ifdef __CUDA_ARCH__
  return __double2hiint(x);
#else
  i64 b;
  memcpy(&b, &x, 8);
  return (int)(b >> 32);
#endif
}
LBM_HD unsigned fx_lo(double x) {
#ifdef __CUDA_ARCH__
  return (unsigned)__double2loint(x);
#else
  i64 b;
  memcpy(&b, &x, 8);
  return (unsigned)b;
#endif
}

// x as a multiple of 2^(E - 1023 - top), E at least x's biased exponent
template <int kTop>
LBM_HD i64 fx_from(double x, int E) {
  const int hi = fx_hi(x);
  const unsigned lo = fx_lo(x);
  const int d = E - ((hi >> 20) & 0x7ff);
  const u64 m = (((u64)(unsigned)hi << 32) | lo) << (kTop - 52);
  const u64 top = (m & ((1ull << kTop) - 1)) | (1ull << kTop);
  u64 v = fx_shr(top, d);
  if ((unsigned)(d - (kTop - 51)) < 55u) v |= 1ull;   // bits were lost: the middle of the interval
  const i64 s = (i64)(hi >> 31);
  return ((i64)v ^ s) - s;
}

// v 2^(E - 1023 - top), rounded to nearest
template <int kTop>
LBM_HD double fx_to(i64 v, int E) {
  const double x = (double)v;
#ifdef __CUDA_ARCH__
  const int hi = __double2hiint(x);       // 0 only for x = 0
  return __hiloint2double(hi != 0 ? hi + ((E - 1023 - kTop) << 20) : 0, __double2loint(x));
#else
  return v != 0 ? ldexp(x, E - 1023 - kTop) : 0.0;
#endif
}

// (v c) >> 64 for 0 <= c <= 2^62, |v| < 2^62.9, without the product of the low halves; the
// cut is centred (+-0.75 units).  Three wide multiply-adds and a shift.
LBM_HD i64 fx_mul(i64 v, FixedCoef c) {
  const int ah = (int)(v >> 32);
  const unsigned al = (unsigned)v;
  const i64 t = (i64)ah * c.lo + (i64)((u64)al * (unsigned)c.hi) + (i64)0xc0000000ll;
  return (i64)ah * c.hi + (t >> 32);
}

// a factor of a runtime product in halves with a signed low half
struct FxHalves {
  int hi, lo;
};
LBM_HD FxHalves fx_halves(i64 v) {
  const int lo = (int)(unsigned)v;
  return {(int)(v >> 32) + (int)((unsigned)lo >> 31), lo};
}
LBM_HD i64 fx_mul(FxHalves a, FxHalves b) {
  const i64 t = (i64)a.hi * b.lo + (i64)a.lo * b.hi + (i64)0x80000000ll;
  return (i64)a.hi * b.hi + (t >> 32);
}

// j_a j_b / rho0 for the components of the momentum, in the block's units
template <int D>
struct FxQuad {
  i64 xx, yy, zz, xy, yz, xz;
  LBM_HD FxQuad(i64 jx, i64 jy, i64 jz, int E, const FixedArgs &fx) {
    const int sh = fx.quad_shift - E;      // >= 0: the range rule bounds E by rho0's exponent
    const FxHalves x = fx_halves(jx << 2), y = fx_halves(jy << 2);
    const FxHalves rx = fx_halves(fx_mul(jx << 2, fx.inv_rho0) << 2), ry = fx_halves(fx_mul(jy << 2, fx.inv_rho0) << 2);
    xx = fx_sar(fx_mul(rx, x), sh);
    yy = fx_sar(fx_mul(ry, y), sh);
    xy = fx_sar(fx_mul(rx, y), sh);
    zz = yz = xz = 0;
    if (D == 3) {
      const FxHalves z = fx_halves(jz << 2), rz = fx_halves(fx_mul(jz << 2, fx.inv_rho0) << 2);
      zz = fx_sar(fx_mul(rz, z), sh);
      yz = fx_sar(fx_mul(ry, z), sh);
      xz = fx_sar(fx_mul(rx, z), sh);
    }
  }
};

// Momentum and relaxed moments of the deviations v: n_k = (m_k - m^eq_k) / fx_neq_scale, the
// equilibrium folded into the moment sums in closed form (meq() in sweep.cuh).  Rows
// whose rate can exceed 1/4 are doubled in the sum.
template <int D>
struct FxMomentum {
  i64 x, y, z;
};
LBM_HD FxMomentum<2> fx_neq(D2Q9, const i64 (&v)[9], i64 (&n)[9], int E, const FixedArgs &fx) {
  const i64 s0 = v[1] + v[3], s1 = v[2] + v[4], s2 = v[5] + v[7], s3 = v[6] + v[8];
  const i64 d0 = v[1] - v[3], d1 = v[2] - v[4], d2 = v[5] - v[7], d3 = v[6] - v[8];
  const i64 F = s0 + s1, K = s2 + s3;
  const i64 jx = d0 + d2 - d3, jy = d1 + d2 + d3;
  const FxQuad<2> q(jx, jy, 0, E, fx);
  const i64 j2 = q.xx + q.yy;
  n[1] = 2 * K + ((F - 2 * v[0] - 3 * j2) >> 1);
  n[2] = v[0] - F + j2;
  n[4] = 2 * jx - 3 * d0;
  n[6] = 2 * jy - 3 * d1;
  n[7] = (s0 - s1 - q.xx + q.yy) << 1;
  n[8] = (s2 - s3 - q.xy) << 1;
  return {jx, jy, 0};
}
LBM_HD FxMomentum<3> fx_neq(D3Q15, const i64 (&v)[15], i64 (&n)[15], int E, const FixedArgs &fx) {
  const i64 s0 = v[1] + v[2], s1 = v[3] + v[4], s2 = v[5] + v[6];
  const i64 d0 = v[1] - v[2], d1 = v[3] - v[4], d2 = v[5] - v[6];
  const i64 s3 = v[7] + v[14], s4 = v[8] + v[13], s5 = v[9] + v[12], s6 = v[10] + v[11];
  const i64 d3 = v[7] - v[14], d4 = v[8] - v[13], d5 = v[9] - v[12], d6 = v[10] - v[11];
  const i64 ca = s3 + s6, cb = s4 + s5, cc = s3 - s6, cd = s4 - s5;
  const i64 ce = d3 + d6, cf = d4 + d5, cg = d3 - d6, ch = d4 - d5;
  const i64 F = s0 + s1 + s2, K = ca + cb;
  const i64 jx = d0 + cg - ch, jy = d1 + cg + ch, jz = d2 + ce + cf;
  const FxQuad<3> q(jx, jy, jz, E, fx);
  const i64 j2 = q.xx + q.yy + q.zz;
  n[1] = 2 * K - v[0] - j2;
  n[2] = 3 * v[0] - F + j2;
  n[4] = 2 * jx - 3 * d0;
  n[6] = 2 * jy - 3 * d1;
  n[8] = 2 * jz - 3 * d2;
  n[9] = 2 * (s0 - q.xx) - s1 - s2 + q.yy + q.zz;
  n[10] = (s1 - s2 - q.yy + q.zz) << 1;
  n[11] = ca - cb - q.xy;
  n[12] = cc + cd - q.yz;
  n[13] = cc - cd - q.xz;
  n[14] = ce - cf;
  return {jx, jy, jz};
}
LBM_HD FxMomentum<3> fx_neq(D3Q19, const i64 (&v)[19], i64 (&n)[19], int E, const FixedArgs &fx) {
  i64 s[9], d[9];
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int p = 0; p < 9; ++p) {
    s[p] = v[2 * p + 1] + v[2 * p + 2];
    d[p] = v[2 * p + 1] - v[2 * p + 2];
  }
  const i64 F = s[0] + s[1] + s[2];
  const i64 Exy = s[3] + s[4], Exz = s[5] + s[6], Eyz = s[7] + s[8], Ey = Exy - Exz;
  const i64 K = Exy + Exz + Eyz, Exyz = Exy + Exz - 2 * Eyz;
  const i64 jx = d[0] + d[3] + d[4] + d[5] + d[6];
  const i64 jy = d[1] + d[3] - d[4] + d[7] + d[8];
  const i64 jz = d[2] + d[5] - d[6] + d[7] - d[8];
  const FxQuad<3> q(jx, jy, jz, E, fx);
  const i64 j2 = q.xx + q.yy + q.zz, pw = q.yy - q.zz, px = 2 * q.xx - q.yy - q.zz;
  n[1] = K - v[0] - j2;
  n[2] = 9 * (v[0] >> 2) - 7 * (F >> 2) - 2 * (K >> 2) + 11 * (j2 >> 3);   // up to 178 g: a quarter of it
  n[4] = jx - 3 * d[0];
  n[6] = jy - 3 * d[1];
  n[8] = jz - 3 * d[2];
  n[9] = 2 * s[0] - s[1] - s[2] + Exyz - px;
  n[10] = 2 * (s[1] + s[2] - 2 * s[0]) + Exyz + (px >> 1);
  n[11] = s[1] - s[2] + Ey - pw;
  n[12] = 2 * (s[2] - s[1]) + Ey + (pw >> 1);
  n[13] = (s[3] - s[4] - q.xy) << 1;
  n[14] = (s[7] - s[8] - q.yz) << 1;
  n[15] = (s[5] - s[6] - q.xz) << 1;
  n[16] = d[3] + d[4] - d[5] - d[6];
  n[17] = d[4] - d[3] + d[7] + d[8];
  n[18] = d[5] - d[6] - d[7] + d[8];
  return {jx, jy, jz};
}
// (m_k - m^eq_k) / n_k, 0 for the conserved rows
template <class L>
LBM_HD constexpr double fx_neq_scale(int k) {
  if (L::conserved(k)) return 0.0;
  if (L::Q == 9) return k == 1 ? 2.0 : (k == 2 ? 3.0 : (k >= 7 ? 0.5 : 1.0));
  if (L::Q == 15) return k == 2 ? 5.0 : (k == 4 || k == 6 || k == 8 ? 5.0 / 3 : (k == 10 ? 0.5 : 1.0));
  return k == 1 ? 19.0 : (k == 2 ? 4.0 : (k == 4 || k == 6 || k == 8 ? 5.0 / 3 : (k >= 13 && k <= 15 ? 0.5 : 1.0)));
}

// Rows e and eps of D3Q19 act through one value per face, edge and the rest node, with
// factors up to 30 on their rates: they are taken 8 and 4 times larger and rounded where
// they are used.
template <class L>
LBM_HD constexpr int fx_fine(int k) { return L::Q == 19 ? (k == 1 ? 3 : (k == 2 ? 2 : 0)) : 0; }

// Change of the populations by the relaxed rows, t = M^T r with r_k = s_k (m_k - m^eq_k)
// / |M_k|^2, and by the force (r = -F on the momentum rows), from the deviations v.
template <class L>
LBM_HD void fx_change(L, const i64 (&v)[L::Q], i64 (&t)[L::Q], i64 Fx, i64 Fy, i64 Fz, int E,
                      const FixedArgs &fx) {
  i64 n[L::Q], r[L::Q];
  fx_neq(L{}, v, n, E, fx);
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int k = 0; k < L::Q; ++k) r[k] = L::conserved(k) ? 0 : fx_mul(n[k], fx.row[k]);
  r[3] = -Fx;
  r[5] = -Fy;
  if (L::D == 3) r[7] = -Fz;
  fmt<false, i64>(L{}, r, t);
}
LBM_HD void fx_change(D3Q19, const i64 (&v)[19], i64 (&t)[19], i64 Fx, i64 Fy, i64 Fz, int E,
                      const FixedArgs &fx) {
  i64 n[19], r[19];
  fx_neq(D3Q19{}, v, n, E, fx);
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int k = 0; k < 19; ++k) r[k] = D3Q19::conserved(k) ? 0 : fx_mul(n[k], fx.row[k]);
  // the back-transform (fmt() in moments.cuh); the rest node gets what keeps the sum over all
  // nodes zero
  const i64 Ce = r[1] + ((r[2] + 2) >> 2), Cf = -((11 * r[1] + 4) >> 3) - r[2];
  const i64 A = r[9] + r[10], B = r[11] + r[12];
  const i64 Y = Cf - r[9] + 2 * r[10], Z = r[11] - 2 * r[12];
  const i64 Pxy = Ce + A + B, Pxz = Ce + A - B, Pyz = Ce - 2 * A;
  i64 ev[9], od[9];
  ev[0] = Cf + 2 * r[9] - 4 * r[10];
  ev[1] = Y + Z;
  ev[2] = Y - Z;
  ev[3] = Pxy + r[13];
  ev[4] = Pxy - r[13];
  ev[5] = Pxz + r[15];
  ev[6] = Pxz - r[15];
  ev[7] = Pyz + r[14];
  ev[8] = Pyz - r[14];
  od[0] = -Fx - 4 * r[4];
  od[1] = -Fy - 4 * r[6];
  od[2] = -Fz - 4 * r[8];
  const i64 xf = r[4] - Fx, yf = r[6] - Fy, zf = r[8] - Fz;
  const i64 xa = xf + r[16], ya = yf - r[17];
  od[3] = xa + ya;
  od[4] = xa - ya;
  const i64 xb = xf - r[16], zb = zf + r[18];
  od[5] = xb + zb;
  od[6] = xb - zb;
  const i64 yc = yf + r[17], zc = zf - r[18];
  od[7] = yc + zc;
  od[8] = yc - zc;
  t[0] = -6 * Cf - 12 * Ce;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int p = 0; p < 9; ++p) {
    t[2 * p + 1] = ev[p] + od[p];
    t[2 * p + 2] = ev[p] - od[p];
  }
}

inline FixedCoef fx_coef(double c) {   // c in [0, 1/4]
  const i64 b = (i64)llrint(ldexp(c, 64));
  const int lo = (int)(unsigned)b;
  return {(int)((b - lo) >> 32), lo};
}
template <class L>
inline FixedArgs fx_args(const double *s, double rho0, const double *F) {
  FixedArgs fx{};
  for (int k = 0; k < L::Q; ++k)
    if (!L::conserved(k)) fx.row[k] = fx_coef(ldexp(fx_neq_scale<L>(k), fx_fine<L>(k)) * s[k] / row_norm2<L>(k));
  int er = 0;
  double mr = frexp(1.0 / rho0, &er);    // [1/2, 1)
  if (mr == 0.5) {
    mr = 1.0;
    --er;
  }
  fx.inv_rho0 = fx_coef(mr / 4);
  fx.quad_shift = kFxTop<L> + 963 - er;
  fx.max_exp = 1023 + (ilogb(rho0) - 5 < 14 ? ilogb(rho0) - 5 : 14);
  // no relaxed row: the populations move on unchanged, which the FP64 form does bit for bit
  bool relaxes = false;
  for (int k = 0; k < L::Q; ++k) relaxes |= !L::conserved(k) && s[k] != 0.0;
  if (fx.max_exp < kFxMinExp || !relaxes) fx.max_exp = -1;
  fx.force_hi = 0;
  for (int a = 0; a < 3; ++a)
    if ((fx_hi(F[a]) & 0x7fffffff) > fx.force_hi) fx.force_hi = fx_hi(F[a]) & 0x7fffffff;
  return fx;
}

// block exponent of a node's deviations: true if the fixed-point form covers them
template <class L>
LBM_HD bool fx_block(const double (&g)[L::Q], const FixedArgs &fx, int &E) {
  int mx = fx.force_hi;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int i = 0; i < L::Q; ++i) {
    const int h = fx_hi(g[i]) & 0x7fffffff;
    mx = h > mx ? h : mx;
  }
  E = mx >> 20;
  const bool ok = (E >= kFxMinExp && E <= fx.max_exp) || mx == 0;
  if (mx == 0) E = kFxMinExp;   // a node at rest without force stays exactly at rest
  return ok;
}

}  // namespace lbm
