// fixed.cuh -- the MRT collision of FP64 storage in 64-bit block fixed point.
//
// Why: the FP64 pipe of this GPU issues one warp instruction in 64 cycles per quarter of
// an SM (about 1.25 TFLOP/s in all), the integer pipe one in one or two.  A collision is
// some 200 additions, small integer multiples and two dozen products; in FP64 that work,
// not memory, bounds the sweep.  Here the Q deviations of a node are aligned to
// the exponent of the largest of them and held as 64-bit integers, so that an addition is
// two integer instructions and exact.
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
// gives what it gave.  With g the largest deviation, |j_a| <= 10 g and j_a j_b / rho0 <= 6.3 g (D2Q9:
// 6 g and 2.3 g), every sum given to fx_mul is below 45 g (D2Q9: 25 g) and every result
// below 55 g (D2Q9: 16 g): all within 64 bits.
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

// logical right shift whose amount may exceed 63 (result 0)
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
  const int hi = __double2hiint(x);
  return __hiloint2double(v != 0 ? hi + ((E - 1023 - kTop) << 20) : 0, __double2loint(x));
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

// Change of the populations by the relaxed rows, t = M^T r with r_k = s_k (m_k - m^eq_k)
// / |M_k|^2, and by the force (r = -F on the momentum rows), from the deviations v.  The
// equilibrium is folded into the moment sums in closed form (meq() in sweep.cuh); the
// constant of a row carries the factor taken out of its sum (fx_row_scale).  Rows
// whose rate can exceed 1/4 are doubled in the sum.
LBM_HD void fx_change(D2Q9, const i64 (&v)[9], i64 (&t)[9], i64 Fx, i64 Fy, i64 Fz, int E,
                      const FixedArgs &fx) {
  i64 r[9];
  const i64 s0 = v[1] + v[3], s1 = v[2] + v[4], s2 = v[5] + v[7], s3 = v[6] + v[8];
  const i64 d0 = v[1] - v[3], d1 = v[2] - v[4], d2 = v[5] - v[7], d3 = v[6] - v[8];
  const i64 F = s0 + s1, K = s2 + s3;
  const i64 jx = d0 + d2 - d3, jy = d1 + d2 + d3;
  const FxQuad<2> q(jx, jy, 0, E, fx);
  const i64 j2 = q.xx + q.yy;
  r[1] = fx_mul(2 * K + ((F - 2 * v[0] - 3 * j2) >> 1), fx.row[1]);
  r[2] = fx_mul(v[0] - F + j2, fx.row[2]);
  r[4] = fx_mul(2 * jx - 3 * d0, fx.row[4]);
  r[6] = fx_mul(2 * jy - 3 * d1, fx.row[6]);
  r[7] = fx_mul((s0 - s1 - q.xx + q.yy) << 1, fx.row[7]);
  r[8] = fx_mul((s2 - s3 - q.xy) << 1, fx.row[8]);
  r[0] = 0;
  r[3] = -Fx;
  r[5] = -Fy;
  fmt<false, i64>(D2Q9{}, r, t);
}
LBM_HD void fx_change(D3Q15, const i64 (&v)[15], i64 (&t)[15], i64 Fx, i64 Fy, i64 Fz, int E,
                      const FixedArgs &fx) {
  i64 r[15];
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
  r[1] = fx_mul(2 * K - v[0] - j2, fx.row[1]);
  r[2] = fx_mul(3 * v[0] - F + j2, fx.row[2]);
  r[4] = fx_mul(2 * jx - 3 * d0, fx.row[4]);
  r[6] = fx_mul(2 * jy - 3 * d1, fx.row[6]);
  r[8] = fx_mul(2 * jz - 3 * d2, fx.row[8]);
  r[9] = fx_mul(2 * (s0 - q.xx) - s1 - s2 + q.yy + q.zz, fx.row[9]);
  r[10] = fx_mul((s1 - s2 - q.yy + q.zz) << 1, fx.row[10]);
  r[11] = fx_mul(ca - cb - q.xy, fx.row[11]);
  r[12] = fx_mul(cc + cd - q.yz, fx.row[12]);
  r[13] = fx_mul(cc - cd - q.xz, fx.row[13]);
  r[14] = fx_mul(ce - cf, fx.row[14]);
  r[0] = 0;
  r[3] = -Fx;
  r[5] = -Fy;
  r[7] = -Fz;
  fmt<false, i64>(D3Q15{}, r, t);
}
LBM_HD void fx_change(D3Q19, const i64 (&v)[19], i64 (&t)[19], i64 Fx, i64 Fy, i64 Fz, int E,
                      const FixedArgs &fx) {
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
  // Rows e and eps act through one value per face, edge and the rest node, with factors
  // up to 30 on their rates: they are taken 8 and 4 times larger, rounded where they are
  // used, and the rest node gets what keeps the sum over all nodes zero.  (The
  // sum of row eps, up to 178 g, is taken in units 4 times larger.)
  const i64 r1 = fx_mul(K - v[0] - j2, fx.row[1]);
  const i64 r2 = fx_mul(9 * (v[0] >> 2) - 7 * (F >> 2) - 2 * (K >> 2) + 11 * (j2 >> 3), fx.row[2]);
  const i64 Ce = r1 + ((r2 + 2) >> 2), Cf = -((11 * r1 + 4) >> 3) - r2;
  const i64 rx = fx_mul(jx - 3 * d[0], fx.row[4]), ry = fx_mul(jy - 3 * d[1], fx.row[6]);
  const i64 rz = fx_mul(jz - 3 * d[2], fx.row[8]);
  const i64 r9 = fx_mul(2 * s[0] - s[1] - s[2] + Exyz - px, fx.row[9]);
  const i64 r10 = fx_mul(2 * (s[1] + s[2] - 2 * s[0]) + Exyz + (px >> 1), fx.row[10]);
  const i64 r11 = fx_mul(s[1] - s[2] + Ey - pw, fx.row[11]);
  const i64 r12 = fx_mul(2 * (s[2] - s[1]) + Ey + (pw >> 1), fx.row[12]);
  const i64 r13 = fx_mul((s[3] - s[4] - q.xy) << 1, fx.row[13]);
  const i64 r14 = fx_mul((s[7] - s[8] - q.yz) << 1, fx.row[14]);
  const i64 r15 = fx_mul((s[5] - s[6] - q.xz) << 1, fx.row[15]);
  const i64 r16 = fx_mul(d[3] + d[4] - d[5] - d[6], fx.row[16]);
  const i64 r17 = fx_mul(d[4] - d[3] + d[7] + d[8], fx.row[17]);
  const i64 r18 = fx_mul(d[5] - d[6] - d[7] + d[8], fx.row[18]);
  // back-transform (fmt() in moments.cuh)
  const i64 A = r9 + r10, B = r11 + r12;
  const i64 Y = Cf - r9 + 2 * r10, Z = r11 - 2 * r12;
  const i64 Pxy = Ce + A + B, Pxz = Ce + A - B, Pyz = Ce - 2 * A;
  i64 ev[9], od[9];
  ev[0] = Cf + 2 * r9 - 4 * r10;
  ev[1] = Y + Z;
  ev[2] = Y - Z;
  ev[3] = Pxy + r13;
  ev[4] = Pxy - r13;
  ev[5] = Pxz + r15;
  ev[6] = Pxz - r15;
  ev[7] = Pyz + r14;
  ev[8] = Pyz - r14;
  od[0] = -Fx - 4 * rx;
  od[1] = -Fy - 4 * ry;
  od[2] = -Fz - 4 * rz;
  const i64 xf = rx - Fx, yf = ry - Fy, zf = rz - Fz;
  const i64 xa = xf + r16, ya = yf - r17;
  od[3] = xa + ya;
  od[4] = xa - ya;
  const i64 xb = xf - r16, zb = zf + r18;
  od[5] = xb + zb;
  od[6] = xb - zb;
  const i64 yc = yf + r17, zc = zf - r18;
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

// factor of row k's constant relative to s_k / |M_k|^2 in fx_change (0: not used)
inline double fx_row_scale(int lattice, int k) {
  if (lattice == D2Q9::kLattice) {
    const double t[9] = {0, 2, 3, 0, 1, 0, 1, 0.5, 0.5};
    return t[k];
  }
  if (lattice == D3Q15::kLattice) {
    const double t[15] = {0, 1, 5, 0, 5.0 / 3, 0, 5.0 / 3, 0, 5.0 / 3, 1, 0.5, 1, 1, 1, 1};
    return t[k];
  }
  const double t[19] = {0, 8 * 19, 16, 0, 5.0 / 3, 0, 5.0 / 3, 0, 5.0 / 3, 1, 1, 1, 1, 0.5, 0.5, 0.5, 1, 1, 1};
  return t[k];
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
    if (!L::conserved(k)) fx.row[k] = fx_coef(fx_row_scale(L::kLattice, k) * s[k] / row_norm2<L>(k));
  int er = 0;
  double mr = frexp(1.0 / rho0, &er);    // [1/2, 1)
  if (mr == 0.5) {
    mr = 1.0;
    --er;
  }
  fx.inv_rho0 = fx_coef(mr / 4);
  fx.quad_shift = kFxTop<L> + 963 - er;
  fx.max_exp = 1023 + (ilogb(rho0) - 5 < 14 ? ilogb(rho0) - 5 : 14);
  if (fx.max_exp < kFxMinExp) fx.max_exp = -1;
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
