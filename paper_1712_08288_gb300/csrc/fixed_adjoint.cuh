// fixed_adjoint.cuh -- the transpose of the collision for the adjoint step (adjoint.cu), in
// the compute type and, for FP64 storage, in block fixed point; callable on the host too,
// as fixed.cuh is.
#pragma once

#include "fixed.cuh"
#include "sweep.cuh"

namespace lbm {

LBM_HD unsigned fx_bits(float x) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(x);
#else
  unsigned b;
  memcpy(&b, &x, 4);
  return b;
#endif
}
LBM_HD double fx_double(unsigned hi, unsigned lo) {
#ifdef __CUDA_ARCH__
  return __hiloint2double((int)hi, (int)lo);
#else
  const u64 b = ((u64)hi << 32) | lo;
  double x;
  memcpy(&x, &b, 8);
  return x;
#endif
}

// v in FP64 by its bits, without the conversion instruction (64 issue cycles): the exponent
// moves by 896, subnormal numbers are scaled by 2^64 first, infinities and NaN keep the
// largest exponent.  Straight-line: a branch to the conversion for the rare values spills the
// adjoint step's registers (D3Q19 FP32, 64^3 x 144 steps: 4.35 ms, 4.17 so, 4.23 converted).
LBM_HD double fx_widen(float v) {
  const bool tiny = fabsf(v) < 1.1754944e-38f;
  const unsigned b = fx_bits(tiny ? v * 1.8446744073709552e19f : v);
  const unsigned bias = (b & 0x7f800000u) == 0x7f800000u ? 0x70000000u : (tiny ? 0x34000000u : 0x38000000u);
  const unsigned hi = (b & 0x7fffffffu) != 0u ? ((b >> 3) & 0x0fffffffu) + bias : 0u;
  return fx_double(hi | (b & 0x80000000u), b << 29);
}

// sum_k smu_k * d meq_k / d(rho, j_x, j_y, j_z) for the equilibrium moments of
// meq() (deviation form), smu_k = s_k mu_k on the non-conserved rows
template <class C>
LBM_HD void meq_adjoint(D2Q9, const C (&smu)[9], C jx, C jy, C, C ir0,
                        C (&out)[4]) {
  out[0] = C(-2) * smu[1] + smu[2];
  const C a = C(6) * (smu[1] - smu[2]) * ir0;
  out[1] = a * jx - smu[4] + (C(2) * smu[7] * jx + smu[8] * jy) * ir0;
  out[2] = a * jy - smu[6] + (C(-2) * smu[7] * jy + smu[8] * jx) * ir0;
  out[3] = C(0);
}
template <class C>
LBM_HD void meq_adjoint(D3Q19, const C (&smu)[19], C jx, C jy, C jz, C ir0,
                        C (&out)[4]) {
  out[0] = C(-11) * smu[1] + C(3) * smu[2];
  const C a = (C(38) * smu[1] - C(11) * smu[2]) * ir0;    // e, eps: 19 j^2, -5.5 j^2
  const C px = (C(4) * smu[9] - C(2) * smu[10]) * ir0;    // 3p_xx, 3pi_xx along j_x
  const C pyz = (C(-2) * smu[9] + smu[10]) * ir0;         // 3p_xx, 3pi_xx along j_y, j_z
  const C w = (C(2) * smu[11] - smu[12]) * ir0;           // p_ww, pi_ww along j_y (-w along j_z)
  const C c23 = C(2.0 / 3.0);
  out[1] = (a + px) * jx - c23 * smu[4] + (smu[13] * jy + smu[15] * jz) * ir0;
  out[2] = (a + pyz + w) * jy - c23 * smu[6] + (smu[13] * jx + smu[14] * jz) * ir0;
  out[3] = (a + pyz - w) * jz - c23 * smu[8] + (smu[14] * jy + smu[15] * jx) * ir0;
}

template <class C>
LBM_HD void meq_adjoint(D3Q15, const C (&smu)[15], C jx, C jy, C jz, C ir0,
                        C (&out)[4]) {
  out[0] = -smu[1] + smu[2];
  const C a = (C(2) * smu[1] - C(10) * smu[2]) * ir0;    // e, eps: j^2, -5 j^2
  const C px = C(4) * smu[9] * ir0;                      // 3p_xx along j_x
  const C pyz = C(-2) * smu[9] * ir0;                    // 3p_xx along j_y, j_z
  const C w = C(2) * smu[10] * ir0;                      // p_ww along j_y (-w along j_z)
  const C c73 = C(7.0 / 3.0);
  out[1] = (a + px) * jx - c73 * smu[4] + (smu[11] * jy + smu[13] * jz) * ir0;
  out[2] = (a + pyz + w) * jy - c73 * smu[6] + (smu[11] * jx + smu[12] * jz) * ir0;
  out[3] = (a + pyz - w) * jz - c73 * smu[8] + (smu[12] * jy + smu[13] * jx) * ir0;
}

// Collision transpose of one node in the compute type: t = M^T nu, gsum_k = dJ/ds_k, through
// the factored transforms (fmoments, fmt), which take fewer operations than the pair form
// (FP32: 0.349 -> 0.340 s for the backward pass at 128^3 x 2000).
template <class L, class C>
LBM_HD void adjoint_plain(const C (&g)[L::Q], const C (&lp)[L::Q], const SweepArgs<C> &sa, C (&t)[L::Q],
                          C (&gsum)[L::Q]) {
  constexpr int Q = L::Q;
  const C ir0 = sa.inv_rho0;
  C m[Q], mu[Q];
  fmoments<C>(L{}, g, m);
  fmoments<C>(L{}, lp, mu);
  const C jx = m[3], jy = m[5], jz = L::D == 3 ? m[7] : C(0);
  C smu[Q], nu[Q];
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int k = 0; k < Q; ++k) {
    if (Rows<L>::cons(k)) {
      smu[k] = C(0);
      mu[k] *= C(1.0 / row_norm2<L>(k));
      continue;
    }
    smu[k] = sa.sn[k] * mu[k];                                      // s_k (M lambda')_k / |M_k|^2
    mu[k] *= C(1.0 / row_norm2<L>(k));
    gsum[k] = mu[k] * (meq(L{}, k, m[0], jx, jy, jz, ir0) - m[k]);   // d m'_k/d s_k
    nu[k] = mu[k] - smu[k];                                         // (1 - s_k) mu_k
  }
  C dq[4];
  meq_adjoint(L{}, smu, jx, jy, jz, ir0, dq);
  nu[0] = mu[0] + dq[0];
  nu[3] = mu[3] + dq[1];
  nu[5] = mu[5] + dq[2];
  if (L::D == 3) nu[7] = mu[7] + dq[3];
  fmt<true, C>(L{}, nu, t);
}

// ---------------------------------------------------------------------------
// The collision transpose of FP64 storage in block fixed point (fixed.cuh): the state's
// moments and the adjoint's are sums of integers, and every factor (s_k, 1/|M_k|^2,
// the velocity) is a fixed-point product.  In FP64 this is some 400 instructions a node
// at one warp instruction in 64 cycles per quarter SM; here the Q results, the dJ/ds
// products and the boundary terms are FP64.  Forward and backward pass over 40 steps:
// D3Q19 96^3 33.1 -> 16.0 ms, 56^3 7.2 -> 3.5; D2Q9 96^2 x 100 2.45 -> 2.05.
//
// The adjoint populations are multiples of 2^(E_l - kAdjIn), E_l their largest exponent, as
// fine as the largest row sum of M allows (16, 48 and 192 times the largest: 2^62, 2^61.6 and
// 2^62.6, fx_mul's limit is 2^62.9).  dJ/ds takes the exact sums M lambda': on a smooth
// adjoint field it consists of the small moments, and with entries in multiples of
// 2^(E_l - 53) and moments of 2^(E_l - 57) its error was up to twice that of the FP64 form
// (rms of a node's largest: D2Q9 4.6e-14, now 2.2e-15, FP64 4.8e-14; D3Q15 6.8e-14, 1.0e-14,
// 3.6e-14; D3Q19 4.0e-14, 1.6e-14, 3.3e-14; tests/test_fixed_point_host.py).  Scaled moments and results are
// multiples of 2^(E_l - 57), the largest adjoint value is below 2^58 of them, and 64 bits
// hold 32 times that.  For every s in [0, 2] and |u_a| < 0.63 (deviations under rho0/16,
// fx_block's range) results stay below 13 times the largest adjoint value and the factors of the
// velocity in fx_meq_adjoint below 8 times (row sums of the transposed operator).  Rows e
// and eps of D3Q19 arrive 8 and 4 times larger: the sums with them stay below 24.4 times
// before their shifts (a in fx_meq_adjoint: 19 x 8 x 2 x 192 / 2394 at s_e = 2, s_eps = 0;
// 38 and 22 for its factors, with a shift by 3, would reach 48.8).  tests/test_fixed_point_host.py
// runs the extremes with overflow checks.  Nodes outside these ranges take the FP64 form.
// ---------------------------------------------------------------------------
template <class L>
constexpr int kAdjIn = L::Q == 9 ? 57 : (L::Q == 15 ? 55 : 54);
constexpr int kAdjOut = 57;
template <class L>
constexpr int row_abs_sum(int k) {
  int s = 0;
  for (int i = 0; i < L::Q; ++i) s += L::M(k, i) < 0 ? -L::M(k, i) : L::M(k, i);
  return s;
}
// left shift of moment k before its products: its sum stays below 2^62 (2^62.6 for row e of D3Q19)
template <class L>
constexpr int adj_shift(int k) {
  int sh = 0;
  while ((i64)row_abs_sum<L>(k) << (sh + 1) <= (i64)1 << (61 - kAdjIn<L>)) ++sh;
  return sh;
}
// what fx_mul takes: 2^62.9 = 1.866 x 2^62, with entries below 2^(kAdjIn + 1)
template <class L>
constexpr bool adj_sums_fit() {
  for (int k = 0; k < L::Q; ++k)
    if (100 * ((i64)row_abs_sum<L>(k) << adj_shift<L>(k)) > (i64)186 << (61 - kAdjIn<L>) || adj_shift<L>(k) > 7)
      return false;
  return true;
}
static_assert(adj_sums_fit<D2Q9>() && adj_sums_fit<D3Q15>() && adj_sums_fit<D3Q19>(), "moments of the adjoint fit fx_mul");
// all rows' shifts, 3 bits each: a literal in device code
template <class L>
constexpr u64 adj_shifts() {
  u64 t = 0;
  for (int k = 0; k < L::Q; ++k) t |= (u64)adj_shift<L>(k) << (3 * k);
  return t;
}
template <class L>
struct AdjShift {
  static constexpr u64 kAll = adj_shifts<L>();
  static __device__ __forceinline__ constexpr int of(int k) { return (int)(kAll >> (3 * k)) & 7; }
};

// constants of the products: 1 / |M_k|^2 and s_k / |M_k|^2 in the units above
template <class L>
inline FixedAdj fx_adj_args(const double *sn) {
  FixedAdj f{};
  for (int k = 0; k < L::Q; ++k) {
    const int e = kAdjOut - kAdjIn<L> - adj_shift<L>(k) + fx_fine<L>(k);
    f.inv_n[k] = fx_coef(ldexp(1.0 / row_norm2<L>(k), e));
    f.s_n[k] = L::conserved(k) ? FixedCoef{0, 0} : fx_coef(ldexp(sn[k], e));
  }
  return f;
}

// sum_k smu_k d meq_k / d(rho, j_a) as in meq_adjoint, with u_a 2^63 for j_a / rho0 and smu in its units
// (D3Q19: rows 1, 2 times 8 and 4)
LBM_HD i64 adj_times(i64 v, FxHalves u) { return fx_mul(fx_halves(v << 1), u); }
LBM_HD FixedCoef const_sixth() { return {0x2aaaaaab, (int)0xaaaaaaab}; }       // 1/6
LBM_HD FixedCoef const_7_48() { return {0x25555555, 0x55555555}; }              // 7/48
LBM_HD void fx_meq_adjoint(D2Q9, const i64 (&smu)[9], FxHalves ux, FxHalves uy, FxHalves,
                           i64 (&out)[4]) {
  out[0] = smu[2] - 2 * smu[1];
  const i64 a = 6 * (smu[1] - smu[2]);
  out[1] = adj_times(a + 2 * smu[7], ux) + adj_times(smu[8], uy) - smu[4];
  out[2] = adj_times(a - 2 * smu[7], uy) + adj_times(smu[8], ux) - smu[6];
  out[3] = 0;
}
LBM_HD void fx_meq_adjoint(D3Q15, const i64 (&smu)[15], FxHalves ux, FxHalves uy, FxHalves uz,
                           i64 (&out)[4]) {
  out[0] = smu[2] - smu[1];
  const i64 a = 2 * smu[1] - 10 * smu[2], yz = a - 2 * smu[9];
  out[1] = adj_times(a + 4 * smu[9], ux) + adj_times(smu[11], uy) + adj_times(smu[13], uz);
  out[2] = adj_times(yz + 2 * smu[10], uy) + adj_times(smu[11], ux) + adj_times(smu[12], uz);
  out[3] = adj_times(yz - 2 * smu[10], uz) + adj_times(smu[12], uy) + adj_times(smu[13], ux);
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int c = 0; c < 3; ++c) out[1 + c] -= fx_mul(smu[4 + 2 * c] << 4, const_7_48());   // 7/3 smu
}
LBM_HD void fx_meq_adjoint(D3Q19, const i64 (&smu)[19], FxHalves ux, FxHalves uy, FxHalves uz,
                           i64 (&out)[4]) {
  out[0] = (6 * smu[2] - 11 * smu[1] + 4) >> 3;              // -11/8, 3/4
  const i64 a = (19 * smu[1] - 11 * smu[2] + 2) >> 2;        // 38/8, -11/4
  const i64 yz = a - 2 * smu[9] + smu[10], w = 2 * smu[11] - smu[12];
  out[1] = adj_times(a + 4 * smu[9] - 2 * smu[10], ux) + adj_times(smu[13], uy) + adj_times(smu[15], uz);
  out[2] = adj_times(yz + w, uy) + adj_times(smu[13], ux) + adj_times(smu[14], uz);
  out[3] = adj_times(yz - w, uz) + adj_times(smu[14], uy) + adj_times(smu[15], ux);
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int c = 0; c < 3; ++c) out[1 + c] -= fx_mul(smu[4 + 2 * c] << 2, const_sixth());   // 2/3 smu
}

// M^T nu with rho; rows 1 and 2 of D3Q19 arrive 8 and 4 times larger
template <class L>
LBM_HD void fx_adj_back(L, const i64 (&nu)[L::Q], i64 (&t)[L::Q]) {
  fmt<true, i64>(L{}, nu, t);
}
LBM_HD void fx_adj_back(D3Q19, const i64 (&nu)[19], i64 (&t)[19]) {
  i64 m[19];
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int k = 0; k < 19; ++k) m[k] = nu[k];
  m[1] = m[2] = 0;
  m[0] = 0;
  fmt<true, i64>(D3Q19{}, m, t);
  t[0] += nu[0] - ((30 * nu[1] + 4) >> 3) + 3 * nu[2];
  const i64 face = nu[0] - ((11 * nu[1] + 4) >> 3) - nu[2], edge = nu[0] + nu[1] + ((nu[2] + 2) >> 2);
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int i = 1; i < 19; ++i) t[i] += i < 7 ? face : edge;
}

// dJ/ds_k over the gsum_k of fx_adjoint
template <class L>
LBM_HD constexpr double fx_gsum_scale(int k) { return L::conserved(k) ? 0.0 : -fx_neq_scale<L>(k) / row_norm2<L>(k); }

// Collision transpose of one node: t = M^T nu from g and lambda' (lp), and gsum_k = mu_k |M_k|^2
// (m_k - m^eq_k) / fx_neq_scale, the exact sum M lambda' times the relaxed moment (products in
// FP64: m_k - m^eq_k is often small, and a product in the moments' units would lose its
// digits); false if the node is outside the integer ranges.
template <class L>
LBM_HD bool fx_adjoint(const double (&g)[L::Q], const double (&lp)[L::Q], const FixedArgs &fx,
                       const FixedAdj &fa, double (&t)[L::Q], double (&gsum)[L::Q]) {
  int Eg, mx = 0;
  if (!fx_block<L>(g, fx, Eg)) return false;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int i = 0; i < L::Q; ++i) {
    const int h = fx_hi(lp[i]) & 0x7fffffff;
    mx = h > mx ? h : mx;
  }
  int El = mx >> 20;
  if (mx != 0 && (El < kFxMinExp || El > 1900)) return false;
  if (El < kFxMinExp) El = kFxMinExp;
  i64 v[L::Q], n[L::Q];
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int i = 0; i < L::Q; ++i) v[i] = fx_from<kFxTop<L>>(g[i], Eg);
  const auto j = fx_neq(L{}, v, n, Eg, fx);
  const int q = fx.quad_shift - Eg - 1;
  const FxHalves ux = fx_halves(fx_sar(fx_mul(j.x << 2, fx.inv_rho0) << 2, q));
  const FxHalves uy = fx_halves(fx_sar(fx_mul(j.y << 2, fx.inv_rho0) << 2, q));
  const FxHalves uz = fx_halves(fx_sar(fx_mul(j.z << 2, fx.inv_rho0) << 2, q));
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int i = 0; i < L::Q; ++i) v[i] = fx_from<kAdjIn<L>>(lp[i], El);
  i64 nu[L::Q], smu[L::Q];
  {
    i64 mu[L::Q];
    fmoments<i64>(L{}, v, mu);
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int k = 0; k < L::Q; ++k) {
      const i64 m = mu[k] << AdjShift<L>::of(k);
      nu[k] = fx_mul(m, fa.inv_n[k]);
      smu[k] = 0;
      if (!Rows<L>::cons(k)) {
        smu[k] = fx_mul(m, fa.s_n[k]);
        gsum[k] = fx_to<kAdjIn<L>>(mu[k], El) * fx_to<kFxTop<L>>(n[k], Eg);
        nu[k] -= smu[k];
      }
    }
  }
  i64 dq[4], r[L::Q];
  fx_meq_adjoint(L{}, smu, ux, uy, uz, dq);
  nu[0] += dq[0];
  nu[3] += dq[1];
  nu[5] += dq[2];
  if (L::D == 3) nu[7] += dq[3];
  fx_adj_back(L{}, nu, r);
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int i = 0; i < L::Q; ++i) t[i] = fx_to<kAdjOut>(r[i], El);
  return true;
}

}  // namespace lbm
