// fixed_adjoint.cuh -- the transpose of the FP64 collision in block fixed point, for the
// adjoint step (adjoint.cu); callable on the host too, as fixed.cuh is.
#pragma once

#include "fixed.cuh"
#include "sweep.cuh"

namespace lbm {

// ---------------------------------------------------------------------------
// The collision transpose of FP64 storage in block fixed point (fixed.cuh): the state's
// moments and the adjoint's are sums of integers, and every factor (s_k, 1/|M_k|^2,
// the velocity) is a fixed-point product.  In FP64 this is some 400 instructions a node
// at one warp instruction in 64 cycles per quarter SM; here the Q results, the dJ/ds
// products and the boundary terms are FP64.  Forward and backward pass over 40 steps:
// D3Q19 96^3 33.1 -> 16.0 ms, 56^3 7.2 -> 3.5; D2Q9 96^2 x 100 2.45 -> 2.05.
//
// The adjoint populations are multiples of 2^(E_l - 53), E_l their largest exponent; sums
// with M (up to 192 times the largest) fit 62 bits.  Scaled moments and results are
// multiples of 2^(E_l - 57), the largest adjoint value is below 2^58 of them, and 64 bits
// hold 32 times that.  For every s in [0, 2] and |u_a| < 0.63 (deviations under rho0/16,
// fx_block's range) results stay below 13 times the largest adjoint value and the factors of the
// velocity in fx_meq_adjoint below 8 times (row sums of the transposed operator).  Rows e
// and eps of D3Q19 arrive 8 and 4 times larger: the sums with them stay below 24.4 times
// before their shifts (a in fx_meq_adjoint: 19 x 8 x 2 x 192 / 2394 at s_e = 2, s_eps = 0;
// 38 and 22 for its factors, with a shift by 3, would reach 48.8).  tests/test_fixed_point_host.py
// runs the extremes with overflow checks.  Nodes outside these ranges take the FP64 form.
// ---------------------------------------------------------------------------
constexpr int kAdjIn = 53, kAdjOut = 57;
template <class L>
constexpr int row_abs_sum(int k) {
  int s = 0;
  for (int i = 0; i < L::Q; ++i) s += L::M(k, i) < 0 ? -L::M(k, i) : L::M(k, i);
  return s;
}
// left shift of moment k before its products: its sum stays below 2^62
template <class L>
constexpr int adj_shift(int k) {
  int sh = 0;
  while (row_abs_sum<L>(k) << (sh + 1) <= 256) ++sh;
  return sh;
}
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
    const int e = kAdjOut - kAdjIn - adj_shift<L>(k) + fx_fine<L>(k);
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

// Collision transpose of one node: t = M^T nu from g and lambda' (lp), and gsum_k =
// mu_k / |M_k|^2 (m^eq_k - m_k) over -fx_neq_scale 2^-fx_fine (products in FP64: m_k - m^eq_k is
// often small, and a product in the moments' units would lose its digits); false if
// the node is outside the integer ranges.
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
  for (int i = 0; i < L::Q; ++i) v[i] = fx_from<kAdjIn>(lp[i], El);
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
        gsum[k] = fx_to<kAdjOut>(nu[k], El) * fx_to<kFxTop<L>>(n[k], Eg);
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
