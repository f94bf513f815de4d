// sweep.cuh -- the fused collide / stream / boundary sweep (one time step).
//
// One thread owns one node.  Populations live in one array in SoA order
// (population i of node n at i*N + n, x fastest) and are updated in place with
// the AA pattern:
//   even step  node x reads slot i of x, writes f'_i to slot opp(i) of x;
//   odd step   node x reads slot opp(i) of x - e_i, writes f'_i to slot i of x + e_i.
// Each node reads exactly the slots it writes, so a step needs one array and no
// synchronisation between threads.
//
// Cut links (Sec. 2 of arXiv:1712.08288).  For a fluid node x_f whose neighbour
// x_f + e_d is solid, the population i = opp(d) that would arrive from that
// neighbour is produced by the single-node scheme, Eqs. 2.10 and 2.13, from the
// node's own pre-collision f_i, f_d and post-collision f'_i, f'_d, which all sit in
// registers at that point.  The value goes where the next step looks for
// f_i(x_f, t+1): after an odd step into slot i of x_f itself (which only the solid
// node would otherwise write); after an even step into the link's entry of a
// compact link buffer, which the next odd step reads in place of slot d of the
// solid neighbour.  Solid nodes' slots are never written.
//
// Collision (Appendix, MRT): in deviation variables g = f - w rho0,
//   m = M g, m'_k = m_k - s_k (m_k - m^eq_k) for the non-conserved rows,
//   g' = g - M^-1 (m - m') + M^-1 (rho0 g_force at the j rows),
// with M^-1 = M^T diag(1/|M_k|^2) (rows of M are orthogonal).  Rows are either
// even or odd under e -> -e, so the products run over the sums s_p = g_i + g_ib
// and differences a_p = g_i - g_ib of opposite pairs.
#pragma once

#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "fixed.cuh"
#include "moments.cuh"

namespace lbm {

// Equilibrium moments m^eq_k in deviation form (rho replaced by rho - rho0) for
// the incompressible equilibrium of Eq. 42, j = rho0 u.  These are the closed forms
// of M f^eq for the moment bases (Lallemand & Luo 2000 for D2Q9; d'Humieres et
// al. 2002 for D3Q19 with w_eps = 3, w_epsj = -11/2, w_xx = -1/2; the Appendix's
// D3Q15 basis below).
template <class C>
LBM_HD C meq(D2Q9, int k, C drho, C jx, C jy, C, C ir0) {
  switch (k) {
    case 1: return C(-2) * drho + C(3) * (jx * jx + jy * jy) * ir0;
    case 2: return drho - C(3) * (jx * jx + jy * jy) * ir0;
    case 4: return -jx;
    case 6: return -jy;
    case 7: return (jx * jx - jy * jy) * ir0;
    case 8: return jx * jy * ir0;
    default: return C(0);
  }
}
template <class C>
LBM_HD C meq(D3Q19, int k, C drho, C jx, C jy, C jz, C ir0) {
  const C j2 = (jx * jx + jy * jy + jz * jz) * ir0;
  switch (k) {
    case 1: return C(-11) * drho + C(19) * j2;
    case 2: return C(3) * drho - C(5.5) * j2;
    case 4: return C(-2.0 / 3.0) * jx;
    case 6: return C(-2.0 / 3.0) * jy;
    case 8: return C(-2.0 / 3.0) * jz;
    case 9: return C(3) * jx * jx * ir0 - j2;
    case 10: return C(-0.5) * (C(3) * jx * jx * ir0 - j2);
    case 11: return (jy * jy - jz * jz) * ir0;
    case 12: return C(-0.5) * (jy * jy - jz * jz) * ir0;
    case 13: return jx * jy * ir0;
    case 14: return jy * jz * ir0;
    case 15: return jx * jz * ir0;
    default: return C(0);
  }
}

// D3Q15 (Appendix basis): e^eq = -rho + j^2/rho0, eps^eq = rho - 5 j^2/rho0,
// q^eq = -7/3 j, second-order rows j_a j_b / rho0 combinations, m_xyz^eq = 0
template <class C>
LBM_HD C meq(D3Q15, int k, C drho, C jx, C jy, C jz, C ir0) {
  const C j2 = (jx * jx + jy * jy + jz * jz) * ir0;
  switch (k) {
    case 1: return -drho + j2;
    case 2: return drho - C(5) * j2;
    case 4: return C(-7.0 / 3.0) * jx;
    case 6: return C(-7.0 / 3.0) * jy;
    case 8: return C(-7.0 / 3.0) * jz;
    case 9: return C(3) * jx * jx * ir0 - j2;
    case 10: return (jy * jy - jz * jz) * ir0;
    case 11: return jx * jy * ir0;
    case 12: return jy * jz * ir0;
    case 13: return jx * jz * ir0;
    default: return C(0);
  }
}

// compile-time row properties
template <class L>
constexpr unsigned odd_row_mask() {
  unsigned m = 0;
  for (int k = 0; k < L::Q; ++k)
    if (row_is_odd<L>(k)) m |= 1u << k;
  return m;
}
template <class L>
constexpr unsigned conserved_row_mask() {
  unsigned m = 0;
  for (int k = 0; k < L::Q; ++k)
    if (L::conserved(k)) m |= 1u << k;
  return m;
}
template <class L>
struct Rows {
  static constexpr unsigned kOdd = odd_row_mask<L>();
  static constexpr unsigned kConserved = conserved_row_mask<L>();
  static __device__ __forceinline__ constexpr bool odd(int k) { return (kOdd >> k) & 1u; }
  static __device__ __forceinline__ constexpr bool cons(int k) { return (kConserved >> k) & 1u; }
};

// acc + m * v with m an integer literal after unrolling (0 and +-1 fold away)
template <class C>
__device__ __forceinline__ C madd(C acc, int m, C v) {
  if (m == 0) return acc;
  if (m == 1) return acc + v;
  if (m == -1) return acc - v;
  return acc + C(m) * v;
}

// D3Q19 collision with the moment sums and the back-transform factored by hand: the
// rows of M share partial sums over the face pairs, the edge pairs of each plane and
// all edges (rho, e, eps from the face and edge sums; the second-order rows from the
// three plane sums; q_a = j_a - 5 d_a), and the back-transform shares the common
// edge and face parts and the plane parts.  Same operator as the generic pair form
// below, with about a third fewer operations; rounding order differs.
template <class C>
LBM_HD void collide_d3q19(const C (&g)[19], C (&gp)[19], const SweepArgs<C> &a, C &drho_out) {
  C s[9], d[9];
#pragma unroll
  for (int p = 0; p < 9; ++p) {
    s[p] = g[2 * p + 1] + g[2 * p + 2];
    d[p] = g[2 * p + 1] - g[2 * p + 2];
  }
  const C F = s[0] + s[1] + s[2];
  const C Exy = s[3] + s[4], Exz = s[5] + s[6], Eyz = s[7] + s[8];
  const C E = Exy + Exz + Eyz;
  const C drho = g[0] + F + E;
  const C jx = d[0] + d[3] + d[4] + d[5] + d[6];
  const C jy = d[1] + d[3] - d[4] + d[7] + d[8];
  const C jz = d[2] + d[5] - d[6] + d[7] - d[8];
  drho_out = drho;
  const C ir0 = a.inv_rho0;
  const C Exyz = Exy + Exz - C(2) * Eyz;
  C m[19];
  m[1] = C(-30) * g[0] - C(11) * F + C(8) * E;
  m[2] = C(12) * g[0] - C(4) * F + E;
  m[4] = jx - C(5) * d[0];
  m[6] = jy - C(5) * d[1];
  m[8] = jz - C(5) * d[2];
  m[9] = C(2) * s[0] - s[1] - s[2] + Exyz;
  m[10] = C(-4) * s[0] + C(2) * (s[1] + s[2]) + Exyz;
  m[11] = s[1] - s[2] + Exy - Exz;
  m[12] = C(2) * (s[2] - s[1]) + Exy - Exz;
  m[13] = s[3] - s[4];
  m[14] = s[7] - s[8];
  m[15] = s[5] - s[6];
  m[16] = d[3] + d[4] - d[5] - d[6];
  m[17] = d[4] - d[3] + d[7] + d[8];
  m[18] = d[5] - d[6] - d[7] + d[8];
  C r[19];
#pragma unroll
  for (int k = 1; k < 19; ++k)
    if (!D3Q19::conserved(k)) r[k] = a.sn[k] * (m[k] - meq(D3Q19{}, k, drho, jx, jy, jz, ir0));
  // back-transform: even parts per pair from shared face / edge / plane terms
  const C Cf = C(-11) * r[1] - C(4) * r[2], Ce = C(8) * r[1] + r[2];
  const C A = r[9] + r[10], B = r[11] + r[12];
  const C Y = Cf - r[9] + C(2) * r[10], Z = r[11] - C(2) * r[12];
  const C Pxy = Ce + A + B, Pxz = Ce + A - B, Pyz = Ce - C(2) * A;
  C ev[9], od[9];
  ev[0] = Cf + C(2) * r[9] - C(4) * r[10];
  ev[1] = Y + Z;
  ev[2] = Y - Z;
  ev[3] = Pxy + r[13];
  ev[4] = Pxy - r[13];
  ev[5] = Pxz + r[15];
  ev[6] = Pxz - r[15];
  ev[7] = Pyz + r[14];
  ev[8] = Pyz - r[14];
  // odd parts minus the force term of the pair's first direction: with the force
  // folded into the flux rates (ra = r_a - F_a) the edge pairs share the sums
  // (ra + r16), (rb - r17), ... of their two directions
  const C F0 = a.F[0], F1 = a.F[1], F2 = a.F[2];
  const C rx = r[4] - F0, ry = r[6] - F1, rz = r[8] - F2;
  od[0] = C(-4) * rx - C(5) * F0;
  od[1] = C(-4) * ry - C(5) * F1;
  od[2] = C(-4) * rz - C(5) * F2;
  const C xa = rx + r[16], ya = ry - r[17];
  od[3] = xa + ya;
  od[4] = xa - ya;
  const C xb = rx - r[16], zb = rz + r[18];
  od[5] = xb + zb;
  od[6] = xb - zb;
  const C yc = ry + r[17], zc = rz - r[18];
  od[7] = yc + zc;
  od[8] = yc - zc;
  gp[0] = g[0] - (C(-30) * r[1] + C(12) * r[2]);
#pragma unroll
  for (int p = 0; p < 9; ++p) {
    gp[2 * p + 1] = g[2 * p + 1] - ev[p] - od[p];
    gp[2 * p + 2] = g[2 * p + 2] - ev[p] + od[p];
  }
}

// MRT collision through the factored transforms (D2Q9, D3Q15): r_k = s_k (m_k - m^eq_k)
// / |M_k|^2 on the relaxed rows, r = -F on the momentum rows (the force term), and
// g' = g - M^T r.
template <class L, class C>
LBM_HD void collide_factored(const C (&g)[L::Q], C (&gp)[L::Q], const SweepArgs<C> &a, C &drho_out) {
  constexpr int Q = L::Q;
  C m[Q];
  fmoments<C>(L{}, g, m);
  const C drho = m[0], jx = m[3], jy = m[5], jz = L::D == 3 ? m[7] : C(0);
  drho_out = drho;
  const C ir0 = a.inv_rho0;
  C r[Q];
#pragma unroll
  for (int k = 0; k < Q; ++k)
    r[k] = Rows<L>::cons(k) ? C(0) : a.sn[k] * (m[k] - meq(L{}, k, drho, jx, jy, jz, ir0));
  r[3] = -a.F[0];
  r[5] = -a.F[1];
  if constexpr (L::D == 3) r[7] = -a.F[2];
  C t[Q];
  fmt<false, C>(L{}, r, t);
#pragma unroll
  for (int i = 0; i < Q; ++i) gp[i] = g[i] - t[i];
}

// the factored form of the lattice
template <class L, class C>
LBM_HD C collide_plain(const C (&g)[L::Q], C (&gp)[L::Q], const SweepArgs<C> &a) {
  C drho;
  if constexpr (std::is_same_v<L, D3Q19>) collide_d3q19<C>(g, gp, a, drho);
  else collide_factored<L, C>(g, gp, a, drho);
  return drho;
}

// FP64 storage: the collision in block fixed point (fixed.cuh) where the node's values
// are in its range, in FP64 otherwise.
template <class L>
LBM_HD bool collide_fixed(const double (&g)[L::Q], double (&gp)[L::Q], const SweepArgs<double> &a) {
  constexpr int Q = L::Q;
  int E;
  if (!fx_block<L>(g, a.fx, E)) return false;
  i64 v[Q], t[Q], Fx = 0, Fy = 0, Fz = 0;
  for (int i = 0; i < Q; ++i) v[i] = fx_from<kFxTop<L>>(g[i], E);
  if (a.fx.force_hi != 0) {
    Fx = fx_from<kFxTop<L>>(a.F[0], E);
    Fy = fx_from<kFxTop<L>>(a.F[1], E);
    if (L::D == 3) Fz = fx_from<kFxTop<L>>(a.F[2], E);
  }
  fx_change(L{}, v, t, Fx, Fy, Fz, E, a.fx);
  for (int i = 0; i < Q; ++i) gp[i] = fx_to<kFxTop<L>>(v[i] - t[i], E);
  return true;
}

// MRT collision with the body force, deviation variables, g -> gp.  T is the
// storage type (it selects the form of the collision).  Returns whether the node's
// density is non-finite or runaway.
template <class L, class C, class T = C>
__device__ __forceinline__ bool collide(const C (&g)[L::Q], C (&gp)[L::Q], const SweepArgs<C> &a) {
  // The factored form where the sweep is bound by instruction issue: 16-bit storage (half
  // the bytes of FP32, the same instructions; 8 % faster) and the nodes that FP64
  // storage does not cover in fixed point.  FP32 storage, bound by the latency of its
  // loads as much as by issue, runs at the same speed with either form, and keeps the
  // generic form, whose rounding tracks FP64 closer (E_r 0.2 % from FP64 after 20000
  // steps, against 2.3 % with the factored form).
  if constexpr (sizeof(C) == 8) {
    if (collide_fixed<L>(g, gp, a)) return false;
  }
  if constexpr (sizeof(C) == 8 || sizeof(T) == 2) {
    return !(fabs(collide_plain<L, C>(g, gp, a)) < C(1e6));
  }
  constexpr int Q = L::Q;
  constexpr int NP = L::NP;
  C s[NP], d[NP];
#pragma unroll
  for (int p = 0; p < NP; ++p) {
    const int i = L::pair_first(p), ib = L::opp(i);
    s[p] = g[i] + g[ib];
    d[p] = g[i] - g[ib];
  }
  // conserved moments
  C drho = g[0];
#pragma unroll
  for (int p = 0; p < NP; ++p) drho += s[p];
  C jx = C(0), jy = C(0), jz = C(0);
#pragma unroll
  for (int p = 0; p < NP; ++p) {
    const int i = L::pair_first(p);
    jx = madd(jx, L::ex(i), d[p]);
    jy = madd(jy, L::ey(i), d[p]);
    jz = madd(jz, L::ez(i), d[p]);
  }
  const C ir0 = a.inv_rho0;
  // relaxed non-equilibrium parts r_k = s_k (m_k - m^eq_k) / |M_k|^2
  C r[Q];
#pragma unroll
  for (int k = 0; k < Q; ++k) {
    if (Rows<L>::cons(k)) {
      r[k] = C(0);
      continue;
    }
    C m = C(0);
    if (Rows<L>::odd(k)) {
#pragma unroll
      for (int p = 0; p < NP; ++p) m = madd(m, L::M(k, L::pair_first(p)), d[p]);
    } else {
      m = madd(m, L::M(k, 0), g[0]);
#pragma unroll
      for (int p = 0; p < NP; ++p) m = madd(m, L::M(k, L::pair_first(p)), s[p]);
    }
    r[k] = a.sn[k] * (m - meq(L{}, k, drho, jx, jy, jz, ir0));
  }
  // back-transform of the change: g' = g - sum_k M(k, i) r_k + force
  {
    C e0 = C(0);
#pragma unroll
    for (int k = 0; k < Q; ++k)
      if (!Rows<L>::cons(k) && !Rows<L>::odd(k)) e0 = madd(e0, L::M(k, 0), r[k]);
    gp[0] = g[0] - e0;
  }
#pragma unroll
  for (int p = 0; p < NP; ++p) {
    const int i = L::pair_first(p), ib = L::opp(i);
    C ev = C(0), od = C(0);
#pragma unroll
    for (int k = 0; k < Q; ++k) {
      if (Rows<L>::cons(k)) continue;
      if (Rows<L>::odd(k)) od = madd(od, L::M(k, i), r[k]);
      else ev = madd(ev, L::M(k, i), r[k]);
    }
    C fi = C(0);
    fi = madd(fi, L::ex(i), a.F[0]);
    fi = madd(fi, L::ey(i), a.F[1]);
    if (L::D == 3) fi = madd(fi, L::ez(i), a.F[2]);
    const C odd_part = od - fi;
    gp[i] = g[i] - ev - odd_part;
    gp[ib] = g[ib] - ev + odd_part;
  }
  return !(fabs(drho) < C(1e6));
}

// Wrap an index that is at most one period outside [0, n).
__device__ __forceinline__ int wrap1(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

// Linear index of the neighbour x + e_k (periodic, x-wrap skewed by (sy, sz) when
// SKEW).  The per-node part (wrapped x +- 1 and the skew-shifted rows) is computed
// once; per direction, row coordinates are wrapped only where that direction can
// leave the range, which the compiler resolves at compile time.
template <class L, bool SKEW>
struct Neighbours {
  int x, y, z, xm, xp, ym, yp, zm, zp, nx, ny, nz;
  __device__ __forceinline__ Neighbours(int x_, int y_, int z_, int nx_, int ny_, int nz_, int sy,
                                        int sz)
      : x(x_), y(y_), z(z_), nx(nx_), ny(ny_), nz(nz_) {
    xm = x - 1;
    xp = x + 1;
    const bool cm = xm < 0, cp = xp >= nx;
    if (cm) xm += nx;
    if (cp) xp -= nx;
    ym = yp = y;
    zm = zp = z;
    if (SKEW) {
      // crossing x = 0 downward lands at (nx-1, y+sy, z+sz); crossing x = nx-1 upward
      // lands at (0, y-sy, z-sz) (the field is invariant under (nx, sy, sz))
      if (cm) { ym += sy; zm += sz; }
      if (cp) { yp -= sy; zp -= sz; }
    }
  }
  __device__ __forceinline__ int operator()(int k) const {
    const int ex = L::ex(k), ey = L::ey(k), ez = L::ez(k);
    const int xx = ex < 0 ? xm : (ex > 0 ? xp : x);
    int yy = (ex < 0 ? ym : (ex > 0 ? yp : y)) + ey;
    if (ey != 0 || (SKEW && ex != 0)) yy = wrap1(yy, ny);
    int zz = 0;
    if (L::D == 3) {
      zz = (ex < 0 ? zm : (ex > 0 ? zp : z)) + ez;
      if (ez != 0 || (SKEW && ex != 0)) zz = wrap1(zz, nz);
    }
    return xx + nx * (yy + ny * zz);
  }
};

// ---------------------------------------------------------------------------
// Bulk-copy pipeline helpers (inline PTX, sm_90+): mbarrier with transaction
// count, cp.async.bulk global -> shared.
// ---------------------------------------------------------------------------
constexpr uint32_t kSuspendHintNs = 1000000;   // 1 ms upper bound per poll
constexpr int kWaitLimit = kWaitLimitDefault;

__device__ __forceinline__ uint32_t smem_addr(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)),
               "r"(bytes)
               : "memory");
}
// try_wait with a suspend-time hint: a thread whose phase has not completed sleeps
// (up to the hint) instead of spinning, so waiting warps do not take issue slots
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(done)
      : "r"(smem_addr(bar)), "r"(parity), "r"(kSuspendHintNs)
      : "memory");
  return done != 0;
}
// bounded wait: gives up after `polls` polls, each suspending for at most
// kSuspendHintNs; the default kWaitLimit polls is about 1 s, far beyond any
// legitimate copy latency
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar, uint32_t parity,
                                                  int polls = kWaitLimit) {
  for (int it = 0; it < polls; ++it)
    if (mbar_try_wait(bar, parity)) return true;
  return false;
}
__device__ __forceinline__ void bulk_copy_g2s(void *dst, const void *src, uint32_t bytes,
                                              uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_addr(dst)),
      "l"(src), "r"(bytes), "r"(smem_addr(bar))
      : "memory");
}

// Work decomposition.  A tile is a run of TW nodes along x (TW = kTileW = 64, or
// 32-node half tiles: the single-context FP64 sweep and, by choice, batches) that
// holds at least one fluid node; tiles are listed once per geometry.  A warp processes a tile TW/32 nodes per lane, one
// node after the other.  Every warp owns a private pipeline of kStages shared-memory
// stages: stage s holds the Q population row windows of one tile (each window up to
// TW + 16/sizeof(T) elements, start aligned down to 16 bytes), filled by bulk copies
// that complete on the warp's own mbarrier.  32-node tiles take more stages with 4-
// and 2-byte storage (3 and 5): a warp keeps most of its bytes in flight while a
// block still fits the shared memory of the 64-node layout.  FP64 storage takes 2
// stages of 32-node tiles or one of 64-node tiles, so that 4 blocks fit an SM (2 stages of
// 64-node tiles at 2 blocks: D2Q9 2048^2 95 against 85 us a step).  Warps never wait
// for each other.
constexpr int kWarpsPerBlock = 4;

#ifndef LBM_STAGES_4B
#define LBM_STAGES_4B 2
#endif
#ifndef LBM_STAGES_8B
#define LBM_STAGES_8B 1
#endif
#ifndef LBM_STAGES_8B_32
#define LBM_STAGES_8B_32 2
#endif
template <class T, int TW = kTileW>
struct StageShape {
  static_assert(TW == 32 || TW == 64, "tiles are one or two nodes per lane wide");
  static constexpr int kStages = TW == 64 ? (sizeof(T) == 8 ? LBM_STAGES_8B : (sizeof(T) == 4 ? LBM_STAGES_4B : 3))
                                          : (sizeof(T) == 2 ? 5 : (sizeof(T) == 8 ? LBM_STAGES_8B_32 : 3));
  static constexpr int kWidth = TW + 16 / (int)sizeof(T);   // elements per window
  static constexpr int kRecs = TW + 4;                       // record window (uint32)
};

// Byte layout of one stage: Q population windows, then the record window; after
// all stages, the barriers and the offsets (Q + 1 per stage).
template <class L, class T, int TW = kTileW>
struct StageLayout {
  using SS = StageShape<T, TW>;
  static constexpr size_t kPop = (size_t)L::Q * SS::kWidth * sizeof(T);
  static constexpr size_t kRec = kPop;
  static constexpr size_t kStage = (kRec + SS::kRecs * sizeof(uint32_t) + 15) / 16 * 16;
  static constexpr size_t kBars = SS::kStages * kStage;
  static constexpr size_t kOffs = kBars + SS::kStages * sizeof(uint64_t);
  static constexpr int kNOff = L::Q + 1;
};

// bytes of one warp's pipeline, a multiple of 128 so that every warp's stages
// start 128-byte aligned
template <class L, class T, int TW = kTileW>
__host__ __device__ constexpr size_t warp_smem_bytes() {
  using SL = StageLayout<L, T, TW>;
  return (SL::kOffs + StageShape<T, TW>::kStages * SL::kNOff * sizeof(int) + 127) / 128 * 128;
}
static_assert(warp_smem_bytes<D3Q19, float>() % 128 == 0, "warp region alignment");
static_assert(warp_smem_bytes<D3Q19, float, 32>() % 128 == 0, "warp region alignment");
static_assert(StageLayout<D3Q19, float, 32>::kRec % 16 == 0 && StageLayout<D3Q19, double, 32>::kRec % 16 == 0 &&
                  StageLayout<D3Q19, __half, 32>::kRec % 16 == 0 && StageLayout<D2Q9, __half, 32>::kRec % 16 == 0 &&
                  StageLayout<D3Q15, __half, 32>::kRec % 16 == 0 && StageLayout<D3Q15, __half>::kRec % 16 == 0,
              "record window alignment");
static_assert(StageLayout<D3Q19, float>::kRec % 16 == 0 && StageLayout<D3Q19, double>::kRec % 16 == 0 &&
                  StageLayout<D3Q19, __half>::kRec % 16 == 0 && StageLayout<D2Q9, __half>::kRec % 16 == 0,
              "record window alignment");
static_assert((StageShape<float>::kWidth * sizeof(float)) % 16 == 0, "window stride");
static_assert((StageShape<double>::kWidth * sizeof(double)) % 16 == 0, "window stride");
static_assert((StageShape<__half>::kWidth * sizeof(__half)) % 16 == 0, "window stride");

// Cut links of FP64 storage go link by link over the lanes of the warp, other storage node by
// node.  In FP64 a boundary value takes 5 instructions of 64 issue cycles each, and a
// lane per node runs them for every cut direction that any node of the warp has (some 8
// on a curved wall, a few lanes each); a lane per link runs them once for up to 32
// links: D3Q19 pipe L = 128, 164 -> 125 us a step; D2Q9 511^2, 14.4 -> 12.0.  The
// exchange between the lanes of nodes and links costs more than it saves where arithmetic is cheap
// (FP32: pipe L = 256, 271 -> 288 us; ensemble of 32 annuli, 62 -> 69).
template <class T>
__host__ __device__ constexpr bool link_parallel() {
  return per_link(sizeof(T) == 8 ? 0 : 1);
}
static_assert(StageShape<double, 32>::kRecs * 4 >= kSparseLinks * 2 + 16 && StageShape<double>::kRecs * 4 >= 2 * kSparseLinks * 2 + 16,
              "the link descriptors of a sparse tile fit the record window");

// aligned-down source of a window and the element offset of its first element
template <class E>
__device__ __forceinline__ const char *align16(const E *p, int &off_elems) {
  const char *pc = reinterpret_cast<const char *>(p);
  const char *pa = reinterpret_cast<const char *>(reinterpret_cast<uintptr_t>(pc) & ~(uintptr_t)15);
  off_elems = (int)((pc - pa) / (long long)sizeof(E));
  return pa;
}

// One warp fills one stage with everything a tile needs, lane i issuing copy i:
// lanes 0..Q-1 the population row windows (even step: window [x0, x0+TW) of slot
// i in the tile's own row; odd step: [x0 - ex_i, x0 - ex_i + TW) of slot opp(i)
// in row (y - ey_i, z - ez_i)), lane Q the tile's packed boundary records.  Every
// copy starts at the 16-byte boundary at or before its first element and covers its
// window rounded up to 16 bytes; off[] records where each first element landed.
// The offsets are stored before lane 0's arrive (release), so a lane that has
// waited on the barrier sees them.  All lanes call.
template <class L, class T, bool ODD, bool ALIGNED, class I, int TW>
__device__ __forceinline__ void issue_tile(const SweepArgs<typename Storage<T>::C> &a,
                                           const TileDesc &td, const TileLinks *tl, unsigned char *stage, int *off,
                                           uint64_t *bar) {
  using SL = StageLayout<L, T, TW>;
  constexpr int W = StageShape<T, TW>::kWidth;
  const int lane = threadIdx.x & 31;
  const int ty = td.yz & 0xffff, tz = td.yz >> 16;
  const char *src = nullptr, *src2 = nullptr;
  void *dst = nullptr, *dst2 = nullptr;
  uint32_t bytes = 0;
  if (lane < L::Q) {
    const int i = lane;
    int slot = i, yy = ty, zz = tz, xs = td.x0;
    if (ODD) {
      slot = L::opp_rt(i);
      yy = wrap1(ty - DirBits<L>::ey(i), a.ny);
      zz = (L::D == 3) ? wrap1(tz - DirBits<L>::ez(i), a.nz) : 0;
      xs = td.x0 - DirBits<L>::ex(i);
    }
    const T *pop = static_cast<const T *>(a.pop);
    const I elem = (I)slot * (I)a.S + (I)a.nx * ((I)yy + (I)a.ny * zz) + xs;
    int o;
    src = align16(pop + elem, o);
    off[i] = o;
    bytes = ((uint32_t)((o + TW) * (int)sizeof(T)) + 15u) & ~15u;
    dst = stage + (size_t)i * W * sizeof(T);
    if constexpr (ODD && ALIGNED) {
      // Windows that cross the periodic x-wrap (rows start on 16-byte boundaries):
      // the element read across x = 0 (column nx-1 of the row shifted by (+sy, +sz))
      // or across x = nx-1 (column 0 of the row shifted by (-sy, -sz)) comes from a
      // second 16-byte copy placed where the window expects it, and the main copy
      // stops at the row's end.
      constexpr int E16 = 16 / (int)sizeof(T);
      const int ex = DirBits<L>::ex(i);
      const bool lo = ex > 0 && td.x0 == 0;
      const bool hi = ex < 0 && td.x0 + TW > a.nx - 1;
      if (lo || hi) {
        const int sy = lo ? a.sy : -a.sy, sz = lo ? a.sz : -a.sz;
        const int yw = wrap1(yy + sy, a.ny);
        const int zw = (L::D == 3) ? wrap1(zz + sz, a.nz) : 0;
        const I rw = (I)slot * (I)a.S + (I)a.nx * ((I)yw + (I)a.ny * zw);
        if (lo) {
          // main copy: [0, TW) behind a 16-byte gap; chunk [nx-E16, nx) in the gap
          src = reinterpret_cast<const char *>(pop + elem + 1);
          dst = stage + ((size_t)i * W + E16) * sizeof(T);
          bytes = TW * sizeof(T);
          src2 = reinterpret_cast<const char *>(pop + rw + (a.nx - E16));
          dst2 = stage + (size_t)i * W * sizeof(T);
        } else {
          // main copy: [x0, nx); chunk [0, E16) of the wrapped row right after it
          bytes = (uint32_t)((a.nx - td.x0) * (int)sizeof(T));
          src2 = reinterpret_cast<const char *>(pop + rw);
          dst2 = stage + ((size_t)i * W + (a.nx - td.x0)) * sizeof(T);
        }
      }
    }
  } else if (lane == L::Q) {
    int o;
    if (link_parallel<T>()) {
      const int nl = tl->dense ? 0 : tl->k0 + tl->k1;     // dense tiles read them from memory
      src = align16(a.geo.ldesc + tl->l0, o);
      bytes = nl > 0 ? (((uint32_t)((o + nl) * (int)sizeof(uint16_t)) + 15u) & ~15u) : 0u;
    } else {
      const int nrec = __popcll(td.bnd);
      src = align16(a.geo.rec32 + td.rb, o);
      bytes = nrec > 0 ? (((uint32_t)((o + nrec) * (int)sizeof(uint32_t)) + 15u) & ~15u) : 0u;
    }
    off[L::Q] = o;
    dst = stage + SL::kRec;
  }
  const uint32_t total = __reduce_add_sync(0xffffffffu, bytes + (src2 ? 16u : 0u));
  __syncwarp();
  if (lane == 0) mbar_arrive_expect_tx(bar, total);
  __syncwarp();
  if (bytes) bulk_copy_g2s(dst, src, bytes, bar);
  if (src2) bulk_copy_g2s(dst2, src2, 16u, bar);
}

// A link's coefficients through the read-only (non-coherent) path.  They do not
// change during a sweep, so the compiler may issue these loads ahead of the
// boundary block's stores (which it could not do with plain loads, since a store
// of the storage type may alias them); each load then costs one L2 round trip per
// warp instead of one per cut direction in turn.
template <class C>
__device__ __forceinline__ LinkCoef<C> load_coef_nc(const LinkCoef<C> *p) {
  LinkCoef<C> c;
  if constexpr (sizeof(C) == 4) {
    const float4 v = __ldg(reinterpret_cast<const float4 *>(p));
    c.a = v.x; c.bb = v.y; c.c = v.z; c.w = v.w;
  } else {
    const double2 v0 = __ldg(reinterpret_cast<const double2 *>(p));
    const double2 v1 = __ldg(reinterpret_cast<const double2 *>(p) + 1);
    c.a = v0.x; c.bb = v0.y; c.c = v1.x; c.w = v1.y;
  }
  return c;
}

// Resident blocks per SM the register budget is sized for (launch bounds), each value the
// fastest of those around it (us a step, smaller / chosen / larger where measured):
//   D3Q19 FP32 5 (96 registers)      pipe L = 256: 282 / 274 / 276 at 4, 5, 6
//   D3Q19 16-bit 6                   pipe L = 192 BF16: 112 / 109 / 117 at 5, 6, 7
//   D3Q15 FP32 5                     131x97x113: 41.5 / 40.2 / 42.1, pipe L = 256: 225 / 215 / 217 at 4, 5, 6
//   D3Q15 16-bit 6                   pipe L = 192 BF16: 92 / 89 at 5, 6 (131x97x113 FP16: 38 / 40)
//   D2Q9 8                           2048^2: 29.2 / 29.2 / 29.6 at 7, 8, 9
// Batch sweeps read their members' arguments from memory into registers:
//   D2Q9 7                           32 annuli FP32: 58.3 / 57.5 / 61.6 at 6, 7, 8
//   D3Q19, D3Q15 5                   8 pipes FP32: 108 / 106 / 125 and 90 / 86 / 93 at 4, 5, 6
#ifndef LBM_MINBLOCKS_F32
#define LBM_MINBLOCKS_F32 5
#endif
#ifndef LBM_MINBLOCKS_D2Q9
#define LBM_MINBLOCKS_D2Q9 8
#endif
#ifndef LBM_MINBLOCKS_BATCH_D2Q9
#define LBM_MINBLOCKS_BATCH_D2Q9 7
#endif
#ifndef LBM_MINBLOCKS_BATCH_3D
#define LBM_MINBLOCKS_BATCH_3D 5
#endif
#ifndef LBM_MINBLOCKS_2B
#define LBM_MINBLOCKS_2B 6
#endif
template <class L, class T, bool BATCH>
struct MinBlocks {
  static constexpr int value =
      BATCH ? (L::Q == 9 ? LBM_MINBLOCKS_BATCH_D2Q9 : LBM_MINBLOCKS_BATCH_3D)
            : (L::Q == 9 ? LBM_MINBLOCKS_D2Q9 : (sizeof(T) == 2 ? LBM_MINBLOCKS_2B : LBM_MINBLOCKS_F32));
};
#ifndef LBM_MINBLOCKS_F64
#define LBM_MINBLOCKS_F64 4
#endif
#ifndef LBM_MINBLOCKS_BATCH_F64
#define LBM_MINBLOCKS_BATCH_F64 4
#endif
template <class L, bool BATCH>
struct MinBlocks<L, double, BATCH> {
  // 4 x 128 threads: 128 registers; batches too (an ensemble of 32 annuli: 161 us a step
  // at 2 blocks, 144 at 4, the members' arguments partly from memory)
  static constexpr int value = BATCH ? LBM_MINBLOCKS_BATCH_F64 : LBM_MINBLOCKS_F64;
};

// One fused time step.  Persistent warps: global warp w handles tiles
// w, w + W_total, ...  I is the index type of a population slot (int when
// Q*S < 2^31, else long long).
// Shared-memory offset of a window's first element when every row starts on a
// 16-byte boundary (nx*sizeof(T) % 16 == 0): the copy of an odd-step window that
// begins at x0 - ex starts 16/sizeof(T) - 1 elements early for ex = +1, one element
// early for ex = -1, exactly for ex = 0.
template <class T>
__device__ __forceinline__ constexpr int aligned_window_offset(int ex) {
  return ex > 0 ? 16 / (int)sizeof(T) - 1 : (ex < 0 ? 1 : 0);
}

// Arguments of the instance a tile belongs to: the kernel parameter for a single
// context, an entry of the instance table for a batch.
template <bool BATCH, class C>
__device__ __forceinline__ const SweepArgs<C> &args_for(const SweepArgs<C> &a, const SweepArgs<C> *inst,
                                                       const int *tile_inst, int tile) {
  if constexpr (BATCH) return inst[tile_inst[tile]];
  else return a;
}

template <class L, class T, bool ODD, bool SKEW, bool ALIGNED, class I, bool BATCH, int TW = kTileW>
__global__ void __launch_bounds__(kWarpsPerBlock * 32, MinBlocks<L, T, BATCH>::value)
    sweep_kernel(const SweepArgs<typename Storage<T>::C> a, const TileDesc *__restrict__ tiles,
                 int n_tiles, const SweepArgs<typename Storage<T>::C> *__restrict__ inst,
                 const int *__restrict__ tile_inst) {
  using C = typename Storage<T>::C;
  using SL = StageLayout<L, T, TW>;
  static_assert(SL::kRec % 16 == 0 && SL::kStage % 16 == 0, "bulk-copy destinations are 16-byte aligned");
  static_assert((StageShape<T, TW>::kWidth * sizeof(T)) % 16 == 0, "window stride");
  constexpr int Q = L::Q;
  constexpr int NS = StageShape<T, TW>::kStages;
  constexpr int W = StageShape<T, TW>::kWidth;
  constexpr int NO = SL::kNOff;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned char *wsm = smem_raw + (size_t)warp * warp_smem_bytes<L, T, TW>();
  uint64_t *bars = reinterpret_cast<uint64_t *>(wsm + SL::kBars);
  int *offs = reinterpret_cast<int *>(wsm + SL::kOffs);

  const TileLinks *const links = reinterpret_cast<const TileLinks *>(tiles + n_tiles);
  const int gw = blockIdx.x * kWarpsPerBlock + warp;
  const int nw = gridDim.x * kWarpsPerBlock;
  // The first tiles' descriptors come in before the wait for the kernel in front: they
  // change only by host copies, which this launch is ordered behind.
  TileDesc first[NS];
  TileLinks first_links[NS];
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    first[s] = TileDesc{};
    first_links[s] = TileLinks{};
    if (gw + s * nw < n_tiles) {
      first[s] = tiles[gw + s * nw];
      if constexpr (link_parallel<T>()) first_links[s] = links[gw + s * nw];
    }
  }
  if (lane == 0) {
    for (int s = 0; s < NS; ++s) mbar_init(&bars[s], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  wait_for_previous();
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    const int tile = gw + s * nw;
    if (tile < n_tiles)
      issue_tile<L, T, ODD, ALIGNED, I, TW>(args_for<BATCH>(a, inst, tile_inst, tile), first[s], first_links + s,
                               wsm + s * SL::kStage, offs + s * NO, &bars[s]);
  }

  int k = 0;
  for (int tile = gw; tile < n_tiles; tile += nw, ++k) {
    const int s = k % NS;
    // the detection wait is limited by the host-set a.wait_polls (lbm_set_wait_limit)
    const bool ok = mbar_wait_bounded(&bars[s], (uint32_t)(k / NS) & 1u, a.wait_polls);
    if (__any_sync(0xffffffffu, !ok)) {
      // a copy did not land in time: flag it, then wait (with the long default
      // limit) for every copy this warp still has in flight into its shared
      // memory before leaving, and stop
      if (lane == 0) atomicOr(args_for<BATCH>(a, inst, tile_inst, tile).status, 2);
      for (int j = 0; j < NS; ++j)
        if (tile + j * nw < n_tiles) mbar_wait_bounded(&bars[(k + j) % NS], (uint32_t)((k + j) / NS) & 1u);
      return;
    }
    const SweepArgs<C> &A = args_for<BATCH>(a, inst, tile_inst, tile);
    T *__restrict__ pop = static_cast<T *>(A.pop);
    const I S = (I)A.S;
    const int nxm1 = A.nx - 1;
    const LinkCoef<C> *coef = static_cast<const LinkCoef<C> *>(A.geo.coef);
    T *const lnk = static_cast<T *>(A.geo.lnk);
    const TileDesc td = tiles[tile];
    const int y = td.yz & 0xffff, z = td.yz >> 16;
    unsigned char *stg = wsm + s * SL::kStage;
    const T *st = reinterpret_cast<const T *>(stg);
    const uint32_t *rec_s = reinterpret_cast<const uint32_t *>(stg + SL::kRec) + offs[s * NO + Q];
    const int row = A.nx * (y + A.ny * z);
    // cut links of the tile, link by link over the lanes
    constexpr bool kLP = link_parallel<T>();
    TileLinks tl{};
    if constexpr (kLP) tl = links[tile];
    const bool tile_links = tl.k0 + tl.k1 > 0;
    C *const ex_s = reinterpret_cast<C *>(stg);
    const uint16_t *desc = tl.dense ? A.geo.ldesc + tl.l0
                                    : reinterpret_cast<const uint16_t *>(stg + SL::kRec) + offs[s * NO + Q];
    auto refill = [&]() {   // stage s consumed: fill it with the tile NS rounds ahead
      const int nt = tile + NS * nw;
      if (nt < n_tiles)
        issue_tile<L, T, ODD, ALIGNED, I, TW>(args_for<BATCH>(a, inst, tile_inst, nt), tiles[nt], links + nt,
                                 wsm + s * SL::kStage, offs + s * NO, &bars[s]);
    };
#pragma unroll 1
    for (int j = 0; j < TW / 32; ++j) {
    const int xl = j * 32 + lane;          // position inside the tile
    const int x = td.x0 + xl;
    const int n = row + x;
    const bool solid = (td.solid >> xl) & 1ull;
    const int nl = j == 0 ? tl.k0 : tl.k1;                   // links of this half
    const int l0 = tl.l0 + (j == 0 ? 0 : tl.k0);
    int boff = 0;
    uint32_t bmask = 0u;
    if (!kLP && ((td.bnd >> xl) & 1ull)) {
      const uint32_t r = rec_s[__popcll(td.bnd & ((1ull << xl) - 1ull))];
      bmask = r & ((1u << kRecShift) - 1u);
      boff = td.lb + (int)(r >> kRecShift);
      asm volatile("prefetch.global.L2 [%0];" ::"l"(coef + boff));
    }

    // lanes on the periodic x-edges: the row windows cannot follow the wrap.  A step
    // across x = 0 lands in column nx-1 of the row shifted by (+sy, +sz), across
    // x = nx-1 in column 0 of the row shifted by (-sy, -sz).
    const bool xlo = ODD && x == 0, xhi = ODD && x == nxm1;
    // node index in the row (y + dy, z + dz) shifted across the wrap, column xc
    auto across = [&](int xc, int dy, int dz) -> I {
      const int yy = wrap1(y + dy, A.ny);
      const int zz = L::D == 3 ? wrap1(z + dz, A.nz) : 0;
      return (I)xc + (I)A.nx * ((I)yy + (I)A.ny * zz);
    };
    const int sy = SKEW ? A.sy : 0, sz = SKEW ? A.sz : 0;

    // element of population i of position xs in the stage
    auto slot = [&](int i, int xs) {
      return i * W + (ALIGNED ? (ODD ? aligned_window_offset<T>(DirBits<L>::ex(i)) : 0) : offs[s * NO + i]) + xs;
    };
    if constexpr (kLP) {
      if (nl > 0) {
        if (lane < nl) asm volatile("prefetch.global.L2 [%0];" ::"l"(coef + l0 + lane));
        if constexpr (ODD) {
          // what does not arrive with the windows goes into the stage first: values
          // across the x-wrap, then the populations that arrive through a cut link,
          // left in the link buffer by the previous (even) step
          if (!ALIGNED) {
            if (xlo && !solid) {
#pragma unroll
              for (int i = 0; i < Q; ++i)
                if (L::ex(i) > 0)
                  ex_s[slot(i, xl)] = Storage<T>::load(pop + (I)L::opp(i) * S + across(nxm1, sy - L::ey(i), sz - L::ez(i)));
            }
            if (xhi && !solid) {
#pragma unroll
              for (int i = 0; i < Q; ++i)
                if (L::ex(i) < 0)
                  ex_s[slot(i, xl)] = Storage<T>::load(pop + (I)L::opp(i) * S + across(0, -sy - L::ey(i), -sz - L::ez(i)));
            }
            __syncwarp();
          }
#pragma unroll 1
          for (int k = lane; k < nl; k += 32) {
            const int e = desc[l0 - tl.l0 + k];
            ex_s[slot(L::opp_rt(e >> kLinkDirShift), j * 32 + (e & 31))] = Storage<T>::load(lnk + l0 + k);
          }
          __syncwarp();
        }
      }
    }
    C g[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const int o = ALIGNED ? (ODD ? aligned_window_offset<T>(L::ex(i)) : 0) : offs[s * NO + i];
      g[i] = Storage<T>::load(st + i * W + o + xl);
    }
    if (j == TW / 32 - 1 && !tile_links) {
      __syncwarp();
      refill();
    }
    // First half of the boundary scheme (Eqs. 2.10, 2.13) with a lane per link: the part
    // of the node's pre-collision values, read from the stage.  A lane per node runs
    // every cut direction that any node of the warp has, a few lanes at a time; a lane per link
    // runs once (a curved wall leaves some 16 links in a half that has any).
    C part[kSparseLinks / 32];
    if constexpr (kLP) {
      if (nl > 0) {
        auto first = [&](int k) {
          const int e = desc[l0 - tl.l0 + k], d = e >> kLinkDirShift, xs = j * 32 + (e & 31);
          const LinkCoef<C> c = load_coef_nc(coef + l0 + k);
          return A.one_minus_b * ex_s[slot(L::opp_rt(d), xs)] + c.a * ex_s[slot(d, xs)];
        };
#pragma unroll
        for (int r = 0; r < kSparseLinks / 32; ++r)
          if (r * 32 + lane < nl) part[r] = first(r * 32 + lane);
#pragma unroll 1
        for (int k = kSparseLinks + lane; k < nl; k += 32) lnk[l0 + k] = first(k);   // free until the step writes it
        __syncwarp();
      }
    }

    if (!solid) {
    // (a node can be on both edges when nx = 1)
    if (ODD && !ALIGNED && xlo && !(kLP && nl > 0)) {          // aligned rows: staged with the windows
#pragma unroll
      for (int i = 0; i < Q; ++i)
        if (L::ex(i) > 0)
          g[i] = Storage<T>::load(pop + (I)L::opp(i) * S + across(nxm1, sy - L::ey(i), sz - L::ez(i)));
    }
    if (ODD && !ALIGNED && xhi && !(kLP && nl > 0)) {
#pragma unroll
      for (int i = 0; i < Q; ++i)
        if (L::ex(i) < 0)
          g[i] = Storage<T>::load(pop + (I)L::opp(i) * S + across(0, -sy - L::ey(i), -sz - L::ez(i)));
    }
    if (ODD && bmask) {
      // populations that arrive through a cut link were left in the link buffer
      // by the previous (even) step
#pragma unroll
      for (int dd = 1; dd < Q; ++dd)
        if (bmask & (1u << dd))
            g[L::opp(dd)] = Storage<T>::load(lnk + boff + __popc(bmask & ((1u << dd) - 1u)));
    }

    if (A.save) {
#pragma unroll
      for (int i = 0; i < Q; ++i) A.save[(long long)i * A.N + n] = g[i];
    }

    C gp[Q];
    if (collide<L, C, T>(g, gp, A)) atomicOr(A.status, 1);

    // start of slot i: a constant operand for a single context, arithmetic for a batch
    // (whose arguments sit in memory)
    auto slot0 = [&](int i) -> I { return BATCH ? (I)i * S : (I)A.kslot[i]; };
    if (!ODD) {
#pragma unroll
      for (int i = 0; i < Q; ++i) Storage<T>::store(pop + (slot0(L::opp(i)) + (I)n), gp[i]);   // slot opp(i) of x
    } else {
      // slot i of x + e_i = column X + row Y + plane Z, each wrapped by itself: a handful
      // of selections per node and the same instructions for every node, instead of
      // separate code for interior rows, wrapped rows and the x-edges (whose
      // instruction fetches cost the FP64 odd step a fifth of its time).
      const I nx = (I)A.nx, nxy = (I)A.nx * A.ny;
      const I X[3] = {(I)(xlo ? nxm1 : x - 1), (I)x, (I)(xhi ? 0 : x + 1)};
      I Y[3][3], Z[3][3];      // [e_x + 1][e + 1]: a skewed wrap shifts the rows across it
#pragma unroll
      for (int e = 0; e < 3; ++e) {
        int ys = y, zs = z;
        if (SKEW && e == 0 && xlo) {
          ys = wrap1(ys + sy, A.ny);
          zs = wrap1(zs + sz, A.nz);
        }
        if (SKEW && e == 2 && xhi) {
          ys = wrap1(ys - sy, A.ny);
          zs = wrap1(zs - sz, A.nz);
        }
        Y[e][0] = nx * (ys == 0 ? A.ny - 1 : ys - 1);
        Y[e][1] = nx * ys;
        Y[e][2] = nx * (ys == A.ny - 1 ? 0 : ys + 1);
        Z[e][0] = L::D == 3 ? nxy * (zs == 0 ? A.nz - 1 : zs - 1) : I(0);
        Z[e][1] = L::D == 3 ? nxy * zs : I(0);
        Z[e][2] = L::D == 3 ? nxy * (zs == A.nz - 1 ? 0 : zs + 1) : I(0);
      }
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        const int ex = L::ex(i) + 1, ey = L::ey(i) + 1, ez = L::ez(i) + 1;
        Storage<T>::store(pop + (X[ex] + (Y[ex][ey] + Z[ex][ez]) + slot0(i)), gp[i]);
      }
    }

    // single-node boundary scheme on the cut links of this node (Eqs. 2.10, 2.13)
    if (bmask) {
#pragma unroll
      for (int dd = 1; dd < Q; ++dd) {
        if (bmask & (1u << dd)) {
          const int kk = boff + __popc(bmask & ((1u << dd) - 1u));
          const LinkCoef<C> c = load_coef_nc(coef + kk);
          const int i = L::opp(dd);
          const C v = A.one_minus_b * g[i] + c.a * g[dd] + c.bb * gp[i] + c.c * gp[dd] + c.w * A.wfac;
          if (!ODD) Storage<T>::store(lnk + kk, v);          // read by the next odd step
          else Storage<T>::store(pop + ((I)i * S + (I)n), v);  // slot i of x_f itself
        }
      }
    }
    if constexpr (kLP) {
      if (nl > 0) {                        // hand f' to the lanes of the links
#pragma unroll
        for (int i = 1; i < Q; ++i) {
          const int o = ALIGNED ? (ODD ? aligned_window_offset<T>(L::ex(i)) : 0) : offs[s * NO + i];
          ex_s[i * W + o + xl] = gp[i];
        }
      }
    }
    }  // !solid

    // second half of the boundary scheme: the part of the post-collision values
    if constexpr (kLP) {
      if (nl > 0) {
        __syncwarp();
        auto second = [&](int k, C p) {
          const int e = desc[l0 - tl.l0 + k], d = e >> kLinkDirShift, i = L::opp_rt(d), xs = j * 32 + (e & 31);
          const LinkCoef<C> c = load_coef_nc(coef + l0 + k);
          const C v = p + c.bb * ex_s[slot(i, xs)] + c.c * ex_s[slot(d, xs)] + c.w * A.wfac;
          if (!ODD) lnk[l0 + k] = v;                                   // read by the next odd step
          else pop[(I)(row + td.x0 + xs) + (I)i * S] = v;              // slot i of x_f itself
        };
#pragma unroll
        for (int r = 0; r < kSparseLinks / 32; ++r)
          if (r * 32 + lane < nl) second(r * 32 + lane, part[r]);
#pragma unroll 1
        for (int k = kSparseLinks + lane; k < nl; k += 32) second(k, lnk[l0 + k]);
      }
      if (j == TW / 32 - 1 && tile_links) {
        // the stage was written by these lanes: order that before the bulk copies
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        refill();
      }
    }
    }
  }
}

// Persistent grid size of one kernel instantiation on the current device
// (resident blocks per SM x SMs).  The first call on each device also raises the
// kernel's dynamic shared-memory limit there (a per-device function attribute) to
// what it uses; both are cached per device ordinal.
constexpr int kMaxDevices = 64;
template <auto Kernel>
int persistent_blocks(int threads, size_t smem) {
  static std::mutex mu;
  static int cached[kMaxDevices] = {0};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= kMaxDevices) dev = 0;
  std::lock_guard<std::mutex> lock(mu);
  if (cached[dev] == 0) {
    int sms = 0, per_sm = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, Kernel, threads, smem);
    cached[dev] = (per_sm > 0 ? per_sm : 1) * (sms > 0 ? sms : 1);
  }
  return cached[dev];
}

template <auto Kernel, class A>
void launch_persistent(const A &a, const TileDesc *tiles, int n_tiles, size_t smem, cudaStream_t st,
                       const A *inst = nullptr, const int *tile_inst = nullptr, int blocks_per_sm = 0,
                       bool prepare_only = false) {
  const int threads = kWarpsPerBlock * 32;
  int grid = persistent_blocks<Kernel>(threads, smem);
  if (blocks_per_sm > 0) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (blocks_per_sm * sms < grid) grid = blocks_per_sm * sms;
  }
  const int need = (n_tiles + kWarpsPerBlock - 1) / kWarpsPerBlock;
  if (grid > need) grid = need;
  if (!prepare_only) launch_early(Kernel, grid, threads, smem, st, a, tiles, n_tiles, inst, tile_inst);
}

// Whether an FP64 context steps in 64-node tiles (one stage a warp, the other 15 warps of
// the SM cover its copies) or 32-node half tiles (two stages).  64-node tiles share a tile's
// bookkeeping between two nodes a lane (D2Q9 1024^2: 27.5 -> 23.9 us a step, D3Q19 128^3
// box 180 -> 162, D3Q15 131 x 97 x 113 120 -> 112, pipe L = 128 122.4 -> 120.0); half tiles leave out empty halves (rows
// of 80 or 96 nodes: D3Q19 80^3 52.9 against 56.5) and spread small grids over more warps
// (D2Q9 64^2 3.9 against 5.8, 724^2 15.8 against 16.2, pipe L = 64 22.1 against 27.3).  The line:
// at least three waves of 64-node tiles over the warps of 4 blocks on 152 SMs, and at
// least 1.6 halves with fluid per tile (1.5 in the rows of 80 and 96, 1.67 in those of 131).
inline bool wide_tiles_f64(int n_tiles64, int n_half) {
  return n_tiles64 >= 3 * 152 * 4 * kWarpsPerBlock && 5ll * n_half >= 8ll * n_tiles64;
}

template <class L, class T, int TW>
cudaError_t launch_sweep_w(bool odd, const SweepArgs<typename Storage<T>::C> &a, const TileDesc *tiles, int n_tiles,
                           cudaStream_t st) {
  if (n_tiles == 0) return cudaSuccess;
  const bool skew = a.sy != 0 || a.sz != 0;
  const bool big = (long long)L::Q * a.S >= (1LL << 31);
  const size_t smem = kWarpsPerBlock * warp_smem_bytes<L, T, TW>();
  const bool aligned = ((long long)a.nx * (long long)sizeof(T)) % 16 == 0;
#define LBM_LAUNCH(O, S, I)                                                                              \
  do {                                                                                                   \
    if (aligned) launch_persistent<sweep_kernel<L, T, O, S, true, I, false, TW>>(a, tiles, n_tiles, smem, st);  \
    else launch_persistent<sweep_kernel<L, T, O, S, false, I, false, TW>>(a, tiles, n_tiles, smem, st);        \
  } while (0)
  if (big) {
    if (odd) { if (skew) LBM_LAUNCH(true, true, long long); else LBM_LAUNCH(true, false, long long); }
    else LBM_LAUNCH(false, false, long long);
  } else {
    if (odd) { if (skew) LBM_LAUNCH(true, true, int); else LBM_LAUNCH(true, false, int); }
    else LBM_LAUNCH(false, false, int);
  }
#undef LBM_LAUNCH
  return cudaGetLastError();
}

template <class L, class T>
cudaError_t launch_sweep_t(bool odd, const SweepArgs<typename Storage<T>::C> &a, const TileDesc *tiles64,
                           int n_tiles64, const TileDesc *tiles_half, int n_half, cudaStream_t st) {
  if constexpr (sizeof(T) == 8) {
    if (!wide_tiles_f64(n_tiles64, n_half)) return launch_sweep_w<L, T, 32>(odd, a, tiles_half, n_half, st);
  }
  return launch_sweep_w<L, T, kTileW>(odd, a, tiles64, n_tiles64, st);
}

// One step of a batch: the tiles of one kernel class of members in one persistent
// launch, each tile reading its member's arguments from the table.  aligned: every
// member's rows start on 16-byte boundaries (aligned-window path); skew: some
// member has a skewed x-wrap.  Batches whose slots need 64-bit indices (big) use
// the general kernel (unaligned windows, skew) for every member, in 64-node tiles.
// TW: the width of the tiles in the list (64, or 32 for lists of half tiles).
// prepare_only: set up the kernel's launch attributes without launching (done once
// before a stream capture).
template <class L, class T, int TW>
cudaError_t launch_sweep_batch_t(bool odd, const SweepArgs<typename Storage<T>::C> *inst,
                                 const TileDesc *tiles, const int *tile_inst, int n_tiles,
                                 bool big, bool aligned, bool skew, int blocks_per_sm, cudaStream_t st,
                                 bool prepare_only) {
  if (n_tiles == 0) return cudaSuccess;
  using A = SweepArgs<typename Storage<T>::C>;
  const size_t smem = kWarpsPerBlock * warp_smem_bytes<L, T, TW>();
  A dummy{};
  dummy.wait_polls = kWaitLimit;
#define LBM_LAUNCH_B(O, S, AL, I)                                                                      \
  launch_persistent<sweep_kernel<L, T, O, S, AL, I, true, TW>>(dummy, tiles, n_tiles, smem, st, inst,  \
                                                               tile_inst, blocks_per_sm, prepare_only)
  if (big) {
    if constexpr (TW != kTileW) {
      return cudaErrorInvalidValue;   // 64-bit slot indices: 64-node tiles only
    } else {
      if (odd) LBM_LAUNCH_B(true, true, false, long long);
      else LBM_LAUNCH_B(false, false, false, long long);
    }
  } else if (!odd) {
    if (aligned) LBM_LAUNCH_B(false, false, true, int);
    else LBM_LAUNCH_B(false, false, false, int);
  } else if (aligned) {
    if (skew) LBM_LAUNCH_B(true, true, true, int);
    else LBM_LAUNCH_B(true, false, true, int);
  } else {
    if (skew) LBM_LAUNCH_B(true, true, false, int);
    else LBM_LAUNCH_B(true, false, false, int);
  }
#undef LBM_LAUNCH_B
  return cudaGetLastError();
}

}  // namespace lbm
