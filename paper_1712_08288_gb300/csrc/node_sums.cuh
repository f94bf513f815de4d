// node_sums.cuh -- a node's populations at either time parity and their FP64 sums rho
// and j, for the read-out kernels (moments, error norms).
//
// The sums run in 64-bit integers aligned to the node's largest population: in FP64 they
// cost some 60 instructions (conversions and additions) at one warp instruction in 64 cycles per
// quarter SM, several times the time that the populations take to arrive from memory
// (rho and u of the D3Q19 FP32 pipe at L = 256: 2360 us in FP64, 270 here; 2048^2 D2Q9 266
// and 55).
// 32-bit and 16-bit storage: every population within 2^33 of the largest is exact, so the
// sums are too; smaller ones lose less than 2^-57 of the largest.  FP64 storage: one unit
// is 1/32 of an ulp of the largest population, where an FP64 sum rounds each
// addition.  Nodes with a non-finite value, with none above the small end of the range, or
// with one so large that a sum could leave the range of FP64, take FP64 sums.
#pragma once

#include "common.cuh"
#include "fixed.cuh"

namespace lbm {

// How a read-out kernel walks the grid: node coordinates by 32-bit arithmetic.
template <int D>
struct NodeAt {
  int x, y, z;
  bool inside;   // no neighbour across a periodic face
  __device__ __forceinline__ NodeAt(int n, const AuxArgs &a) {
    const unsigned r = (unsigned)n / (unsigned)a.nx;
    x = n - (int)r * a.nx;
    z = (int)(r / (unsigned)a.ny);
    y = (int)r - z * a.ny;
    inside = x > 0 && x < a.nx - 1 && y > 0 && y < a.ny - 1 && (D == 2 || (z > 0 && z < a.nz - 1));
  }
};

// f_i(x_n, t) - w_i rho0 for all i, in the compute type (population_address() for one)
template <class L, class T>
__device__ __forceinline__ void load_node(typename Storage<T>::C (&g)[L::Q], int n, int cls, bool odd,
                                          const AuxArgs &a) {
  const T *pop = static_cast<const T *>(a.pop) + n;
  if (!odd) {
#pragma unroll
    for (int i = 0; i < L::Q; ++i) g[i] = Storage<T>::load(pop + (long long)i * a.S);
    return;
  }
  const NodeAt<L::D> at(n, a);
  if (at.inside) {
    const long long sx = a.nx, sxy = (long long)a.nx * a.ny;
#pragma unroll
    for (int i = 0; i < L::Q; ++i)
      g[i] = Storage<T>::load(pop + ((long long)L::opp(i) * a.S - L::ex(i) - L::ey(i) * sx - L::ez(i) * sxy));
  } else {
#pragma unroll
    for (int i = 0; i < L::Q; ++i)
      g[i] = Storage<T>::load(pop - n + (long long)L::opp(i) * a.S +
                              wrap_index(at.x, at.y, at.z, -L::ex(i), -L::ey(i), -L::ez(i), a.nx, a.ny, a.nz, a.sy, a.sz));
  }
  if (cls == kBoundary) {
    const int b = a.bidx[n];
    const uint32_t m = a.bmask[b];
    const T *lnk = static_cast<const T *>(a.lnk) + a.boff[b];
#pragma unroll
    for (int d = 1; d < L::Q; ++d)
      if ((m >> d) & 1u) g[L::opp(d)] = Storage<T>::load(lnk + __popc(m & ((1u << d) - 1u)));
  }
}

// rho - rho0, j / rho0 and j of a node
struct NodeSums {
  double drho, u[3], j[3];
};

// Sums of the integers times 2^scale, by adding to the exponent of the converted sum:
// the caller has checked that scale (and scale - rho0_exp) keeps every sum of 1 to 2^63
// units within the exponents of normal numbers.  A power of two rho0 divides j exactly
// through the exponents (AuxArgs::rho0_exp), at no cost.
template <class L>
__device__ __forceinline__ NodeSums scaled_sums(const i64 (&v)[L::Q], int scale, const AuxArgs &a) {
  i64 m[L::Q];
  fmoments<i64>(L{}, v, m);   // rho and j are used, the rest is never computed
  auto times = [&](double d, int sc) {
    const int hi = __double2hiint(d);      // 0 only for d = 0
    return __hiloint2double(hi != 0 ? hi + (sc << 20) : 0, __double2loint(d));
  };
  const bool two = a.rho0_exp != AuxArgs::kNoPowerOfTwo;
  const double x = (double)m[3], y = (double)m[5], z = L::D == 3 ? (double)m[7] : 0.0;
  NodeSums r;
  r.drho = times((double)m[0], scale);
  r.j[0] = times(x, scale);
  r.j[1] = times(y, scale);
  r.j[2] = times(z, scale);
  const int su = two ? scale - a.rho0_exp : scale;
  r.u[0] = times(x, su);
  r.u[1] = times(y, su);
  r.u[2] = times(z, su);
  if (!two) {
#pragma unroll
    for (int k = 0; k < L::D; ++k) r.u[k] /= a.rho0;
  }
  return r;
}

template <class L, class C>
__device__ __forceinline__ NodeSums plain_sums(const C (&g)[L::Q], const AuxArgs &a) {
  double drho = 0.0, j[3] = {0.0, 0.0, 0.0};
#pragma unroll
  for (int i = 0; i < L::Q; ++i) {
    const double v = (double)g[i];
    drho += v;
    if (L::ex(i) != 0) j[0] += L::ex(i) * v;
    if (L::ey(i) != 0) j[1] += L::ey(i) * v;
    if (L::ez(i) != 0) j[2] += L::ez(i) * v;
  }
  return {drho, {j[0] / a.rho0, j[1] / a.rho0, j[2] / a.rho0}, {j[0], j[1], j[2]}};
}

template <class L>
__device__ __forceinline__ NodeSums node_sums(const float (&g)[L::Q], const AuxArgs &a) {
  constexpr int kTop = 57;        // 19 (2^58) < 2^63
  unsigned mx = 0;
#pragma unroll
  for (int i = 0; i < L::Q; ++i) mx = max(mx, __float_as_uint(g[i]) & 0x7fffffffu);
  const int E = (int)(mx >> 23);
  if (mx != 0 && (E < 64 || E == 255)) {   // below 64 a subnormal number could count
    return plain_sums<L>(g, a);
  }
  i64 v[L::Q];
#pragma unroll
  for (int i = 0; i < L::Q; ++i) {
    const unsigned b = __float_as_uint(g[i]);
    const int d = max(E, 64) - (int)((b >> 23) & 0xffu);
    const u64 top = (u64)(((b & 0x7fffffu) | 0x800000u) << (kTop - 23 - 32)) << 32;
    const i64 s = (i64)((int)b >> 31);
    v[i] = ((i64)fx_shr(top, d) ^ s) - s;
  }
  return scaled_sums<L>(v, max(E, 64) - 127 - kTop, a);
}

template <class L>
__device__ __forceinline__ NodeSums node_sums(const double (&g)[L::Q], const AuxArgs &a) {
  constexpr int kTop = 57;
  int mx = 0;
#pragma unroll
  for (int i = 0; i < L::Q; ++i) mx = max(mx, __double2hiint(g[i]) & 0x7fffffff);
  const int E = mx >> 20;
  // exponents of the sums' units, over rho0 too where that is a shift: see scaled_sums()
  const int Eu = a.rho0_exp != AuxArgs::kNoPowerOfTwo ? E - a.rho0_exp : E;
  if (mx != 0 && (min(E, Eu) < kFxMinExp || max(E, Eu) > 1900)) return plain_sums<L>(g, a);
  i64 v[L::Q];
#pragma unroll
  for (int i = 0; i < L::Q; ++i) v[i] = fx_from<kTop>(g[i], max(E, kFxMinExp));
  return scaled_sums<L>(v, max(E, kFxMinExp) - 1023 - kTop, a);
}

// reported velocity component: j / rho0 + g / 2
__device__ __forceinline__ double velocity(const NodeSums &s, const AuxArgs &a, int k) {
  return a.g[k] != 0.0 ? s.u[k] + 0.5 * a.g[k] : s.u[k];
}

// |x| as an ordered integer, 0 for NaN (which fmax ignores): maxima and finiteness without
// the FP64 pipe
__device__ __forceinline__ i64 magnitude_bits(double x) {
  const i64 b = __double_as_longlong(x) & 0x7fffffffffffffffll;
  return b > 0x7ff0000000000000ll ? 0 : b;
}
__device__ __forceinline__ i64 warp_max(i64 v) {
  for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ bool finite_bits(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }

}  // namespace lbm
