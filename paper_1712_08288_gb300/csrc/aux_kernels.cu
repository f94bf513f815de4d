// aux_kernels.cu -- kernels off the time-step path: equilibrium initialisation
// (Eq. 42), population import/export, FP64 moments (Appendix, rho and rho0 u) and
// the FP64 block reductions behind the error norms (Sec. 3.1, E_r).
//
// All of them read populations through the AA layout of the sweep: after an even
// number of steps f_i(x) sits in slot i of x, after an odd number in slot opp(i)
// of x - e_i, or in the link buffer for a cut link.  They compute in double
// whatever the storage type.
#include "common.cuh"
#include "node_sums.cuh"

namespace lbm {

namespace {

__device__ __forceinline__ double quiet_nan() { return __longlong_as_double(0x7ff8000000000000LL); }

template <class L, class T>
__global__ void init_eq_kernel(AuxArgs a, const double *rho, const double *u) {
  T *pop = static_cast<T *>(a.pop);
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < a.N;
       n += (long long)gridDim.x * blockDim.x) {
    if (a.cls[n] == kSolid) {
      for (int i = 0; i < L::Q; ++i) Storage<T>::store(pop + (long long)i * a.S + n, 0.0);
      continue;
    }
    const double drho = rho ? rho[n] - a.rho0 : 0.0;
    double ux = 0, uy = 0, uz = 0;
    if (u) {
      ux = u[n * L::D];
      uy = u[n * L::D + 1];
      if (L::D == 3) uz = u[n * L::D + 2];
    }
    // Eq. 42 minus w_i rho0, c_s^2 = 1/3: w_i (drho + rho0 (3 c + 4.5 c^2 - 1.5 u^2)) with c =
    // e_i.u, the even part shared by a direction and its opposite (FP64 instructions are
    // what this kernel costs: 128^3 D3Q19 455 -> 266 us)
    const double A = drho - 1.5 * a.rho0 * (ux * ux + uy * uy + uz * uz);
    Storage<T>::store(pop + n, L::w(0) * A);
#pragma unroll
    for (int p = 0; p < L::NP; ++p) {
      const int i = L::pair_first(p);
      const double c = L::ex(i) * ux + L::ey(i) * uy + L::ez(i) * uz, rc = a.rho0 * c;
      const double even = L::w(i) * (A + 4.5 * rc * c), odd = 3.0 * L::w(i) * rc;
      Storage<T>::store(pop + (long long)i * a.S + n, even + odd);
      Storage<T>::store(pop + (long long)L::opp(i) * a.S + n, even - odd);
    }
  }
}

template <class L, class T>
__global__ void get_pop_kernel(AuxArgs a, bool odd, double *f) {
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < a.N;
       n += (long long)gridDim.x * blockDim.x) {
    const bool solid = a.cls[n] == kSolid;
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
      double v = quiet_nan();
      if (!solid) v = L::w(i) * a.rho0 + (double)Storage<T>::load(population_address<L, T>(i, n, odd, a));
      f[(long long)i * a.N + n] = v;
    }
  }
}

template <class L, class T>
__global__ void set_pop_kernel(AuxArgs a, const double *f) {
  T *pop = static_cast<T *>(a.pop);
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < a.N;
       n += (long long)gridDim.x * blockDim.x) {
    const bool solid = a.cls[n] == kSolid;
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
      const double v = solid ? 0.0 : f[(long long)i * a.N + n] - L::w(i) * a.rho0;
      Storage<T>::store(pop + (long long)i * a.S + n, v);
    }
  }
}

// Density and velocity of every node.  One thread per node; the velocities of a warp (D
// doubles per node, node-major) pass through shared memory, so that each store covers
// whole sectors.
constexpr int kMomThreads = 256;
template <class L, class T>
__global__ void __launch_bounds__(kMomThreads) moments_kernel(AuxArgs a, bool odd, double *rho, double *u) {
  constexpr int D = L::D;
  __shared__ double sh[kMomThreads / 32][32 * D];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  wait_for_previous();
  for (long long base = (blockIdx.x * (long long)kMomThreads) + warp * 32; base < a.N;
       base += (long long)gridDim.x * kMomThreads) {
    const int n = (int)base + lane;
    double r = quiet_nan(), v[3] = {r, r, r};
    const int cls = base + lane < a.N ? (int)a.cls[n] : (int)kSolid;
    if (cls != kSolid) {
      typename Storage<T>::C g[L::Q];
      load_node<L, T>(g, n, cls, odd, a);
      const NodeSums s = node_sums<L>(g, a);
      r = a.rho0 + s.drho;
#pragma unroll
      for (int k = 0; k < D; ++k) v[k] = velocity(s, a, k);
    }
    if (rho && base + lane < a.N) rho[n] = r;
    if (u) {
#pragma unroll
      for (int k = 0; k < D; ++k) sh[warp][lane * D + k] = v[k];
      __syncwarp();
#pragma unroll
      for (int k = 0; k < D; ++k) {
        const long long o = base * D + k * 32 + lane;
        if (o < a.N * D) u[o] = sh[warp][k * 32 + lane];
      }
      __syncwarp();
    }
  }
}

constexpr int kNormThreads = 256;

template <class L, class T>
__global__ void __launch_bounds__(kNormThreads, 3)
    norm_partials_kernel(AuxArgs a, bool odd, const double *u_ref, double *u_prev,
                         double *partials) {
  wait_for_previous();
  double acc[kNormFields];
#pragma unroll
  for (int k = 0; k < kNormFields; ++k) acc[k] = 0.0;
  i64 worst = 0;
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < a.N;
       n += (long long)gridDim.x * blockDim.x) {
    const int cls = a.cls[n];
    if (cls == kSolid) continue;
    typename Storage<T>::C g[L::Q];
    load_node<L, T>(g, (int)n, cls, odd, a);
    const NodeSums s = node_sums<L>(g, a);
    const double rho = a.rho0 + s.drho;
    if (!finite_bits(rho)) acc[9] += 1.0;
    acc[3] += rho;
    acc[4] += s.j[0];
    acc[5] += s.j[1];
    acc[6] += s.j[2];
#pragma unroll
    for (int k = 0; k < L::D; ++k) {
      const double uk = velocity(s, a, k);
      if (u_ref) {
        const double r = u_ref[n * L::D + k];
        const double df = r - uk;
        acc[0] += df * df;
        acc[1] += r * r;
        worst = max(worst, magnitude_bits(df));
      }
      const double dp = uk - u_prev[n * L::D + k];
      acc[7] += dp * dp;
      acc[8] += uk * uk;
      u_prev[n * L::D + k] = uk;
    }
  }
  // block reduction (fixed order -> deterministic); 16 additions a lane for the 9 sums
  __shared__ double sh[kNormThreads / 32][kNormFields];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double v16[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) v16[k] = k < kNormFields ? acc[k] : 0.0;
  const double sum = warp_sum16(v16);
  worst = warp_max(worst);
  const int field = lane >> 1;
  if ((lane & 1) == 0 && field < kNormFields) sh[warp][field] = field == 2 ? __longlong_as_double(worst) : sum;
  __syncthreads();
  if (threadIdx.x < kNormFields) {
    const int k = threadIdx.x;
    double v = sh[0][k];
    for (int w = 1; w < kNormThreads / 32; ++w) v = (k == 2) ? fmax(v, sh[w][k]) : v + sh[w][k];
    partials[(long long)blockIdx.x * kNormFields + k] = v;
  }
}

// warp k reduces field k over the blocks' records, in a fixed order
__global__ void __launch_bounds__(32 * kNormFields) norm_finish_kernel(const double *partials, int n_blocks,
                                                                     double *out) {
  const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
  wait_for_previous();
  double v = 0.0;
#pragma unroll 8
  for (int b = lane; b < n_blocks; b += 32) {
    const double w = partials[(long long)b * kNormFields + k];
    v = (k == 2) ? fmax(v, w) : v + w;
  }
  for (int o = 16; o > 0; o >>= 1) {
    const double w = __shfl_down_sync(0xffffffffu, v, o);
    v = (k == 2) ? fmax(v, w) : v + w;
  }
  if (lane == 0) out[k] = v;
}

int aux_blocks(long long N) {
  long long b = (N + 255) / 256;
  if (b > 152 * 16) b = 152 * 16;
  if (b < 1) b = 1;
  return (int)b;
}

}  // namespace

int norm_blocks_for(long long N) {
  long long b = (N + kNormThreads - 1) / kNormThreads;
  if (b > 152 * 6) b = 152 * 6;   // whole waves of 3 blocks per SM
  if (b < 1) b = 1;
  return (int)b;
}

cudaError_t launch_init_equilibrium(int lattice, int precision, const AuxArgs &a,
                                    const double *rho, const double *u, cudaStream_t st) {
  return with_lattice(lattice, [&](auto lat) {
    using L = decltype(lat);
    return with_storage(precision, [&](auto *tp) {
      using T = std::remove_pointer_t<decltype(tp)>;
      init_eq_kernel<L, T><<<aux_blocks(a.N), 256, 0, st>>>(a, rho, u);
      return cudaGetLastError();
    });
  });
}

cudaError_t launch_get_populations(int lattice, int precision, const AuxArgs &a, bool odd,
                                   double *f, cudaStream_t st) {
  return with_lattice(lattice, [&](auto lat) {
    using L = decltype(lat);
    return with_storage(precision, [&](auto *tp) {
      using T = std::remove_pointer_t<decltype(tp)>;
      get_pop_kernel<L, T><<<aux_blocks(a.N), 256, 0, st>>>(a, odd, f);
      return cudaGetLastError();
    });
  });
}

cudaError_t launch_set_populations(int lattice, int precision, const AuxArgs &a,
                                   const double *f, cudaStream_t st) {
  return with_lattice(lattice, [&](auto lat) {
    using L = decltype(lat);
    return with_storage(precision, [&](auto *tp) {
      using T = std::remove_pointer_t<decltype(tp)>;
      set_pop_kernel<L, T><<<aux_blocks(a.N), 256, 0, st>>>(a, f);
      return cudaGetLastError();
    });
  });
}

cudaError_t launch_moments(int lattice, int precision, const AuxArgs &a, bool odd, double *rho,
                           double *u, cudaStream_t st) {
  return with_lattice(lattice, [&](auto lat) {
    using L = decltype(lat);
    return with_storage(precision, [&](auto *tp) {
      using T = std::remove_pointer_t<decltype(tp)>;
      return launch_early(moments_kernel<L, T>, aux_blocks(a.N), kMomThreads, 0, st, a, odd, rho, u);
    });
  });
}

cudaError_t launch_norm_partials(int lattice, int precision, const AuxArgs &a, bool odd,
                                 const double *u_ref, double *u_prev, double *partials,
                                 int n_blocks, cudaStream_t st) {
  return with_lattice(lattice, [&](auto lat) {
    using L = decltype(lat);
    return with_storage(precision, [&](auto *tp) {
      using T = std::remove_pointer_t<decltype(tp)>;
      return launch_early(norm_partials_kernel<L, T>, n_blocks, kNormThreads, 0, st, a, odd, u_ref, u_prev, partials);
    });
  });
}

cudaError_t launch_norm_finish(const double *partials, int n_blocks, double *out,
                               cudaStream_t st) {
  return launch_early(norm_finish_kernel, 1, 32 * kNormFields, 0, st, partials, n_blocks, out);
}

}  // namespace lbm
