// adjoint.cu -- discrete adjoint (reverse mode) of the fused time step, for a
// velocity-mismatch loss J = sum over masked fluid nodes of |u(x, T) - u*(x)|^2.
//
// Kernels:
//   export_state   AA layout (any storage) -> natural layout deviations g[i*N+n]
//                  in the compute type (checkpoints, segment states);
//   import_state   natural layout -> AA even layout (restore a checkpoint);
//   loss           J and lambda(T) = dJ/df(T) = 2 (u - u*).e_i / rho0;
//   adjoint_step   lambda(t) from lambda(t+1) and the pre-collision state f(t),
//                  accumulating dJ/ds_k, dJ/dq and dJ/dphi of every link.
//
// The adjoint of one step, per fluid node x (Sec. 2 and Appendix restated in
// reverse):
//   advection (Eq. 2.2b): the adjoint of f'_i(x) gathers lambda_i(x + e_i) from
//     fluid neighbours;
//   boundary (Eq. 2.13): for a cut link (x, d), i = opp(d), the new f_i(x) is
//     (1-b) f_i + bA f_d + bB f'_i + bC f'_d + bW, so lambda_i(x) of the next step
//     is sent back with those weights, and d/dgamma, d/dphi of the same
//     expression give the link gradients;
//   collision (Appendix, MRT): with mu = M^-T lambda' (M^-T = diag(1/|M_k|^2) M),
//     nu_k = (1 - s_k) mu_k for non-conserved rows and
//     nu_k = mu_k + sum_l s_l (d meq_l / d m_k) mu_l for rho and j, with the
//     derivatives of the closed-form equilibrium moments written out per lattice
//     (meq_adjoint); lambda(t) = M^T nu + boundary terms, and
//     dJ/ds_k += mu_k * (-(m_k - meq_k)).
// Adjoint entries of solid nodes are zero and stay zero (never written).
#include "fixed_adjoint.cuh"
#include "node_sums.cuh"
#include "sweep.cuh"

namespace lbm {

namespace {

constexpr int kAdjThreads = 128;
// resident blocks per SM the FP32 adjoint step is compiled for (register budget)
#ifndef LBM_ADJ_MINB_F32
#define LBM_ADJ_MINB_F32 6
#endif

__device__ __forceinline__ void atomic_add_double(double *p, double v) { atomicAdd(p, v); }

template <class L, class T, class C>
__global__ void export_state_kernel(AuxArgs a, bool odd, C *out) {
  wait_for_previous();
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < a.N;
       n += (long long)gridDim.x * blockDim.x) {
    const int cls = a.cls[n];
    C g[L::Q];
#pragma unroll
    for (int i = 0; i < L::Q; ++i) g[i] = C(0);
    if (cls != kSolid) load_node<L, T>(g, (int)n, cls, odd, a);
#pragma unroll
    for (int i = 0; i < L::Q; ++i) out[(long long)i * a.N + n] = g[i];
  }
}

template <class L, class T, class C>
__global__ void import_state_kernel(AuxArgs a, const C *in) {
  T *pop = static_cast<T *>(a.pop);
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < a.N;
       n += (long long)gridDim.x * blockDim.x) {
    const bool solid = a.cls[n] == kSolid;
#pragma unroll
    for (int i = 0; i < L::Q; ++i)
      Storage<T>::store(pop + (long long)i * a.S + n, solid ? C(0) : in[(long long)i * a.N + n]);
  }
}

// J and lambda(T) from the state in the AA layout: lambda_i = 2 (u - u*).e_i / rho0 on
// masked fluid nodes, zero elsewhere (where only the zeros are written: FP64 arithmetic
// is what this kernel would otherwise spend its time on).
template <class L, class T>
__global__ void loss_kernel(AuxArgs a, bool odd, const uint8_t *mask, const double *u_target,
                            typename Storage<T>::C *lam, double *J) {
  using C = typename Storage<T>::C;
  wait_for_previous();
  double acc = 0.0;
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < a.N;
       n += (long long)gridDim.x * blockDim.x) {
    const int cls = mask[n] ? (int)a.cls[n] : (int)kSolid;
    C v[3] = {C(0), C(0), C(0)}, vxy[2] = {C(0), C(0)}, vxz[2] = {C(0), C(0)}, vyz[2] = {C(0), C(0)};
    C vc[4] = {C(0), C(0), C(0), C(0)};
    if (cls != kSolid) {
      C g[L::Q];
      load_node<L, T>(g, (int)n, cls, odd, a);
      double d[3] = {0.0, 0.0, 0.0};
      const NodeSums s = node_sums<L>(g, a);
#pragma unroll
      for (int k = 0; k < L::D; ++k) {
        const double diff = velocity(s, a, k) - u_target[n * L::D + k];
        acc += diff * diff;
        d[k] = 2.0 / a.rho0 * diff;
        v[k] = C(d[k]);
      }
      // e_i . d for one direction of each pair (the other has the opposite sign)
      const double p = d[0] + d[1], m = d[0] - d[1];
      if (L::Q != 15) {
        vxy[0] = C(p);
        vxy[1] = C(m);
      }
      if (L::Q == 19) {
        vxz[0] = C(d[0] + d[2]);
        vxz[1] = C(d[0] - d[2]);
        vyz[0] = C(d[1] + d[2]);
        vyz[1] = C(d[1] - d[2]);
      }
      if (L::Q == 15) {
        vc[0] = C(p + d[2]);
        vc[1] = C(p - d[2]);
        vc[2] = C(m + d[2]);
        vc[3] = C(m - d[2]);
      }
    }
    if (!lam) continue;
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
      const int ex = L::ex(i), ey = L::ey(i), ez = L::ez(i);
      C w = C(0);
      if (ex && ey && ez) w = (ex * ey > 0 ? (ex * ez > 0 ? vc[0] : vc[1]) : (ex * ez > 0 ? vc[2] : vc[3])) * C(ex);
      else if (ex && ey) w = (ex * ey > 0 ? vxy[0] : vxy[1]) * C(ex);
      else if (ex && ez) w = (ex * ez > 0 ? vxz[0] : vxz[1]) * C(ex);
      else if (ey && ez) w = (ey * ez > 0 ? vyz[0] : vyz[1]) * C(ey);
      else if (ex) w = v[0] * C(ex);
      else if (ey) w = v[1] * C(ey);
      else if (ez) w = v[2] * C(ez);
      lam[(long long)i * a.N + n] = w;
    }
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0 && acc != 0.0) atomic_add_double(J, acc);
}

// Link data of the adjoint step.  The gradients with respect to a link's wall
// fraction q and wall velocity phi are linear in two sums over the steps
// (Eq. 2.13 differentiated through l(q); a(t) the step's wall-velocity factor):
//   dJ/dq   = b sum_t lambda_i (A' f_d + B' f'_i + C' f'_d) + b W' sum_t a(t) lambda_i,
//   dJ/dphi = b 2 w_i rho0 e_i / ((1 + l) c_s^2) sum_t a(t) lambda_i,
// with ' = d/dq.  The kernel accumulates only sum_t a(t) lambda_i and the first sum,
// per link in FP64, with reductions that L2 carries out (one thread adds to a link in a
// step, so their order is fixed); the host folds in the other factors.  FP32 sums would
// lose digits with the length of the run or need a flush to FP64 every sqrt(T) steps, a
// launch each (forward and backward pass, D3Q19 FP32 32^3 x 100: 1.66 ms with flushes, 1.50
// so; 64^3 x 144 4.33 and 4.17; D2Q9 FP64 96^2 x 100 1.65 and 1.61); FP32 sums that carry
// their rounding (two-sum) spill: 64^3 4.88.
struct AdjGeo {
  const void *dcoef;          // LinkCoef<C> per link: (A', B', C', 0)
  double *acc;                // 2 per link: sum lambda_i, sum lambda_i (A' g_d + B' g'_i + C' g'_d)
  FixedAdj fx;                // FP64 storage: constants of the fixed-point collision transpose
};

__device__ __forceinline__ double to_f64(double v) { return v; }
__device__ __forceinline__ double to_f64(float v) { return fx_widen(v); }

// position of row k among the non-conserved rows
template <class L>
__host__ __device__ constexpr int nc_slot(int k) {
  int s = 0;
  for (int r = 0; r < k; ++r)
    if (!L::conserved(r)) ++s;
  return s;
}
static_assert(nc_slot<D3Q19>(19) <= 16 && nc_slot<D3Q15>(15) <= 16 && nc_slot<D2Q9>(9) <= 16,
              "at most 16 relaxed rows");

// One step back in time, one node per thread.  SMALL: node indices fit in 31 bits,
// so neighbour indices come from the node's wrapped coordinates in 32-bit
// arithmetic.
template <class L, class C, bool SMALL>
__global__ void __launch_bounds__(kAdjThreads, sizeof(C) == 4 ? LBM_ADJ_MINB_F32 : 3)
    adjoint_step_kernel(const SweepArgs<C> sa, AuxArgs a, AdjGeo ag, const C *__restrict__ f,
                        const C *__restrict__ lam_in, C *__restrict__ lam_out, double *gs_part) {
  constexpr int Q = L::Q;
  const long long N = a.N;
  const long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  C gsum[Q];
#pragma unroll
  for (int k = 0; k < Q; ++k) gsum[k] = C(0);
  wait_for_previous();
  const uint8_t cls = n < N ? a.cls[n] : (uint8_t)kSolid;
  if (cls != kSolid) {
    int x, y, z;
    {
      const long long r = n / a.nx;
      x = (int)(n - r * a.nx);
      y = (int)(r % a.ny);
      z = (int)(r / a.ny);
    }
    C g[Q], lp[Q], lpre[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      g[i] = f[(long long)i * N + n];
      lpre[i] = C(0);
    }
    // advection transpose: lambda'_i(x) = lambda_i(x + e_i); solid entries of the
    // adjoint are kept at zero, so no class test is needed.  Neighbours follow the
    // periodic wrap, skewed along x by (sy, sz).
    const bool inside = x > 0 && x < a.nx - 1 && y > 0 && y < a.ny - 1 &&
                        (L::D == 2 || (z > 0 && z < a.nz - 1));
    if (inside) {
      // away from the faces of the box: a constant offset per direction
      const long long sx = a.nx, sxy = (long long)a.nx * a.ny;
      const C *base = lam_in + n;
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        long long o = (long long)i * N;
        if (L::ex(i)) o += L::ex(i);
        if (L::ey(i)) o += L::ey(i) > 0 ? sx : -sx;
        if (L::ez(i)) o += L::ez(i) > 0 ? sxy : -sxy;
        lp[i] = base[o];
      }
    } else if constexpr (SMALL) {
      const Neighbours<L, true> nb(x, y, z, a.nx, a.ny, a.nz, a.sy, a.sz);
#pragma unroll
      for (int i = 0; i < Q; ++i) lp[i] = lam_in[(long long)i * N + nb(i)];
    } else {
#pragma unroll
      for (int i = 0; i < Q; ++i)
        lp[i] = lam_in[(long long)i * N + wrap_index(x, y, z, L::ex(i), L::ey(i), L::ez(i), a.nx,
                                                     a.ny, a.nz, a.sy, a.sz)];
    }
    // boundary transpose and link gradients (Eq. 2.13)
    if (cls == kBoundary) {
      C gp[Q];
      collide<L, C>(g, gp, sa);
      const LinkCoef<C> *coef = static_cast<const LinkCoef<C> *>(sa.geo.coef);
      const int bi = a.bidx[n];
      const uint32_t mask = a.bmask[bi];
      const int off = a.boff[bi];
#pragma unroll
      for (int dd = 1; dd < Q; ++dd) {
        if (mask & (1u << dd)) {
          const int k = off + __popc(mask & ((1u << dd) - 1u));
          const LinkCoef<C> c = coef[k];
          const int i = L::opp(dd);
          const C av = lam_in[(long long)i * N + n];
          lp[i] += c.bb * av;
          lp[dd] += c.c * av;
          if constexpr (sizeof(C) == 4) {
            lpre[i] += sa.one_minus_b * av;
            lpre[dd] += c.a * av;
          }
          // deviations suffice: A' + B' + C' = 0 removes the w_i rho0 parts
          const LinkCoef<C> dc = static_cast<const LinkCoef<C> *>(ag.dcoef)[k];
          double *acc = ag.acc + 2 * (long long)k;
          atomic_add_double(acc, to_f64(av * sa.wfac));           // W and its derivatives carry the step's factor
          atomic_add_double(acc + 1, to_f64(av * (dc.a * g[dd] + dc.bb * gp[i] + dc.c * gp[dd])));
        }
      }
    }
    // collision transpose in moment space, lambda(t) = M^T nu + boundary terms
    C t[Q];
    bool done = false;
    if constexpr (sizeof(C) == 8) done = fx_adjoint<L>(g, lp, sa.fx, ag.fx, t, gsum);
    if (!done) {
      adjoint_plain<L, C>(g, lp, sa, t, gsum);
      if constexpr (sizeof(C) == 8) {
#pragma unroll
        for (int k = 0; k < Q; ++k)
          if (!Rows<L>::cons(k)) gsum[k] *= 1.0 / fx_gsum_scale<L>(k);
      }
    }
    if constexpr (sizeof(C) == 8) {
      // boundary terms of the pre-collision values (held in lpre otherwise)
      if (cls == kBoundary) {
        const LinkCoef<C> *coef = static_cast<const LinkCoef<C> *>(sa.geo.coef);
        const int bi = a.bidx[n];
        const uint32_t mask = a.bmask[bi];
        const int off = a.boff[bi];
#pragma unroll
        for (int dd = 1; dd < Q; ++dd) {
          if (mask & (1u << dd)) {
            const C ca = coef[off + __popc(mask & ((1u << dd) - 1u))].a;
            const C av = lam_in[(long long)L::opp(dd) * N + n];
            t[L::opp(dd)] += sa.one_minus_b * av;
            t[dd] += ca * av;
          }
        }
      }
    } else {
#pragma unroll
      for (int i = 0; i < Q; ++i) t[i] = lpre[i] + t[i];
    }
#pragma unroll
    for (int i = 0; i < Q; ++i) lam_out[(long long)i * N + n] = t[i];
  }
  // dJ/ds: block sums in the compute type (FP64 arithmetic is slow on this GPU),
  // added in FP64 to this block's own partial record (no atomics)
  C v[16];
#pragma unroll
  for (int j = 0; j < 16; ++j) v[j] = C(0);
#pragma unroll
  for (int k = 0; k < Q; ++k)
    if (!Rows<L>::cons(k)) v[nc_slot<L>(k)] = gsum[k];
  const C wsum = warp_sum16(v);
  __shared__ C sh[kAdjThreads / 32][16];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if ((lane & 1) == 0) sh[warp][lane >> 1] = wsum;
  __syncthreads();
  if (threadIdx.x < Q && !Rows<L>::cons(threadIdx.x)) {
    int slot = 0;
    C scale = C(1);
#pragma unroll
    for (int k = 0; k < Q; ++k)
      if (k == (int)threadIdx.x) {
        slot = nc_slot<L>(k);
        if constexpr (sizeof(C) == 8) scale = fx_gsum_scale<L>(k);
      }
    C t = C(0);
    for (int w = 0; w < kAdjThreads / 32; ++w) t += sh[w][slot];
    if constexpr (sizeof(C) == 8) t *= scale;
    gs_part[(long long)blockIdx.x * Q + threadIdx.x] += (double)t;
  }
}

// One forward step in the natural layout, for recomputing a segment (push form):
// every fluid node collides its pre-collision populations f(t) (fin) and sends
// f'_i to slot i of x + e_i in fout, which then holds f(t+1); the populations that
// arrive through a cut link come from the single-node scheme (Eqs. 2.10, 2.13)
// into the node's own slot.  Same arithmetic as the fused sweep, so the states
// agree with the forward run's; slots of solid nodes receive values nobody reads.
// Reads and writes Q values per node, against the sweep-with-save's three.
template <class L, class C, bool SMALL>
__global__ void __launch_bounds__(kAdjThreads, sizeof(C) == 4 ? 6 : 3)
    recompute_step_kernel(const SweepArgs<C> sa, AuxArgs a, const C *__restrict__ fin,
                          C *__restrict__ fout) {
  constexpr int Q = L::Q;
  const long long N = a.N;
  const long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  wait_for_previous();
  if (n >= N) return;
  C g[Q], gp[Q];
  const uint8_t cls = a.cls[n];
  if (cls == kSolid) return;
  int x, y, z;
  {
    const long long r = n / a.nx;
    x = (int)(n - r * a.nx);
    y = (int)(r % a.ny);
    z = (int)(r / a.ny);
  }
#pragma unroll
  for (int i = 0; i < Q; ++i) g[i] = fin[(long long)i * N + n];
  if (collide<L, C>(g, gp, sa)) atomicOr(sa.status, 1);
  const bool inside = x > 0 && x < a.nx - 1 && y > 0 && y < a.ny - 1 &&
                      (L::D == 2 || (z > 0 && z < a.nz - 1));
  if (inside) {
    const long long sx = a.nx, sxy = (long long)a.nx * a.ny;
    C *base = fout + n;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      long long o = (long long)i * N;
      if (L::ex(i)) o += L::ex(i);
      if (L::ey(i)) o += L::ey(i) > 0 ? sx : -sx;
      if (L::ez(i)) o += L::ez(i) > 0 ? sxy : -sxy;
      base[o] = gp[i];
    }
  } else if constexpr (SMALL) {
    const Neighbours<L, true> nb(x, y, z, a.nx, a.ny, a.nz, a.sy, a.sz);
#pragma unroll
    for (int i = 0; i < Q; ++i) fout[(long long)i * N + nb(i)] = gp[i];
  } else {
#pragma unroll
    for (int i = 0; i < Q; ++i)
      fout[(long long)i * N + wrap_index(x, y, z, L::ex(i), L::ey(i), L::ez(i), a.nx, a.ny, a.nz,
                                         a.sy, a.sz)] = gp[i];
  }
  if (cls == kBoundary) {
    const LinkCoef<C> *coef = static_cast<const LinkCoef<C> *>(sa.geo.coef);
    const int bi = a.bidx[n];
    const uint32_t mask = a.bmask[bi];
    const int off = a.boff[bi];
#pragma unroll
    for (int dd = 1; dd < Q; ++dd) {
      if (mask & (1u << dd)) {
        const LinkCoef<C> c = coef[off + __popc(mask & ((1u << dd) - 1u))];
        const int i = L::opp(dd);
        fout[(long long)i * N + n] =
            sa.one_minus_b * g[i] + c.a * g[dd] + c.bb * gp[i] + c.c * gp[dd] + c.w * sa.wfac;
      }
    }
  }
}

// add the links' sums of the last steps to their totals and clear them
__global__ void link_flush_kernel(double *acc, double *tot, long long n) {
  wait_for_previous();
  for (long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x; j < n;
       j += (long long)gridDim.x * blockDim.x) {
    tot[j] += acc[j];
    acc[j] = 0.0;
  }
}

// sum of the per-block partial records: grad_s[k] = sum_b part[b*Q + k]; block k
// sums row k with a fixed order (deterministic)
template <int Q>
__global__ void __launch_bounds__(256) gs_finish_kernel(const double *part, long long n_blocks,
                                                        double *grad_s) {
  wait_for_previous();
  const int k = blockIdx.x;
  double v = 0.0;
  for (long long b = threadIdx.x; b < n_blocks; b += blockDim.x) v += part[b * Q + k];
  __shared__ double sh[256];
  sh[threadIdx.x] = v;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) grad_s[k] = sh[0];
}

int adj_blocks(long long N) {
  long long b = (N + kAdjThreads - 1) / kAdjThreads;
  if (b > 152 * 8) b = 152 * 8;
  return (int)(b < 1 ? 1 : b);
}

}  // namespace

cudaError_t launch_export_state(int lattice, int precision, const AuxArgs &a, bool odd, void *out,
                                cudaStream_t st) {
  return with_lattice(lattice, [&](auto lat) {
    using L = decltype(lat);
    return with_storage(precision, [&](auto *tp) {
      using T = std::remove_pointer_t<decltype(tp)>;
      using C = typename Storage<T>::C;
      return launch_early(export_state_kernel<L, T, C>, adj_blocks(a.N), 256, 0, st, a, odd, static_cast<C *>(out));
    });
  });
}

cudaError_t launch_import_state(int lattice, int precision, const AuxArgs &a, const void *in,
                                cudaStream_t st) {
  return with_lattice(lattice, [&](auto lat) {
    using L = decltype(lat);
    return with_storage(precision, [&](auto *tp) {
      using T = std::remove_pointer_t<decltype(tp)>;
      using C = typename Storage<T>::C;
      import_state_kernel<L, T, C><<<adj_blocks(a.N), 256, 0, st>>>(a, static_cast<const C *>(in));
      return cudaGetLastError();
    });
  });
}

cudaError_t launch_loss(int lattice, int precision, const AuxArgs &a, bool odd, const uint8_t *mask,
                        const double *u_target, void *lam, double *J, cudaStream_t st) {
  return with_lattice(lattice, [&](auto lat) {
    using L = decltype(lat);
    return with_storage(precision, [&](auto *tp) {
      using T = std::remove_pointer_t<decltype(tp)>;
      using C = typename Storage<T>::C;
      return launch_early(loss_kernel<L, T>, adj_blocks(a.N), 256, 0, st, a, odd, mask, u_target,
                          static_cast<C *>(lam), J);
    });
  });
}

cudaError_t launch_adjoint_step(int lattice, int precision, const SweepArgs<double> &a64,
                                const SweepArgs<float> &a32, const AuxArgs &a, const void *dcoef,
                                double *link_acc, const void *f, const void *lam_in, void *lam_out,
                                double *gs_part, cudaStream_t st) {
  AdjGeo ag{dcoef, link_acc, {}};
  const unsigned blocks = (unsigned)adjoint_partial_blocks(a.N);
  const bool small = a.N < (1LL << 31);
  return with_lattice(lattice, [&](auto lat) {
    using L = decltype(lat);
    auto go = [&](const auto &sa, auto sm) {
      using C = std::remove_cv_t<std::remove_reference_t<decltype(sa.inv_rho0)>>;
      if constexpr (sizeof(C) == 8) ag.fx = fx_adj_args<L>(sa.sn);
      return launch_early(adjoint_step_kernel<L, C, decltype(sm)::value>, blocks, kAdjThreads, 0, st, sa, a, ag,
                          static_cast<const C *>(f), static_cast<const C *>(lam_in), static_cast<C *>(lam_out),
                          gs_part);
    };
    if (precision == 0) return small ? go(a64, std::true_type{}) : go(a64, std::false_type{});
    return small ? go(a32, std::true_type{}) : go(a32, std::false_type{});
  });
}

cudaError_t launch_recompute_step(int lattice, int precision, const SweepArgs<double> &a64,
                                  const SweepArgs<float> &a32, const AuxArgs &a, const void *fin,
                                  void *fout, cudaStream_t st) {
  const unsigned blocks = (unsigned)adjoint_partial_blocks(a.N);
  const bool small = a.N < (1LL << 31);
  return with_lattice(lattice, [&](auto lat) {
    using L = decltype(lat);
    auto go = [&](const auto &sa, auto sm) {
      using C = std::remove_cv_t<std::remove_reference_t<decltype(sa.inv_rho0)>>;
      return launch_early(recompute_step_kernel<L, C, decltype(sm)::value>, blocks, kAdjThreads, 0, st, sa, a,
                          static_cast<const C *>(fin), static_cast<C *>(fout));
    };
    if (precision == 0) return small ? go(a64, std::true_type{}) : go(a64, std::false_type{});
    return small ? go(a32, std::true_type{}) : go(a32, std::false_type{});
  });
}

cudaError_t launch_link_flush(double *link_acc, double *tot, long long n, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const int blocks = (int)std::min<long long>((n + 255) / 256, 152 * 8);
  return launch_early(link_flush_kernel, blocks, 256, 0, st, link_acc, tot, n);
}

long long adjoint_partial_blocks(long long N) { return (N + kAdjThreads - 1) / kAdjThreads; }

cudaError_t launch_adjoint_finish(int lattice, const double *gs_part, long long n_blocks,
                                  double *grad_s, cudaStream_t st) {
  return with_lattice(lattice, [&](auto lat) {
    constexpr int Q = decltype(lat)::Q;
    return launch_early(gs_finish_kernel<Q>, Q, 256, 0, st, gs_part, n_blocks, grad_s);
  });
}

}  // namespace lbm
