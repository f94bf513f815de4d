// fixed_host.cu -- runs the library's fixed-point arithmetic (fixed.cuh, fixed_adjoint.cuh)
// on the host for tests/test_fixed_point_host.py.
//
//   fixed_host collide|adjoint|adjoint_fp64 D2Q9|D3Q15|D3Q19 < in > out
//
//   fixed_host widen any < floats > doubles (fx_widen of each)
//
// in:  doubles n, rho0, F[3] (the force on the momentum rows), s[19], then per node g[Q]
//      and, for the adjoint forms, lambda'[Q].
// out: per node 1.0 where the fixed-point form covers it (else 0.0), then for collide g'[Q]
//      in fixed point and g'[Q] in FP64, for the adjoint forms the transpose t[Q] and dJ/ds[Q].
#include <stdio.h>
#include <string.h>

#include <vector>

#include "fixed_adjoint.cuh"

using namespace lbm;

static bool get(double *p, size_t n) { return fread(p, sizeof(double), n, stdin) == n; }
static void put(const double *p, size_t n) { fwrite(p, sizeof(double), n, stdout); }

template <class L>
static int run(bool adjoint, bool fp64) {
  double head[5], s[19];
  if (!get(head, 5) || !get(s, 19)) return 2;
  SweepArgs<double> a{};
  for (int k = 0; k < L::Q; ++k) a.sn[k] = L::conserved(k) ? 0.0 : s[k] / row_norm2<L>(k);
  for (int k = 0; k < 3; ++k) a.F[k] = head[2 + k];
  a.inv_rho0 = 1.0 / head[1];
  a.fx = fx_args<L>(s, head[1], a.F);
  const FixedAdj fa = fx_adj_args<L>(a.sn);
  for (long long n = (long long)head[0]; n > 0; --n) {
    double g[L::Q], x[L::Q], y[L::Q] = {}, z[L::Q] = {};
    if (!get(g, L::Q) || (adjoint && !get(x, L::Q))) return 2;
    bool ok;
    if (adjoint && fp64) {
      ok = true;
      adjoint_plain<L, double>(g, x, a, y, z);
    } else if (adjoint) {
      ok = fx_adjoint<L>(g, x, a.fx, fa, y, z);
      for (int k = 0; k < L::Q; ++k) z[k] *= fx_gsum_scale<L>(k);
    } else {
      ok = collide_fixed<L>(g, y, a);
      collide_plain<L>(g, z, a);
    }
    const double flag = ok ? 1.0 : 0.0;
    put(&flag, 1);
    put(y, L::Q);
    put(z, L::Q);
  }
  return 0;
}

int main(int argc, char **argv) {
  if (argc != 3) return 2;
  if (strcmp(argv[1], "widen") == 0) {
    float v;
    while (fread(&v, sizeof v, 1, stdin) == 1) {
      const double d = fx_widen(v);
      put(&d, 1);
    }
    return 0;
  }
  const bool fp64 = strcmp(argv[1], "adjoint_fp64") == 0, adjoint = fp64 || strcmp(argv[1], "adjoint") == 0;
  if (strcmp(argv[2], "D2Q9") == 0) return run<D2Q9>(adjoint, fp64);
  if (strcmp(argv[2], "D3Q15") == 0) return run<D3Q15>(adjoint, fp64);
  return run<D3Q19>(adjoint, fp64);
}
