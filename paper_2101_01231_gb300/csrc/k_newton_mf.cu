// Host side of the matrix-free Newton prediction (k_newton_mf.cuh): tables and launch.
#include "k_newton_mf.cuh"

#include <vector>

#include "tables.h"

namespace ridg {
namespace nl {

template <int NB, int NP>
Rule<NB, NP> make_rule() {
  Rule<NB, NP> T{};
  std::vector<double> x, w, v(NB), dv(NB);
  gauss_legendre(NP, x, w);
  for (int q = 0; q < Rule<NB, NP>::H; ++q) {
    phi_values(NB, x[q], v.data(), dv.data());
    for (int b = 0; b < NB; ++b) {
      T.V[b][q] = v[b];
      T.wV[b][q] = w[q] * v[b];
      T.wD[b][q] = w[q] * dv[b];
    }
  }
  phi_values(NB, 1.0, T.ep, nullptr);
  return T;
}
template Rule<2, 2> make_rule<2, 2>();
template Rule<3, 4> make_rule<3, 4>();
template Rule<4, 5> make_rule<4, 5>();
template Rule<5, 7> make_rule<5, 7>();
template Rule<2, 3> make_rule<2, 3>();
template Rule<3, 5> make_rule<3, 5>();

}  // namespace nl

namespace mf {
namespace {

template <int NB>
Tab<NB> make_tab() {
  Tab<NB> T{};
  (Rule<NB>&)T = make_rule<NB>();
  std::vector<double> x, w, v(NB), dv(NB);
  const Tables1D t1 = tables1d(NB);
  std::vector<double> A(NB * NB), inv(NB * NB);
  for (int a = 0; a < NB; ++a) {
    for (int g = 0; g < NB; ++g)
      A[a * NB + g] = T.Mt[a][g] = t1.ep[a] * t1.ep[g] - t1.D[a * NB + g];
  }
  std::vector<int> perm;
  lu_factor(NB, A.data(), perm);  // (nonsingular at every degree)
  for (int g = 0; g < NB; ++g) {
    std::vector<double> b(NB, 0.0);
    b[g] = 1.0;
    lu_solve(NB, A.data(), perm, b.data());
    for (int a = 0; a < NB; ++a) inv[a * NB + g] = b[a];
  }
  gauss_legendre(NB, x, w);
  std::vector<double> V(NB * NB), dV(NB * NB);
  for (int n = 0; n < NB; ++n) {
    phi_values(NB, x[n], v.data(), dv.data());
    for (int b = 0; b < NB; ++b) {
      V[b * NB + n] = v[b];
      dV[b * NB + n] = dv[b];
    }
  }
  for (int n = 0; n < NB; ++n)
    for (int k = 0; k < NB; ++k) {
      T.N[k][n] = (float)V[k * NB + n];
      T.M[k][n] = (float)(0.5 * w[n] * V[k * NB + n]);
      double tn = 0.0, ti = 0.0, d = 0.0;
      for (int b = 0; b < NB; ++b) {
        tn += V[b * NB + n] * inv[b * NB + k];
        d += V[b * NB + n] * dV[b * NB + k];
        for (int c = 0; c < NB; ++c) ti += V[b * NB + n] * inv[b * NB + c] * 0.5 * w[k] * V[c * NB + k];
      }
      T.TN[n][k] = (float)tn;
      T.Ti[n][k] = (float)ti;
      T.D[n][k] = (float)(w[k] * d);
    }
  for (int n = 0; n < NB; ++n) {
    double e[2] = {0.0, 0.0};
    for (int b = 0; b < NB; ++b) {
      e[0] += V[b * NB + n] * t1.ep[b];
      e[1] += V[b * NB + n] * t1.em[b];
    }
    for (int s = 0; s < 2; ++s) {
      T.E[s][n] = (float)e[s];
      T.L[s][n] = (float)(0.5 * w[n] * e[s]);
    }
  }
  return T;
}

template <int NB, int MV, int FLUX, bool F64>
cudaError_t launch_prec(const NewtonMfArgs& a, cudaStream_t s) {
  using K = Cfg<NB, MV, F64>;
  static_assert(K::bytes <= 232448, "shared memory above the per-CTA limit");
  static const Tab<NB> tab = make_tab<NB>();
  static const Rule<NB, K::NP> jrule = make_rule<NB, K::NP>();
  auto kern = a.ninst > 0 ? newton_mf_kernel<NB, MV, FLUX, F64, true>
                          : newton_mf_kernel<NB, MV, FLUX, F64, false>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)K::bytes);
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(a.list_count, 0, sizeof(int), s);
  if (e != cudaSuccess) return e;
  kern<<<(unsigned)a.ncell, K::NT, K::bytes, s>>>(a, tab, jrule);
  return cudaGetLastError();
}

template <int NB, int MV, int FLUX>
cudaError_t launch_one(const NewtonMfArgs& a, cudaStream_t s) {
  return a.fp64 ? launch_prec<NB, MV, FLUX, true>(a, s) : launch_prec<NB, MV, FLUX, false>(a, s);
}

}  // namespace
}  // namespace mf

cudaError_t launch_newton_mf(int nb, int m, int kind, const NewtonMfArgs& a, cudaStream_t s) {
  if (kind == RIDG_FLUX_BURGERS && m == 1) {
    switch (nb) {
      case 2: return mf::launch_one<2, 1, RIDG_FLUX_BURGERS>(a, s);
      case 3: return mf::launch_one<3, 1, RIDG_FLUX_BURGERS>(a, s);
      case 4: return mf::launch_one<4, 1, RIDG_FLUX_BURGERS>(a, s);
      case 5: return mf::launch_one<5, 1, RIDG_FLUX_BURGERS>(a, s);
      default: break;
    }
  } else if (kind == RIDG_FLUX_EULER && m == 4) {
    switch (nb) {
      case 2: return mf::launch_one<2, 4, RIDG_FLUX_EULER>(a, s);
      case 3: return mf::launch_one<3, 4, RIDG_FLUX_EULER>(a, s);
      default: break;
    }
  }
  return cudaErrorInvalidValue;
}

}  // namespace ridg
