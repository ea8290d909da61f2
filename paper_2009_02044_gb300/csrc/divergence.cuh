// The left side of the discrete Gauss law (Sec. 3, Eq. gauss) at one site, in
// FP64 for either state, shared by the two entry points of the residual: they
// agree to the last bits of a residual that is itself rounding.
#pragma once
#include "glasma_internal.cuh"

namespace glasma {

// d^a = sum_i [E_i(x) - U_i^dag(x-i) E_i(x-i) U_i(x-i)]^a / a_i^2, the terms of
// the directions x and y (of one weight) added up in the form that the transport
// gives: SU(3) 460 operations of the FP64 pipe, link by link 510.
template <int NC, typename R>
__device__ __forceinline__ void divergence_at(const typename V2T<R>::T* U, const R* E, const Geom& g,
                                              const SiteNbr& n, const double* ia2, double* d) {
  typedef Group<NC, double> G;
  constexpr int NA = G::NA;
  auto add = [&](int i, typename G::Acc& t) {
    const int64_t sm = nbr_m(n, i);
    double q[NA];
#pragma unroll
    for (int c = 0; c < NA; ++c) q[c] = -widen<double>(E[(int64_t)(i * NA + c) * g.V + sm]);
    G::template conj_add<true>(LinkIO<NC, R>::template load<double>(U, i, g.V, sm), q, t);
  };
  double ez[NA];
#pragma unroll
  for (int c = 0; c < NA; ++c)
    d[c] = widen<double>(E[(int64_t)c * g.V + n.s]) + widen<double>(E[(int64_t)(NA + c) * g.V + n.s]);
  typename G::Acc t = G::acc(d);
#pragma unroll (NC == 3 ? 2 : 1)
  for (int i = 0; i < 2; ++i) add(i, t);
  G::from_acc(t, d);
#pragma unroll
  for (int c = 0; c < NA; ++c) ez[c] = widen<double>(E[(int64_t)(2 * NA + c) * g.V + n.s]);
  if (n.iz > 0) {
    t = G::acc(ez);
    add(2, t);
    G::from_acc(t, ez);
  }
#pragma unroll
  for (int c = 0; c < NA; ++c) d[c] = fma(ia2[2], ez[c], ia2[0] * d[c]);
}

}  // namespace glasma
