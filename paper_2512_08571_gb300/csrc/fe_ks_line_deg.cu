// One FE degree and one quadrature order of the default cell kernel (compiled once
// per pair with -DFEKS_P=<p> -DFEKS_NQX=<n_q - n_p>).
#include "fe_ks_line.cuh"
#include "fe_ks_line_ff.cuh"

#ifndef FEKS_P
#error "FEKS_P must be defined"
#endif
#ifndef FEKS_NQX
#define FEKS_NQX 0
#endif

namespace feks {

template <typename T, typename TS, int P, int NQX>
cudaError_t launch_line_deg(const Ctx& c, const LocalParams<T, TS>& prm, cudaStream_t s) {
  constexpr int NP = P + 1, NQ = NP + NQX;
  if constexpr (std::is_same<T, ff2>::value) {
    return c.cplx ? launch_line_ff_t<NP, NQ, true>(c, prm, s) : launch_line_ff_t<NP, NQ, false>(c, prm, s);
  } else {
    if constexpr (std::is_same<T, float>::value) {
      if (prm.cell_coef)
        return c.cplx ? launch_line_t<T, TS, NP, NQ, true, true>(c, prm, s)
                      : launch_line_t<T, TS, NP, NQ, false, true>(c, prm, s);
    }
    return c.cplx ? launch_line_t<T, TS, NP, NQ, true, false>(c, prm, s)
                  : launch_line_t<T, TS, NP, NQ, false, false>(c, prm, s);
  }
}

template cudaError_t launch_line_deg<double, double, FEKS_P, FEKS_NQX>(const Ctx&, const LocalParams<double, double>&,
                                                                       cudaStream_t);
template cudaError_t launch_line_deg<float, float, FEKS_P, FEKS_NQX>(const Ctx&, const LocalParams<float, float>&,
                                                                     cudaStream_t);
template cudaError_t launch_line_deg<ff2, double, FEKS_P, FEKS_NQX>(const Ctx&, const LocalParams<ff2, double>&,
                                                                    cudaStream_t);
}  // namespace feks
