// FP64 passes of the Chebyshev iteration on the Schur complement (kernel: cheb2d.cuh): one
// iteration per pass and one point per thread, 128 columns (bound by the FP64 pipe: a longer
// chain's halo would be computed for nothing).
#include "cheb2d.cuh"

namespace apfc {

namespace {

template <int M>
bool go(const OpCoef& c, const ChebStep* w, const ChebPass& cp, int Ly, const ChebBufs<double>& b, int pass,
        cudaStream_t s) {
  return pass == 0 ? launch_cheb_pass<double, M, 1, 1, 128, 2, true>(c, w, cp, Ly, b, pass, s, nullptr)
                   : launch_cheb_pass<double, M, 1, 1, 128, 2, false>(c, w, cp, Ly, b, pass, s, nullptr);
}

}  // namespace

template <>
bool launch_cheb2d<double>(int m, const OpCoef& c, const ChebStep* w, const ChebPass& cp, int Ly,
                           const ChebBufs<double>& b, int pass, cudaStream_t s, const BatchLaunch*) {
  switch (m) {
    case 1: return go<1>(c, w, cp, Ly, b, pass, s);
    case 2: return go<2>(c, w, cp, Ly, b, pass, s);
    case 3: return go<3>(c, w, cp, Ly, b, pass, s);
    case 4: return go<4>(c, w, cp, Ly, b, pass, s);
    default: return false;
  }
}

}  // namespace apfc
