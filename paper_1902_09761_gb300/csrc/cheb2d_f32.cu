// FP32 passes of the preconditioned Chebyshev iteration on the Schur complement (kernel: cheb2d.cuh):
// two points per thread at M = 1, one at M > 1 (deeper chains, more registers).
#include "cheb2d.cuh"

namespace apfc {

namespace {

template <int M, int NI, int V, int NT>
bool go(const OpCoef& c, const ChebStep* w, const ChebPass& cp, int Ly, const ChebBufs<float>& b, int pass,
        cudaStream_t s, const BatchLaunch* bl) {
  return pass == 0 ? launch_cheb_pass<float, M, NI, V, NT, 3, true>(c, w, cp, Ly, b, pass, s, bl)
                   : launch_cheb_pass<float, M, NI, V, NT, 3, false>(c, w, cp, Ly, b, pass, s, bl);
}

}  // namespace

template <>
bool launch_cheb2d<float>(int m, const OpCoef& c, const ChebStep* w, const ChebPass& cp, int Ly,
                          const ChebBufs<float>& b, int pass, cudaStream_t s, const BatchLaunch* bl) {
  switch (m) {
    case 1: return go<1, 2, 2, 64>(c, w, cp, Ly, b, pass, s, bl);
    case 2: return go<2, 1, 1, 128>(c, w, cp, Ly, b, pass, s, bl);
    case 3: return go<3, 1, 1, 128>(c, w, cp, Ly, b, pass, s, bl);
    case 4: return go<4, 1, 1, 128>(c, w, cp, Ly, b, pass, s, bl);
    default: return false;
  }
}

}  // namespace apfc
