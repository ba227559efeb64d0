// FP32 passes of the Chebyshev iteration on the Schur complement itself (kernel: gauge2d.cuh).
#include "gauge2d.cuh"

namespace apfc {

namespace {

// Three terms a pass (six stages), two points per thread, three rows ahead.  Measured at 4096^2
// (us per term): two terms 153 (at the HBM rate of its 40 bytes a point), three 123, four 126 (240
// registers, two blocks of 128 threads per SM); one point per thread 172 at best.
template <int NT>
bool go(const OpCoef& c, const GaugeTab<float>& gt, const GaugeWeights& w, int Ly, const ChebBufs<float>& b, int pass,
        cudaStream_t s, const BatchLaunch* bl, int take) {
  constexpr int MB = 384 / NT;
  return pass == 0 ? launch_gauge_pass<float, kGaugeNI32, 2, NT, 3, MB, true>(c, gt, w, Ly, b, pass, s, bl, take)
                   : launch_gauge_pass<float, kGaugeNI32, 2, NT, 3, MB, false>(c, gt, w, Ly, b, pass, s, bl, take);
}

}  // namespace

// Strips of 128 columns (variants 0, 1, 3) or 256 (2, 4, 5): as fast at 4096^2, the narrow ones ahead
// on grids that give an SM few blocks (1024^2: 37 against 51 us a pass).
bool launch_gauge2d(int tile, const OpCoef& c, const GaugeTab<float>& gt, const GaugeWeights& w, int Ly,
                    const ChebBufs<float>& b, int pass, cudaStream_t s, const BatchLaunch* bl, int take) {
  return tile == 2 || tile == 4 || tile == 5 ? go<128>(c, gt, w, Ly, b, pass, s, bl, take)
                                             : go<64>(c, gt, w, Ly, b, pass, s, bl, take);
}

}  // namespace apfc
