// FP64 passes of the Chebyshev iteration on the Schur complement itself (kernel: gauge2d.cuh): one
// term a pass, one point per thread, 128 columns (bound by the FP64 pipe: a longer chain's halo
// would be computed for nothing).
#include "gauge2d.cuh"

namespace apfc {

template <>
bool launch_gauge2d<double>(int, const OpCoef& c, const GaugeTab<double>& gt, const GaugeWeights& w, int Ly,
                            const ChebBufs<double>& b, int pass, cudaStream_t s, const BatchLaunch*) {
  return pass == 0 ? launch_gauge_pass<double, kGaugeNI64, 1, 128, 3, 4, true>(c, gt, w, Ly, b, pass, s, nullptr)
                   : launch_gauge_pass<double, kGaugeNI64, 1, 128, 3, 4, false>(c, gt, w, Ly, b, pass, s, nullptr);
}

}  // namespace apfc
