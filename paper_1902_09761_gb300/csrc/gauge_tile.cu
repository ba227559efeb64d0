// Chebyshev iteration on the Schur complement itself, small 2D grids (kernel: gauge_tile.cuh).
#include "gauge_tile.cuh"

namespace apfc {

// Eight warps of 64 x 10 points, two units (six terms).  us per three terms, three amplitudes, at
// 256^2 / 512^2 / 1024^2 / 2048^2: 5.6 / 12.4 / 38 / 133; 12 warps of 64 x 6 5.2 / 11.4 / 40 / 140;
// 8 of 64 x 8 5.2 / 14.5 / 45 / 165; 16 of 64 x 4 5.3 / 15.5 / 47 / 173; one unit a launch 10.3 /
// 14.5 / 45 / 162 (the launch and the first loads are 6 us of it); k_gauge2d at its best height 12.7
// / 20.8 / 39 / 115.
bool launch_gauge_tile(const OpCoef& c, const GaugeTab<float>& gt, const GaugeWeights& w, const ChebBufs<float>& b,
                       int pass, int sms, cudaStream_t s, const BatchLaunch* bl) {
  using SH = TileShape<8, 10, kTileUnits, false, false>;
  static_assert(SH::TX == kTileX && SH::TY == kTileY, "gauge_tiled counts these tiles");
  if (c.jd32 != nullptr)
    return pass == 0 ? launch_tile_pass<8, 10, kTileUnits, 1, true, true>(c, gt, w, b, pass, sms, s, bl)
                     : launch_tile_pass<8, 10, kTileUnits, 1, false, true>(c, gt, w, b, pass, sms, s, bl);
  return pass == 0 ? launch_tile_pass<8, 10, kTileUnits, 1, true>(c, gt, w, b, pass, sms, s, bl)
                   : launch_tile_pass<8, 10, kTileUnits, 1, false>(c, gt, w, b, pass, sms, s, bl);
}

}  // namespace apfc
