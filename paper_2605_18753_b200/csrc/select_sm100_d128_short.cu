// Routing kernel for head_dim 128, rows of up to 256 candidates (see select_sm100.cuh).
#include "select_sm100_band.cuh"

namespace dash {
DASH_SELECT_BAND(select_band_d128_short) {
  (void)cluster;      // always a plain block
  return launch_band_hd<1, 1, 128>(dm, tq, tkb, a, clusters, st);
}
}  // namespace dash
