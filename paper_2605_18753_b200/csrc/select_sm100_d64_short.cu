// Routing kernel for head_dim 64, rows of up to 256 candidates (see select_sm100.cuh).
#include "select_sm100_band.cuh"

namespace dash {
DASH_SELECT_BAND(select_band_d64_short) {
  (void)cluster;      // always a plain block
  return launch_band_hd<1, 1, 64>(dm, tq, tkb, a, clusters, st);
}
}  // namespace dash
