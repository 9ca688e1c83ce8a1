// Routing kernel for head_dim 128, rows of more than 256 candidates (see select_sm100.cuh).
#include "select_sm100_band.cuh"

namespace dash {
DASH_SELECT_BAND(select_band_d128_long) {
  switch (cluster) {
    case 1: return launch_band_hd<3, 1, 128>(dm, tq, tkb, a, clusters, st);
    case 2: return launch_band_hd<3, 2, 128>(dm, tq, tkb, a, clusters, st);
    default: return launch_band_hd<3, 4, 128>(dm, tq, tkb, a, clusters, st);
  }
}
}  // namespace dash
