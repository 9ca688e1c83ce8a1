// What the tensor-core routing kernel (select_sm100_band.cuh) and its launcher (select_sm100.cu) share.  The kernel's
// instantiations are spread over four translation units, by head_dim and by the length of the rows, to be compiled in parallel.
#pragma once
#include <cuda.h>

#include "common.cuh"

namespace dash {

constexpr int SELECT_SC = 64;                 // candidate chunks per MMA block / staged summary tile
constexpr int SELECT_CLUSTER_COLS = 512;      // candidates one block (of a cluster) holds in tensor memory
constexpr int SELECT_MAX_CS = 4;              // widest cluster

struct SelectTcArgs {
  Dims dm;
  int TQ, tile_base, n_tiles;   // tiles [tile_base, tile_base + n_tiles) of every (batch, KV head) are handled here
  uint32_t tmem_cols;     // power of two >= 32 covering the widest tile
  long long plane_rows;   // rows of one bf16 plane = batch * h_kv * T_s
  uint32_t* mask;
  int* count;
  int* blk_idx;
  float* blk_bias;
  float* tau;
  StatusBlock* sb;
};

// Rows of up to 256 candidates, and longer ones in clusters of 1, 2 or 4 blocks.
#define DASH_SELECT_BAND(NAME) \
  cudaError_t NAME(const Dims& dm, int cluster, const CUtensorMap& tq, const CUtensorMap& tkb, const SelectTcArgs& a, long long clusters, cudaStream_t st)
DASH_SELECT_BAND(select_band_d64_short);
DASH_SELECT_BAND(select_band_d64_long);
DASH_SELECT_BAND(select_band_d128_short);
DASH_SELECT_BAND(select_band_d128_long);

}  // namespace dash
