// Key-cache fill of the retrieval layer: K = PE(X W_K^T + b) written into the cache (Eq. 1 with
// the RoPE of Eq. 3; Section 3.3, the step at the retrieval layer).
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace ilre {

static constexpr int kFillBlockK = 64;          // model channels per pipeline stage (128 B rows)
static constexpr int kFillTileM = 256;          // tokens per output tile (128 in each CTA of the pair)
static constexpr int kFillThreads = 256;        // warps 0 and 2 TMA, warp 1 MMA, warps 4..7 epilogue
static constexpr int kRopeLoRows = 1024;        // position = hi * kRopeLoRows + lo

struct FillParams {
  long long n_tok;        // tokens of this call
  int d_model;            // multiple of kFillBlockK
  int n_kv;               // kv heads; W has n_kv * 128 rows
  long long pos0;         // position of the first token
  const uint16_t* bias;   // optional bf16 [n_kv * 128], or null
  const float2* rope_lo;  // [kRopeLoRows][64]: (cos, sin) of lo * theta^(-2c/128)
  const float2* rope_hi;  // [..][64]: (cos, sin) of hi * kRopeLoRows * theta^(-2c/128)
  uint16_t* k_cache;      // bf16 [L][n_kv][128]
  int* status;
  // Work split (fill_plan): tiles 0 .. n_wide - 1 are whole units of kFillTileM tokens by unit_width
  // channels, the others parts of units, tail_width channels wide.
  int unit_width, tail_width;
  int n_wide, n_tiles;
};

// Fills in the work split from n_tok and n_kv.
void fill_plan(int n_sm, FillParams* p);
cudaError_t launch_rope_pos_tables(float2* lo, float2* hi, int hi_rows, double theta,
                                   cudaStream_t st);
// The box of map_w has unit_width / 2 weight rows, that of map_w_tail tail_width / 2.
cudaError_t launch_fill(const CUtensorMap& map_x, const CUtensorMap& map_w, const CUtensorMap& map_w_tail,
                        const FillParams& p, bool new_tables, int n_sm, cudaStream_t st);

}  // namespace ilre
