// Streaming chunked prefill attention of one chunk (Eq. 2 with the Lambda-shaped mask): the
// layers before the retrieval layer attend to the cached sink + sliding-window keys/values and,
// causally, to the chunk's own.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace ilre {

static constexpr int kAttnThreads = 352;     // warp 0 TMA, warp 1 S MMAs, warp 2 PV MMAs, warps 3..6 / 7..10 softmax

struct AttnParams {
  int c;             // query tokens of the chunk
  int n_prefix;      // rows of K/V visible to every query (sink + sliding window)
  int n_q, n_kv;     // query heads, kv heads
  int n_qt;          // query tiles of 128 tokens
  int split_from;    // query tiles >= split_from get one CTA per head (n_qt = none)
  float c2;          // log2(e) / sqrt(d)
  int* status;
};

size_t attn_smem_bytes();
// One CTA per (query tile, head pair) -- or per head, for the query tiles from split_from on;
// fills p.n_qt and p.split_from (n_sm: SMs of the device).  map_o: the output, bf16 [c][n_q][128], in boxes of 32 rows.
cudaError_t launch_chunk_attention(const CUtensorMap& map_q, const CUtensorMap& map_k,
                                   const CUtensorMap& map_v, const CUtensorMap& map_o, AttnParams p, int n_sm,
                                   cudaStream_t st);

}  // namespace ilre
