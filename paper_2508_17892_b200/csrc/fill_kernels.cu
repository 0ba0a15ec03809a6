// Key projection of the retrieval layer fused with RoPE and the write into the key cache:
//   K[pos, g, :] = R(pos) (X[pos, :] W_K[g*128:(g+1)*128, :]^T + b)      (Eq. 1, Eq. 3)
// A dense contraction, so it runs on the tensor cores: TMA -> shared memory (128-byte
// swizzle) -> tcgen05.mma with the accumulator in tensor memory -> epilogue warps that read
// the accumulator one token per thread, rotate the channel pairs (c, c + 64) of each head,
// round to bf16 and store the cache rows.
//
// Two CTAs of a cluster share a tile of 256 tokens by `width` channels (cta_group::2): each loads
// its own 128 tokens and half of the weight rows, so that at width 256 an SM reads 8 KB of operands
// per 128 cycles of math (12 KB with one CTA per tile).  Persistent pairs walk the tiles; tiles of
// one token block are neighbours in that order, so the block's activations are read from HBM once
// and served from L2 to the other heads.
//
// Tensor pipe and board power bound long calls (100001 tokens x 4096 -> 1024 channels, one CTA per
// 128-token tile -> pairs: single calls on a cool board 641 -> 595 us = 1.41 PFLOP/s, calls in a row at the
// power cap 752 -> 679 = 1.24), the chain of one CTA's 64 blocks short ones (1024 tokens 25.4 -> 20.8 us,
// 4096 tokens 46 -> 33.9).
#include <cuda_bf16.h>

#include "fill_kernels.cuh"
#include "launch.cuh"
#include "sm100_ptx.cuh"

namespace ilre {

static constexpr int kFillStages = 7;
static constexpr int kFillBatch = 4;            // barriers tested at once
static constexpr int kFillEpilogueWarps = 4;
static constexpr int kFillTailBytes = 256;

struct FillTail {
  uint64_t full[kFillStages];       // full and acc_empty: used in the first CTA only
  uint64_t empty[kFillStages];
  uint64_t acc_full[2];
  uint64_t acc_empty[2];
  uint32_t tmem_base;
  int abort_flag;
};
static_assert(sizeof(FillTail) <= kFillTailBytes, "tail too large");

__global__ void rope_pos_table_kernel(float2* __restrict__ lo, float2* __restrict__ hi, int hi_rows,
                                      double theta) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  const int n_lo = kRopeLoRows * 64;
  if (idx >= n_lo + hi_rows * 64) return;
  const bool is_lo = idx < n_lo;
  const int e = is_lo ? idx : idx - n_lo;
  const int row = e / 64, c = e % 64;
  const double pos = is_lo ? static_cast<double>(row)
                           : static_cast<double>(row) * static_cast<double>(kRopeLoRows);
  const double ang = pos * pow(theta, -2.0 * static_cast<double>(c) / 128.0);
  double sn, cs;
  sincos(ang, &sn, &cs);
  (is_lo ? lo : hi)[e] = make_float2(static_cast<float>(cs), static_cast<float>(sn));
}

// One tile: tokens [m0, m0 + 256) by `width` channels.  width 256: the heads `head` and head + 1,
// one per CTA of the pair.  width <= 128: of head `head` the channels c0 .. c0 + width / 2 - 1
// (first CTA) and the same plus 64 (second CTA), which are each other's rotation partners.
struct FillTile {
  int m0, head, c0, width;
};

__device__ __forceinline__ FillTile fill_tile(const FillParams& p, int t) {
  FillTile x;
  int unit, part = 0;
  if (t < p.n_wide) {
    unit = t;
    x.width = p.unit_width;
  } else {
    const int parts = p.unit_width / p.tail_width;
    unit = p.n_wide + (t - p.n_wide) / parts;
    part = (t - p.n_wide) % parts;
    x.width = p.tail_width;
  }
  const int per_block = p.n_kv * 128 / p.unit_width;
  x.m0 = (unit / per_block) * kFillTileM;
  x.head = (unit % per_block) * (p.unit_width / 128);
  x.c0 = 0;
  if (x.width <= 128) {                                    // part = (head of the unit, channel block)
    const int blocks = 128 / x.width;
    x.head += part / blocks;
    x.c0 = (part % blocks) * (x.width / 2);
  }
  return x;
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kFillThreads, 1)
fill_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w,
            const __grid_constant__ CUtensorMap map_w_tail, const FillParams p) {
  constexpr int kStageBytesA = 128 * kFillBlockK * 2;                  // per CTA: 128 tokens
  constexpr int kStageBytes = 2 * kStageBytesA;                        // and up to 128 weight rows
  extern __shared__ __align__(1024) uint8_t smem[];
  const uint32_t smem_base = smem_u32(smem);
  FillTail* tail = reinterpret_cast<FillTail*>(smem + kFillStages * kStageBytes);
  volatile int* abort_flag = &tail->abort_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const int first = blockIdx.x >> 1, step = gridDim.x >> 1;
  const int k_blocks = p.d_model / kFillBlockK;

  if (threadIdx.x == 0) {
    tma_prefetch_desc(&map_x);
    tma_prefetch_desc(p.n_wide > 0 ? &map_w : &map_w_tail);
    tail->abort_flag = 0;
    if (smem_base & 1023u) {
      tail->abort_flag = 1;
      atomicCAS(p.status, 0, kDevSmemAlign);
    }
    for (int s = 0; s < kFillStages; ++s) {
      mbar_init(smem_u32(&tail->full[s]), 1);
      mbar_init(smem_u32(&tail->empty[s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&tail->acc_full[b]), 1);
      mbar_init(smem_u32(&tail->acc_empty[b]), 2 * kFillEpilogueWarps);
    }
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc_pair(smem_u32(&tail->tmem_base), 512);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  __syncwarp();
  cluster_sync_all();                      // from here on either CTA may signal the other's barriers
  tc_fence_after();
  const uint32_t tmem_base = tail->tmem_base;
  const bool run = (*abort_flag == 0);
  grid_dep_wait();                         // everything above overlaps the kernel before this one
  grid_dep_launch();

  // The loading and issuing threads test the barriers of up to kFillBatch blocks at once: a test
  // waits behind the copies or MMAs that the thread has issued before it and what follows waits for
  // its result, so a test per block cost 450 to 550 cycles per block of a narrow tile, whose four
  // MMAs take 57 cycles each.
  if (warp == 0 || warp == 2) {
    // two loading threads: warp 0 the tokens, warp 2 the weight rows
    if (lane == 0 && run) {
      const bool tokens = (warp == 0);
      int s = 0;                           // ring position as (stage, phase) counters: no division
      uint32_t phase = 0;
      bool ok = true;
      for (int t = first; t < p.n_tiles && ok; t += step) {
        const FillTile x = fill_tile(p, t);
        const CUtensorMap* map = tokens ? &map_x : (t < p.n_wide) ? &map_w : &map_w_tail;
        const int row = tokens ? x.m0 + static_cast<int>(rank) * 128
                               : (x.width == 256) ? (x.head + static_cast<int>(rank)) * 128
                                                  : x.head * 128 + static_cast<int>(rank) * 64 + x.c0;
        const uint32_t bytes = 2 * kStageBytesA + x.width * (kFillBlockK * 2);     // of both CTAs
        const uint32_t dst0 = smem_base + (tokens ? 0 : kStageBytesA);
        for (int kb = 0; kb < k_blocks && ok;) {
          bool vacant[kFillBatch];
          int s1 = s;
          uint32_t ph1 = phase;
#pragma unroll
          for (int j = 0; j < kFillBatch; ++j) {
            vacant[j] = mbar_test_wait(smem_u32(&tail->empty[s1]), ph1 ^ 1u);
            if (++s1 == kFillStages) { s1 = 0; ph1 ^= 1u; }
          }
          if (!vacant[0]) {
            ok = mbar_wait(smem_u32(&tail->empty[s]), phase ^ 1u, abort_flag, p.status, kDevWaitKEmpty);
            if (!ok) break;
            vacant[1] = false;
          }
#pragma unroll
          for (int j = 0; j < kFillBatch; ++j) {
            if (j > 0 && (!vacant[j] || kb >= k_blocks)) break;
            const uint32_t bar = smem_u32(&tail->full[s]);
            if (tokens && rank == 0) mbar_arrive_expect_tx(bar, bytes);
            tma_load_2d_pair(dst0 + s * kStageBytes, map, kb * kFillBlockK, row, cluster_addr(bar, 0));
            if (++s == kFillStages) { s = 0; phase ^= 1u; }
            ++kb;
          }
        }
      }
      // The releases of the last blocks, which no load waits for, arrive in both CTAs' barriers: this CTA
      // must not leave before they have.
      for (int j = 0; j < kFillStages && ok; ++j) {
        ok = mbar_wait(smem_u32(&tail->empty[s]), phase ^ 1u, abort_flag, p.status, kDevWaitKEmpty);
        if (++s == kFillStages) { s = 0; phase ^= 1u; }
      }
    }
  } else if (warp == 1) {
    if (lane == 0 && run && rank == 0) {
      uint32_t local = 0;
      int s = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int t = first; t < p.n_tiles && ok; t += step, ++local) {
        const FillTile x = fill_tile(p, t);
        const uint32_t idesc = umma_idesc_bf16(256, x.width);
        const uint32_t buf = local & 1u, use = local >> 1;
        ok = mbar_wait(smem_u32(&tail->acc_empty[buf]), (use & 1u) ^ 1u, abort_flag, p.status,
                       kDevWaitAccEmpty);
        if (!ok) break;
        tc_fence_after();
        for (int kb = 0; kb < k_blocks && ok;) {
          bool arrived[kFillBatch];
          int s1 = s;
          uint32_t ph1 = phase;
#pragma unroll
          for (int j = 0; j < kFillBatch; ++j) {
            arrived[j] = mbar_test_wait(smem_u32(&tail->full[s1]), ph1);
            if (++s1 == kFillStages) { s1 = 0; ph1 ^= 1u; }
          }
          if (!arrived[0]) {
            ok = mbar_wait(smem_u32(&tail->full[s]), phase, abort_flag, p.status, kDevWaitKFull);
            if (!ok) break;
            arrived[1] = false;
          }
          tc_fence_after();
#pragma unroll
          for (int j = 0; j < kFillBatch; ++j) {
            if (j > 0 && (!arrived[j] || kb >= k_blocks)) break;
            const uint64_t da = umma_desc_sw128(smem_base + s * kStageBytes);
            const uint64_t db = umma_desc_sw128(smem_base + s * kStageBytes + kStageBytesA);
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)
              umma_bf16_pair(tmem_base + buf * 256, da + ((ks * 32) >> 4), db + ((ks * 32) >> 4), idesc,
                             (kb | ks) != 0);
            umma_commit_pair(smem_u32(&tail->empty[s]));
            if (++s == kFillStages) { s = 0; phase ^= 1u; }
            ++kb;
          }
        }
        if (ok) umma_commit_pair(smem_u32(&tail->acc_full[buf]));
      }
    }
  } else if (warp >= 4) {
    // Epilogue: thread = token row of this CTA's half of the tile (TMEM lane), warp = lane quadrant;
    // 16 channel pairs at a time.
    const int quad = warp & 3;
    uint32_t local = 0;
    bool ok = run;
    for (int t = first; t < p.n_tiles && ok; t += step, ++local) {
      const FillTile x = fill_tile(p, t);
      const uint32_t buf = local & 1u, use = local >> 1;
      const int token = x.m0 + static_cast<int>(rank) * 128 + quad * 32 + lane;
      const bool live = token < p.n_tok;
      const long long pos = p.pos0 + (live ? token : 0);
      const float4* t_lo = reinterpret_cast<const float4*>(p.rope_lo + (pos % kRopeLoRows) * 64 + x.c0);
      const float4* t_hi = reinterpret_cast<const float4*>(p.rope_hi + (pos / kRopeLoRows) * 64 + x.c0);
      const int groups = (x.width == 256) ? 8 : x.width / 32;          // of 16 channel pairs
      const int hi_off = (x.width == 256) ? 64 : x.width / 2;
      const uint32_t trow = tmem_base + (static_cast<uint32_t>(quad * 32) << 16) + buf * 256;
      const uint32_t empty_bar = cluster_addr(smem_u32(&tail->acc_empty[buf]), 0);
      // (cos, sin) of pos * theta_c by angle addition of the two table entries; the first group's
      // before the accumulator is complete
      float cs[16], sn[16];
      auto angles = [&](int g) {
        const int c4 = (g & 3) * 8;                        // 16 pairs = 8 float4
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const float4 a = __ldg(t_lo + c4 + j), b = __ldg(t_hi + c4 + j);
          cs[2 * j] = fmaf(a.x, b.x, -a.y * b.y);
          sn[2 * j] = fmaf(a.y, b.x, a.x * b.y);
          cs[2 * j + 1] = fmaf(a.z, b.z, -a.w * b.w);
          sn[2 * j + 1] = fmaf(a.w, b.z, a.z * b.w);
        }
      };
      angles(0);
      ok = mbar_wait(smem_u32(&tail->acc_full[buf]), use & 1u, abort_flag, p.status, kDevWaitAccFull);
      if (!ok) break;
      tc_fence_after();
#pragma unroll 1
      for (int g = 0; g < groups; ++g) {
        const int col = (g >> 2) * 128 + (g & 3) * 16;     // width 256: four groups per head
        const int head = x.head + (g >> 2), c0 = x.c0 + (g & 3) * 16;
        float v_lo[16], v_hi[16];
        tmem_ld16(trow + col, v_lo);
        tmem_ld16(trow + col + hi_off, v_hi);
        tmem_ld_wait();
        if (g == groups - 1) {                             // accumulator fully read
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(empty_bar);
        }
        uint32_t out_lo[8], out_hi[8];
#pragma unroll
        for (int j = 0; j < 16; j += 2) {
          float l0 = v_lo[j], l1 = v_lo[j + 1], h0 = v_hi[j], h1 = v_hi[j + 1];
          if (p.bias) {
            // ordinary loads: the kernel before this one may have written the bias
            const uint16_t* bp = p.bias + head * 128 + c0 + j;
            l0 += __uint_as_float(static_cast<uint32_t>(bp[0]) << 16);
            l1 += __uint_as_float(static_cast<uint32_t>(bp[1]) << 16);
            h0 += __uint_as_float(static_cast<uint32_t>(bp[64]) << 16);
            h1 += __uint_as_float(static_cast<uint32_t>(bp[65]) << 16);
          }
          const __nv_bfloat162 pl = __floats2bfloat162_rn(fmaf(l0, cs[j], -h0 * sn[j]),
                                                          fmaf(l1, cs[j + 1], -h1 * sn[j + 1]));
          const __nv_bfloat162 ph = __floats2bfloat162_rn(fmaf(l0, sn[j], h0 * cs[j]),
                                                          fmaf(l1, sn[j + 1], h1 * cs[j + 1]));
          out_lo[j >> 1] = *reinterpret_cast<const uint32_t*>(&pl);
          out_hi[j >> 1] = *reinterpret_cast<const uint32_t*>(&ph);
        }
        if (live) {
          uint16_t* row = p.k_cache + ((p.pos0 + token) * p.n_kv + head) * 128 + c0;
          uint4* dst_lo = reinterpret_cast<uint4*>(row);
          uint4* dst_hi = reinterpret_cast<uint4*>(row + 64);
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            dst_lo[q] = make_uint4(out_lo[4 * q], out_lo[4 * q + 1], out_lo[4 * q + 2], out_lo[4 * q + 3]);
            dst_hi[q] = make_uint4(out_hi[4 * q], out_hi[4 * q + 1], out_hi[4 * q + 2], out_hi[4 * q + 3]);
          }
        }
        if (g + 1 < groups) angles(g + 1);
      }
    }
  }
  // Neither CTA may leave while the other can still signal its barriers or read its operands (every commit
  // has been waited for, by the epilogue warps or by the loading threads).
  tc_fence_before();
  __syncwarp();
  cluster_sync_all();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, 512);
  }
}

void fill_plan(int n_sm, FillParams* p) {
  // Units of 256 tokens by two heads (one with an odd number of heads), one per CTA pair and pass.
  // The units of the last, incomplete pass (all of them in a short call) are cut along the channels
  // so that they spread over more pairs.  A narrow tile costs more per channel, since the 128
  // tokens of each CTA are loaded whatever the width: `cost` is the measured time of one pass over
  // 4096 model channels in units of the widest tile's (25, 17, 14 and 12 us and about 7 us of
  // launch, set-up and output in each call).  Fewer than 16 tokens: every pair loads the same few rows, and
  // dozens of pairs hold one another up at them, so there are no more than 16 tiles narrower than a head
  // (4096 model channels, 16 heads: 64 tiles 30 to 34 us, 16 tiles 25 to 28; 32 heads: 64 tiles 32 to 34, 32
  // tiles 27 to 34; from 16 tokens on 64 tiles 24 to 26 and the wider ones no faster).
  const int widths[4] = {256, 128, 64, 32};
  const int cost[4] = {100, 70, 55, 50};
  const int workers = n_sm / 2 > 0 ? n_sm / 2 : 1;
  p->unit_width = (p->n_kv % 2 == 0) ? 256 : 128;
  const long long blocks = (p->n_tok + kFillTileM - 1) / kFillTileM;
  const long long units = blocks * (p->n_kv * 128 / p->unit_width);
  p->n_wide = static_cast<int>(units / workers * workers);
  const long long rest = units - p->n_wide;
  long long best = -1;
  for (int i = 0; i < 4; ++i) {
    if (widths[i] > p->unit_width) continue;
    if (p->n_tok < 16 && widths[i] < 128 && p->n_kv * 128 / widths[i] > 16) continue;
    const long long tiles = rest * (p->unit_width / widths[i]);
    const long long c = (tiles + workers - 1) / workers * cost[i];
    if (best < 0 || c < best) { best = c; p->tail_width = widths[i]; }
  }
  p->n_tiles = static_cast<int>(p->n_wide + rest * (p->unit_width / p->tail_width));
}

cudaError_t launch_rope_pos_tables(float2* lo, float2* hi, int hi_rows, double theta,
                                   cudaStream_t st) {
  const int n = (kRopeLoRows + hi_rows) * 64;
  rope_pos_table_kernel<<<(n + 255) / 256, 256, 0, st>>>(lo, hi, hi_rows, theta);
  return cudaGetLastError();
}

cudaError_t launch_fill(const CUtensorMap& map_x, const CUtensorMap& map_w, const CUtensorMap& map_w_tail,
                        const FillParams& p, bool new_tables, int n_sm, cudaStream_t st) {
  constexpr int kSmem = kFillStages * 2 * 128 * kFillBlockK * 2 + kFillTailBytes;
  cudaError_t e = cudaFuncSetAttribute(fill_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
  if (e != cudaSuccess) return e;
  const int workers = n_sm / 2 > 0 ? n_sm / 2 : 1;
  const int grid = 2 * (p.n_tiles < workers ? p.n_tiles : workers);
  if (new_tables) {                        // read through the non-coherent path: no overlap with their kernel
    fill_kernel<<<grid, kFillThreads, kSmem, st>>>(map_x, map_w, map_w_tail, p);
    return cudaGetLastError();
  }
  return launch_after_previous(fill_kernel, grid, kFillThreads, kSmem, st, map_x, map_w, map_w_tail, p);
}

}  // namespace ilre
