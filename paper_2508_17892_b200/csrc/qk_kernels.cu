// Query-context attention kernels of the recall path (Eq. 4 and Eq. 5 of the paper).
//
// The [heads, q_len, L] probability tensor is never written to memory.  Two passes over the
// key cache, both TMA -> shared memory -> tcgen05.mma -> tensor memory:
//   row statistics: D[row, key] tiles, one thread per query row keeps an online (max, sum-exp);
//   scores:         D[key, row] tiles (operands swapped), one thread per context position keeps
//                   max over rows of (logit - lse_row); exp is monotone, so one exp per position
//                   is taken afterwards.
#include "launch.cuh"
#include "qk_kernels.cuh"
#include <utility>
#include "sm100_ptx.cuh"

namespace ilre {

// Clears the per-run state: encoded scores, empty bitmap, selection state.
__device__ __forceinline__ void clear_state(const PrepParams& p, long long tid, long long nthreads) {
  for (long long t = tid; t < p.L; t += nthreads) p.enc[t] = 0u;
  const long long n_words = (p.L + 31) / 32;
  for (long long w = tid; w < n_words; w += nthreads) {
    const long long left = p.L - p.n_sink - w * 32;       // bits past the end never look free
    const uint32_t bits = (left >= 32) ? 0u : (left <= 0) ? 0xFFFFFFFFu : 0xFFFFFFFFu << left;
    p.bitmap[w] = bits;
  }
  for (long long e = tid; e < p.hist_words; e += nthreads) p.hist[e] = 0u;
  if (tid == 0) *p.grid_barrier = 0u;
  for (long long c = tid; c < p.sel_state_words; c += nthreads) p.cand_count[c] = 0u;
}

// ---------------------------------------------------------------------------------------
// shared-memory tail layout (after the Q block and the K stages)
// ---------------------------------------------------------------------------------------
struct SmemTail {
  uint64_t q_full;
  uint64_t k_full[kMaxStages];
  uint64_t k_empty[kMaxStages];
  uint64_t acc_full[4];
  uint64_t acc_empty[4];
  uint32_t tmem_base;
  int abort_flag;
  long long stamp_cycles;            // start of the optional clock stamp (kept out of registers)
  unsigned long long stamp_ns;
};
static_assert(sizeof(SmemTail) <= kSmemTailBytes, "tail too large");

struct CtaItem {
  int chunk, group, g;
  int tile_begin, n_tiles;
  // The statistics pass walks its key tiles upwards, the scores pass downwards: what the former
  // read last is still in L2 when the latter starts.
  __device__ __forceinline__ int tile_down(int i) const { return tile_begin + n_tiles - 1 - i; }
};

__device__ __forceinline__ CtaItem decode_item(const QkParams& p, int item) {
  CtaItem it;
  it.chunk = item / p.n_groups;
  it.group = item % p.n_groups;
  it.g = it.group / p.n_rb;
  const long long t0 = static_cast<long long>(it.chunk) * p.n_tiles / p.cpg;
  const long long t1 = static_cast<long long>(it.chunk + 1) * p.n_tiles / p.cpg;
  it.tile_begin = static_cast<int>(t0);
  it.n_tiles = static_cast<int>(t1 - t0);
  return it;
}

// Common prologue: barrier init, TMEM allocation.  Returns the TMEM base address.
__device__ __forceinline__ uint32_t cta_setup(SmemTail* tail, uint32_t smem_base, int stages,
                                              int n_acc, int acc_readers, int* status,
                                              int k_releasers, const CUtensorMap* tmapK, const CUtensorMap* tmapQ) {
  const int warp = threadIdx.x >> 5;
  if (threadIdx.x == 32) {                         // the descriptors, while this CTA sets itself up
    tma_prefetch_desc(tmapK);
    tma_prefetch_desc(tmapQ);
  }
  if (threadIdx.x == 0) {
    tail->abort_flag = 0;
    if (smem_base & 1023u) {                       // swizzled tiles need 1024-byte alignment
      tail->abort_flag = 1;
      atomicCAS(status, 0, kDevSmemAlign);
    }
    mbar_init(smem_u32(&tail->q_full), 1);
    for (int s = 0; s < stages; ++s) {
      mbar_init(smem_u32(&tail->k_full[s]), 1);
      mbar_init(smem_u32(&tail->k_empty[s]), k_releasers);
    }
    for (int b = 0; b < n_acc; ++b) {
      mbar_init(smem_u32(&tail->acc_full[b]), 1);
      mbar_init(smem_u32(&tail->acc_empty[b]), acc_readers);
    }
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&tail->tmem_base), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  return tail->tmem_base;
}

__device__ __forceinline__ void cta_teardown(uint32_t tmem_base) {
  tc_fence_before();
  __syncthreads();
  if ((threadIdx.x >> 5) == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
}

// A box of query rows of kv head g from row `row` on, channels 64 kb ..: from the packed copy, or straight from
// the caller's [q_len][n_q][128] array, whose rows of one kv head are `group` heads of consecutive tokens.
__device__ __forceinline__ void load_query_tile(const CUtensorMap* tmapQ, const QkParams& p, int g, int row, int kb,
                                                uint32_t dst, uint32_t bar) {
  if (p.group > 0) tma_load_3d(dst, tmapQ, kb * 64, g * p.group, row / p.group, bar);
  else tma_load_2d(dst, tmapQ, kb * 64, g * p.kv_rows + row, bar);
}

// TMA producer: the resident Q block of mts row tiles once, then the K tiles of this CTA's key range.  Row tile
// `copied` (-1: none) is made of copies of its first copy_rows rows, in boxes of 32 rows (tmapQ32).
__device__ __forceinline__ void producer_loop(const CUtensorMap* tmapK, const CUtensorMap* tmapQ, const CUtensorMap* tmapQ32,
                                              const QkParams& p, const CtaItem& it,
                                              SmemTail* tail, uint32_t q_s, uint32_t k_s, bool down,
                                              int stages, int mts, int copied = -1, int copy_rows = 128, int skip_tiles = 0) {
  volatile int* abort_flag = &tail->abort_flag;
  const uint32_t qf = smem_u32(&tail->q_full);
  mbar_arrive_expect_tx(qf, static_cast<uint32_t>(mts) * (128u * 256u));
  const int row0 = (it.group % p.n_rb) * p.rb_rows;
  for (int kb = 0; kb < 2; ++kb)
    for (int mt = 0; mt < mts; ++mt) {
      const uint32_t dst = q_s + kb * mts * 16384 + mt * 16384;
      if (mt != copied) load_query_tile(tmapQ, p, it.g, row0 + mt * 128, kb, dst, qf);
      else                                                   // the same rows again in each copy
        for (int quad = 0; quad < 4; ++quad)
          load_query_tile(tmapQ32, p, it.g, row0 + mt * 128 + quad * 32 % copy_rows, kb, dst + quad * 4096, qf);
    }
  // ring position as (stage, phase) counters: no division by the run-time stage count
  int s = 0;
  uint32_t phase = 0;
  for (int i = 0; i < it.n_tiles - skip_tiles; ++i) {
    if (!mbar_wait(smem_u32(&tail->k_empty[s]), phase ^ 1u, abort_flag, p.status, kDevWaitKEmpty))
      break;
    const uint32_t kf = smem_u32(&tail->k_full[s]);
    mbar_arrive_expect_tx(kf, kStageBytes);
    const int row = (down ? it.tile_down(i) : it.tile_begin + i) * kTileKeys;
    tma_load_2d(k_s + s * kStageBytes, tmapK, it.g * 128, row, kf);
    tma_load_2d(k_s + s * kStageBytes + 16384, tmapK, it.g * 128 + 64, row, kf);
    if (++s == stages) { s = 0; phase ^= 1u; }
  }
}

// Sum over 32 logits of 2^(v * c2 + nm).  Of every 16 pairs, NPOLY take the polynomial on the
// FMA pipe and the rest the special-function unit, so that both pipes work in parallel.
template <int NPOLY>
__device__ __forceinline__ float chunk_sum_exp2(const float (&v)[32], float c2, float nm) {
  const float2 c2v = make_float2(c2, c2), nmv = make_float2(nm, nm);
  float2 acc0 = make_float2(0.f, 0.f), acc1 = make_float2(0.f, 0.f);
#pragma unroll
  for (int pr = 0; pr < 16; ++pr) {
    const float2 x = ffma2(make_float2(v[2 * pr], v[2 * pr + 1]), c2v, nmv);
    float2 e;
    if (((pr + 1) * NPOLY) / 16 > (pr * NPOLY) / 16) {
      e = exp2_poly2(x);
    } else {
      e.x = ex2_approx(x.x);
      e.y = ex2_approx(x.y);
    }
    if (pr & 1) acc1 = fadd2(acc1, e); else acc0 = fadd2(acc0, e);
  }
  return (acc0.x + acc0.y) + (acc1.x + acc1.y);
}

// Online (max, sum-exp) update of one query row with 32 more logits of the key tile.  Keys
// past L (ragged last tile) become -inf: the special-function path maps them to 0 and the
// polynomial's clamp to 2^-125, which vanishes against the row's sum (>= 1).
template <int NPOLY>
__device__ __forceinline__ void row_chunk_update(float (&v)[32], int col0, int valid, float c2,
                                                 float& m, float& z) {
  if (valid < kTileKeys) {
#pragma unroll
    for (int j = 0; j < 32; ++j)
      if (col0 + j >= valid) v[j] = -INFINITY;
  }
  float cm0 = fmax3(v[0], v[1], v[2]), cm1 = fmax3(v[3], v[4], v[5]);
#pragma unroll
  for (int j = 6; j < 30; j += 4) {
    cm0 = fmax3(cm0, v[j], v[j + 1]);
    cm1 = fmax3(cm1, v[j + 2], v[j + 3]);
  }
  const float m_new = fmaxf(fmax3(m, cm0, cm1), fmaxf(v[30], v[31]));
  const float nm = -m_new * c2;
  const float sum = chunk_sum_exp2<NPOLY>(v, c2, nm);
  if (m_new > m) {                         // rare once the first tiles have been seen
    z *= ex2_approx((m - m_new) * c2);
    m = m_new;
  }
  z += sum;
}

// The same with 64 logits of a tile that lies inside the context: one maximum and one comparison
// per 64 logits, and the two halves' independent chains interleave.
template <int NPOLY>
__device__ __forceinline__ void row_update64(const float (&va)[32], const float (&vb)[32], float c2, float& m,
                                             float& z) {
  float ca0 = fmax3(va[0], va[1], va[2]), ca1 = fmax3(va[3], va[4], va[5]);
  float cb0 = fmax3(vb[0], vb[1], vb[2]), cb1 = fmax3(vb[3], vb[4], vb[5]);
#pragma unroll
  for (int j = 6; j < 30; j += 4) {
    ca0 = fmax3(ca0, va[j], va[j + 1]);
    cb0 = fmax3(cb0, vb[j], vb[j + 1]);
    ca1 = fmax3(ca1, va[j + 2], va[j + 3]);
    cb1 = fmax3(cb1, vb[j + 2], vb[j + 3]);
  }
  ca0 = fmax3(ca0, va[30], va[31]);
  cb0 = fmax3(cb0, vb[30], vb[31]);
  const float m_new = fmax3(fmax3(m, ca0, ca1), cb0, cb1);
  const float nm = -m_new * c2;
  float sum = chunk_sum_exp2<NPOLY>(va, c2, nm);
  sum += chunk_sum_exp2<NPOLY>(vb, c2, nm);
  if (m_new > m) {                         // rare once the first tiles have been seen
    z *= ex2_approx((m - m_new) * c2);
    m = m_new;
  }
  z += sum;
}

// ---------------------------------------------------------------------------------------
// Pass A: row statistics.  MT = number of 128-row tiles of the resident Q block.
// ---------------------------------------------------------------------------------------
// Row tile of accumulator j of key tile i.  A warpgroup always meets the same accumulator of four; where the last
// row tile is short it would have less to do than the others (TAIL), so the tiles take turns.
template <int MT, bool TAIL>
__device__ __forceinline__ int row_tile(int i, int j) {
  static_assert(!TAIL || MT > 1, "a short row tile is copied behind a full one only");
  if constexpr (!TAIL || MT == 3) return j;
  if constexpr (MT == 2) return j ^ ((i >> 1) & 1);
  return (i + j) & 3;
}

template <int MT, int NPOLY, bool TAIL>
__global__ void __launch_bounds__(kStatsThreads<MT>, 1)
row_stats_kernel(const __grid_constant__ CUtensorMap tmapK,
                 const __grid_constant__ CUtensorMap tmapQ, const __grid_constant__ CUtensorMap tmapQ32, const QkParams p,
             const PrepParams pp) {
  extern __shared__ __align__(1024) uint8_t smem[];
  const uint32_t smem_base = smem_u32(smem);
  const uint32_t q_s = smem_base;
  const uint32_t k_s = smem_base + MT * 128 * 256;
  SmemTail* tail = reinterpret_cast<SmemTail*>(smem + MT * 128 * 256 + p.stages * kStageBytes);
  volatile int* abort_flag = &tail->abort_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const CtaItem it = decode_item(p, blockIdx.x);

  const int live_rows = min(p.rb_rows, p.rows_per_kv - (it.group % p.n_rb) * p.rb_rows);
  // the last live row tile: its rows' copies, rows per copy
  const int tail_tile = (live_rows - 1) / 128, copies = TAIL ? stats_tail_copies(live_rows) : 1;
  const int copy_rows = 128 / copies;
  constexpr uint32_t kIssuers = kStatsIssuers<MT>;       // every one reads every key tile
  const uint32_t tmem_base = cta_setup(tail, smem_base, p.stages, 4, 4, p.status, kIssuers, &tmapK, &tmapQ);
  const bool run = (it.n_tiles > 0) && (*abort_flag == 0);
  const bool stamp = (p.clk != nullptr) && blockIdx.x == 0 && threadIdx.x == 0;
  if (stamp) {
    unsigned long long ns0;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(ns0));
    tail->stamp_cycles = clock64();
    tail->stamp_ns = ns0;
  }

  if (warp == 0) {
    if (lane == 0 && run) {
      // The packed query (or, as the first kernel of a run, whatever else this one reads) comes from
      // the kernel before this one, which may still be running.  After that the next kernel's CTAs
      // may come in as SMs fall free.
      grid_dep_wait();
      grid_dep_launch();
      producer_loop(&tmapK, &tmapQ, &tmapQ32, p, it, tail, q_s, k_s, false, p.stages, MT, copies > 1 ? tail_tile : -1,
                    copy_rows, p.skip_tiles);
    }
  } else if (warp == 1 || warp >= 2 + kStatsConsumerWarps) {
    if (lane == 0 && run) {
      // Accumulator u is filled by issuing thread u % kIssuers.  A barrier test waits behind the MMAs that
      // its thread has issued: one thread took 1030 cycles per accumulator for 512 cycles of MMAs, and
      // the consumers waited 1700 of 4160 cycles for each of theirs; with two threads 450 of 4010
      // (row statistics at 256K keys, 512 rows per kv head: 278 -> 272 us; 1M keys, 1024 rows: 2489 -> 2424 us).
      const uint32_t mine = (warp == 1) ? 0u : 1u;
      constexpr uint32_t idesc = umma_idesc_bf16(128, kTileKeys);
      bool ok = mbar_wait(smem_u32(&tail->q_full), 0, abort_flag, p.status, kDevWaitQFull, p.wait_limit);
      tc_fence_after();
      uint32_t u = 0;
      int s = 0;
      uint32_t kphase = 0;
      for (int i = 0; i < it.n_tiles && ok; ++i) {
        ok = mbar_wait(smem_u32(&tail->k_full[s]), kphase, abort_flag, p.status, kDevWaitKFull, p.wait_limit);
        if (!ok) break;
        tc_fence_after();
        for (int j = 0; j < MT; ++j, ++u) {
          if (u % kIssuers != mine) continue;
          const int mt = row_tile<MT, TAIL>(i, j);
          const uint32_t b = u & 3u, use = u >> 2;
          ok = mbar_wait(smem_u32(&tail->acc_empty[b]), (use & 1u) ^ 1u, abort_flag, p.status,
                         kDevWaitAccEmpty, p.wait_limit);
          if (!ok) break;
          tc_fence_after();
#pragma unroll
          for (int kb = 0; kb < 2; ++kb)
#pragma unroll
            for (int ks = 0; ks < 4; ++ks) {
              const uint64_t a = umma_desc_sw128(q_s + kb * (MT * 128 * 128) + mt * 16384 + ks * 32);
              const uint64_t bd = umma_desc_sw128(k_s + s * kStageBytes + kb * 16384 + ks * 32);
              umma_bf16(tmem_base + b * 128, a, bd, idesc, (kb | ks) != 0);
            }
          umma_commit(smem_u32(&tail->acc_full[b]));
        }
        umma_commit(smem_u32(&tail->k_empty[s]));
        if (++s == p.stages) { s = 0; kphase ^= 1u; }
      }
    }
  } else {
    // Consumer warpgroups take the accumulator buffers in turn, so that they sit in different
    // phases (waiting, loading, taking maxima, exponentials) and keep the special-function
    // and FMA pipes fed.  Each thread owns one query row of the buffer and takes its 128 columns
    // in two halves of 64 (32 at a time with the next 32 loading meanwhile: 2508 against 2410 us
    // at L = 1M, q_len 256 -- more registers' worth of independent work beats the prefetch).
    const int wg = (warp - 2) >> 2;
    const int quad = warp & 3;               // TMEM lane quadrant this warp may read
    if (pp.clear) {                          // while the first tiles are on their way
      grid_dep_wait();                       // the run before this one may still read that state
      clear_state(pp, static_cast<long long>(blockIdx.x) * (kStatsConsumerWarps * 32) + threadIdx.x - 64,
                  static_cast<long long>(gridDim.x) * (kStatsConsumerWarps * 32));
    }
    // Accumulator u belongs to warpgroup u % 4 and holds row tile u % MT.  With 1, 2 or 4 row
    // tiles a warpgroup therefore always meets the same row tile (wg % MT) and a thread keeps
    // one (max, sum) pair; only with 3 row tiles, or tiles that take turns, does it meet all of them.
    constexpr int kStates = (MT == 3 || TAIL) ? MT : 1;
    float m[kStates], z[kStates];
#pragma unroll
    for (int j = 0; j < kStates; ++j) { m[j] = -1e30f; z[j] = 0.f; }
    const float c2 = p.c2;
    const int tail_col = quad * 32 / copy_rows * copy_rows;      // this warp's columns of a copied row tile
    const uint32_t n_acc = run ? static_cast<uint32_t>(it.n_tiles) * MT : 0u;
    // One copy of the loop body serves every (key tile, row tile): the warpgroups run at
    // different places of the loop, and a body unrolled over the row tiles would not fit the
    // instruction cache between them.
#pragma unroll 1
    for (uint32_t u = wg; u < n_acc; u += kStatsWarpgroups) {
      const int i = static_cast<int>(u / MT), mt = row_tile<MT, TAIL>(i, static_cast<int>(u % MT));
      const long long key0 = static_cast<long long>(it.tile_begin + i) * kTileKeys;
      const int valid = static_cast<int>(min(static_cast<long long>(kTileKeys), p.L - key0));
      const uint32_t b = u & 3u, use = u >> 2;
      if (!mbar_wait(smem_u32(&tail->acc_full[b]), use & 1u, abort_flag, p.status,
                     kDevWaitAccFull, p.wait_limit))
        break;
      tc_fence_after();
      const bool shared = TAIL && mt == tail_tile;
      if (mt * 128 + (shared ? quad * 32 % copy_rows : quad * 32) >= live_rows) {    // padding rows only: nothing to compute
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&tail->acc_empty[b]));
        continue;
      }
      float mr = m[0], zr = z[0];
      if (kStates > 1) {
#pragma unroll
        for (int j = 1; j < kStates; ++j)
          if (j == mt) { mr = m[j]; zr = z[j]; }
      }
      const uint32_t taddr = tmem_base + (static_cast<uint32_t>(quad * 32) << 16) + b * 128;
      const int col0 = shared ? tail_col : 0, col1 = shared ? col0 + copy_rows : kTileKeys;
      if (valid >= kTileKeys && (!TAIL || col1 - col0 >= 64)) {
#pragma unroll 1
        for (int c = col0; c < col1; c += 64) {
          float va[32], vb[32];
          tmem_ld32(taddr + c, va);
          tmem_ld32(taddr + c + 32, vb);
          tmem_ld_wait();
          if (c + 64 == col1) {                      // read completely: back to the MMA thread
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&tail->acc_empty[b]));
          }
          row_update64<NPOLY>(va, vb, c2, mr, zr);
        }
      } else {                               // the context ends inside this tile, or four copies
#pragma unroll 1
        for (int c = col0; c < col1; c += 32) {
          float v[32];
          tmem_ld32(taddr + c, v);
          tmem_ld_wait();
          row_chunk_update<NPOLY>(v, c, valid, c2, mr, zr);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&tail->acc_empty[b]));
      }
      if (kStates > 1) {
#pragma unroll
        for (int j = 0; j < kStates; ++j)
          if (j == mt) { m[j] = mr; z[j] = zr; }
      } else {
        m[0] = mr; z[0] = zr;
      }
    }
    // Merge the warpgroups' statistics through shared memory and write this CTA's partial
    // statistics: (max in log2 units, sum).  Every warpgroup stores a pair for every row tile
    // (a neutral one for the row tiles it never met); warpgroup 0 merges.  The scratch aliases
    // the first K stage, which is idle once every warpgroup has read its last accumulator
    // (every MMA, hence every TMA load, has completed by then).
    float2* scratch = reinterpret_cast<float2*>(smem + MT * 128 * 256);
    const int row_in_tile = quad * 32 + lane;
    asm volatile("bar.sync 1, %0;" ::"r"(kStatsConsumerWarps * 32) : "memory");
#pragma unroll
    for (int mt = 0; mt < MT; ++mt) {
      float2 mine = make_float2(-1e30f, 0.f);
      if (kStates > 1) {
#pragma unroll
        for (int j = 0; j < kStates; ++j)
          if (j == mt) mine = make_float2(m[j], z[j]);
      } else if (mt == wg % MT) {
        mine = make_float2(m[0], z[0]);
      }
      scratch[(wg * MT + mt) * 128 + row_in_tile] = mine;
    }
    asm volatile("bar.sync 1, %0;" ::"r"(kStatsConsumerWarps * 32) : "memory");
    if (wg == 0) {
      float2* out = reinterpret_cast<float2*>(p.partial) +
                    (static_cast<size_t>(it.group) * p.cpg + it.chunk) * p.rb_rows;
#pragma unroll
      for (int mt = 0; mt < MT; ++mt) {
        if (mt * 128 + row_in_tile >= live_rows) break;
        const int n_copy = (TAIL && mt == tail_tile) ? copies : 1;
        float mm = -1e30f;
        for (int x = 0; x < n_copy; ++x)
#pragma unroll
          for (int w = 0; w < kStatsWarpgroups; ++w)
            mm = fmaxf(mm, scratch[(w * MT + mt) * 128 + x * copy_rows + row_in_tile].x);
        float zz = 0.f;
        for (int x = 0; x < n_copy; ++x)
#pragma unroll
          for (int w = 0; w < kStatsWarpgroups; ++w) {
            const float2 o = scratch[(w * MT + mt) * 128 + x * copy_rows + row_in_tile];
            zz += o.y * exp2f((o.x - mm) * c2);
          }
        out[mt * 128 + row_in_tile] = make_float2(mm * c2, zz);
      }
    }
  }
  if (stamp) {
    unsigned long long ns1;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(ns1));
    p.clk[0] = static_cast<unsigned long long>(clock64() - tail->stamp_cycles);
    p.clk[1] = ns1 - tail->stamp_ns;
  }
  cta_teardown(tmem_base);
}

// Combines the partial statistics of one row (per key chunk of the statistics pass, or per key
// shard) into (max in log2 units, sum); -lse in log2 units for the scores pass (-inf marks a
// padding row); `publish` also stores the user-visible natural-log lse.  rg: row of kv head g.
__device__ __forceinline__ float2 merged_stats(const MergeParams& p, int g, int rg, int* user_row) {
  *user_row = -1;
  if (rg >= p.group_size * p.q_len) return make_float2(-INFINITY, 0.f);
  const int i = rg / p.group_size, j = rg % p.group_size;
  *user_row = i * p.n_q + g * p.group_size + j;
  const float2* part;
  size_t stride;
  int n;
  if (p.n_ext > 0) {                     // one entry per key shard
    part = p.ext_stats + *user_row;
    stride = static_cast<size_t>(p.q_len) * p.n_q;
    n = p.n_ext;
  } else {                               // one entry per key chunk of the statistics pass
    const int group = g * p.n_rb + rg / p.rb_rows;
    part = reinterpret_cast<const float2*>(p.partial) +
           static_cast<size_t>(group) * p.cpg * p.rb_rows + rg % p.rb_rows;
    stride = p.rb_rows;
    n = p.cpg;
  }
  // kHold entries at a time, since each read is a trip to the L2, and no more, since the code is met cold (18
  // entries between the end of the statistics pass and the first step of the scores: one after another and
  // twice 2.7 us, 20 at a time 2.2, so 1.7; L = 1M 4.8, 3.2).
  constexpr int kHold = 10;
  float mm = -INFINITY, zz = 0.f;
#pragma unroll 1
  for (int c0 = 0; c0 < n; c0 += kHold) {
    float2 v[kHold];
    float top = mm;
#pragma unroll
    for (int c = 0; c < kHold; ++c) v[c] = (c0 + c < n) ? __ldcg(&part[(c0 + c) * stride]) : make_float2(-INFINITY, 0.f);
#pragma unroll
    for (int c = 0; c < kHold; ++c) top = fmaxf(top, v[c].x);
    if (top == -INFINITY) continue;                          // empty shards so far
    zz *= exp2f(mm - top);
    mm = top;
#pragma unroll
    for (int c = 0; c < kHold; ++c) zz += v[c].y * exp2f(v[c].x - mm);
  }
  return make_float2(mm, zz);
}

__device__ __forceinline__ float merged_neg_lse2(const MergeParams& p, int g, int rg, bool publish) {
  int user_row;
  const float2 st = merged_stats(p, g, rg, &user_row);
  if (user_row < 0) return -INFINITY;
  const float lse2 = st.x + log2f(st.y);
  if (publish) p.row_lse[user_row] = lse2 * 0.69314718055994530942f;
  return -lse2;
}

__global__ void export_stats_kernel(MergeParams p, float2* __restrict__ out) {
  const int rows = p.group_size * p.q_len;
  const int row = blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= p.n_kv * rows) return;
  int user_row;
  const float2 st = merged_stats(p, row / rows, row % rows, &user_row);
  if (user_row >= 0) out[user_row] = st;
}

__global__ void decode_scores_kernel(const uint32_t* __restrict__ enc, float* __restrict__ out,
                                     long long L) {
  const long long t = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t < L) out[t] = exp2f(ordered_to_float(enc[t]));
}

// ---------------------------------------------------------------------------------------
// Pass B: scores.  D[key, row]; per context position max over rows of log2-probability.
// ---------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kQkThreads, 1)
scores_kernel(const __grid_constant__ CUtensorMap tmapK,
              const __grid_constant__ CUtensorMap tmapQ, const QkParams p, const MergeParams mp) {
  extern __shared__ __align__(1024) uint8_t smem[];
  const uint32_t smem_base = smem_u32(smem);
  const uint32_t q_s = smem_base;
  const uint32_t k_s = smem_base + p.rb_rows * 256;
  SmemTail* tail = reinterpret_cast<SmemTail*>(smem + p.rb_rows * 256 + p.stages * kStageBytes);
  float* nl = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(tail) + kSmemTailBytes);
  volatile int* abort_flag = &tail->abort_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const CtaItem it = decode_item(p, blockIdx.x);
  // query rows of the block, rounded up to the consumers' step of 32: the tensor time goes with them
  const int n_rows = scores_block_rows(p.rb_rows, p.rows_per_kv, it.group % p.n_rb);
  const int n_nh = scores_row_halves(n_rows);
  const int stages = scores_ring_stages(p.stages, n_nh);

  // Two MMA-issuing threads (warps 1 and 2), one per accumulator buffer: tcgen05.mma holds its
  // issuing thread until the tensor pipe takes the instruction, so the waits and commits of
  // one thread overlap the MMAs of the other.  With two row halves per key tile each thread
  // issues one half of every tile and both release the tile's stage; with one, the threads
  // take the tiles in turn.
  const int k_releasers = (n_nh >= 2) ? 2 : 1;
  const uint32_t tmem_base = cta_setup(tail, smem_base, stages, 2, kConsumerWarps, p.status, k_releasers, &tmapK, &tmapQ);
  const bool run = (it.n_tiles > 0) && (*abort_flag == 0);

  if (warp == 0) {
    if (lane == 0 && run) {
      // keys and query are the caller's; a packed query comes from a kernel that the kernel before this
      // one waited for, unless that was the prepare kernel itself
      if (p.group == 0 && mp.n_ext > 0) grid_dep_wait();
      grid_dep_launch();                 // the next kernel's CTAs may come in as SMs fall free
      producer_loop(&tmapK, &tmapQ, nullptr, p, it, tail, q_s, k_s, true, stages, p.rb_rows / 128);
    }
  } else if (warp == 1 || warp == 2) {
    if (lane == 0 && run) {
      const uint32_t mine = static_cast<uint32_t>(warp - 1);          // accumulator buffer
      bool ok = mbar_wait(smem_u32(&tail->q_full), 0, abort_flag, p.status, kDevWaitQFull);
      tc_fence_after();
      uint32_t u = 0;
      int s = -1;
      uint32_t kphase = 1;
      for (int i = 0; i < it.n_tiles && ok; ++i) {
        if (++s == stages) s = 0;                        // stage and phase of key tile i
        if (s == 0) kphase ^= 1u;
        if (n_nh == 1 && ((static_cast<uint32_t>(i) & 1u) != mine)) { ++u; continue; }
        ok = mbar_wait(smem_u32(&tail->k_full[s]), kphase, abort_flag, p.status, kDevWaitKFull);
        if (!ok) break;
        tc_fence_after();
        for (int nh = 0; nh < n_nh; ++nh, ++u) {
          if ((u & 1u) != mine) continue;
          const int N = min(256, n_rows - nh * 256);
          const uint32_t idesc = umma_idesc_bf16(128, N);
          const uint32_t b = u & 1u, use = u >> 1;
          ok = mbar_wait(smem_u32(&tail->acc_empty[b]), (use & 1u) ^ 1u, abort_flag, p.status,
                         kDevWaitAccEmpty);
          if (!ok) break;
          tc_fence_after();
#pragma unroll
          for (int kb = 0; kb < 2; ++kb)
#pragma unroll
            for (int ks = 0; ks < 4; ++ks) {
              const uint64_t a = umma_desc_sw128(k_s + s * kStageBytes + kb * 16384 + ks * 32);
              const uint64_t bd =
                  umma_desc_sw128(q_s + kb * (p.rb_rows * 128) + nh * (256 * 128) + ks * 32);
              umma_bf16(tmem_base + b * 256, a, bd, idesc, (kb | ks) != 0);
            }
          umma_commit(smem_u32(&tail->acc_full[b]));
        }
        umma_commit(smem_u32(&tail->k_empty[s]));
      }
    }
  } else if (warp >= 4) {
    // The consumer warps merge the per-key-chunk statistics of the CTA's rows (a few KB from
    // L2; the CTAs of the first key chunk also publish the natural-log lse).  The statistics
    // come from the kernel before this one, which may still be running when this CTA starts
    // (the set-up above does not wait for it).
    grid_dep_wait();
    for (int i = threadIdx.x - 128; i < p.rb_rows; i += kConsumerWarps * 32)
      nl[i] = merged_neg_lse2(mp, it.g, (it.group % p.n_rb) * p.rb_rows + i, it.chunk == 0);
    asm volatile("bar.sync 2, %0;" ::"r"(kConsumerWarps * 32) : "memory");
    const int wg = (warp - 4) >> 2;
    const int quad = warp & 3;
    const float c2 = p.c2;
    bool ok = run;
    uint32_t u = 0;
    for (int i = 0; i < it.n_tiles && ok; ++i) {
      float best = -INFINITY;
      for (int nh = 0; nh < n_nh && ok; ++nh) {
        const int N = min(256, n_rows - nh * 256);
        const uint32_t b = u & 1u, use = u >> 1;
        ++u;
        ok = mbar_wait(smem_u32(&tail->acc_full[b]), use & 1u, abort_flag, p.status,
                       kDevWaitAccFull);
        if (!ok) break;
        tc_fence_after();
        // the warpgroups take the 32-column steps in turn, first one and then the other begins
        const uint32_t taddr = tmem_base + (static_cast<uint32_t>(quad * 32) << 16) + b * 256;
        const float4* nl4 = reinterpret_cast<const float4*>(nl + nh * 256);
        float b0 = -INFINITY, b1 = -INFINITY, b2 = -INFINITY, b3 = -INFINITY;
        for (int c = ((wg ^ i) & 1) * 32; c < N; c += 64) {
          float v[32];
          tmem_ld32(taddr + c, v);
          tmem_ld_wait();
#pragma unroll
          for (int j = 0; j < 32; j += 4) {
            const float4 n4 = nl4[(c + j) >> 2];
            b0 = fmaxf(b0, fmaf(v[j], c2, n4.x));
            b1 = fmaxf(b1, fmaf(v[j + 1], c2, n4.y));
            b2 = fmaxf(b2, fmaf(v[j + 2], c2, n4.z));
            b3 = fmaxf(b3, fmaf(v[j + 3], c2, n4.w));
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&tail->acc_empty[b]));
        best = fmaxf(best, fmaxf(fmaxf(b0, b1), fmaxf(b2, b3)));
      }
      const long long t = static_cast<long long>(it.tile_down(i)) * kTileKeys + quad * 32 + lane;
      if (ok && t < p.L) atomicMax(p.enc + t, float_to_ordered(best));
    }
  }
  cta_teardown(tmem_base);
}

// ---------------------------------------------------------------------------------------
// Pass B by CTA pairs, for long query parts
// ---------------------------------------------------------------------------------------
// Two CTAs of a cluster share tensor-core tiles of M = 256 keys by N = 256 query rows (tcgen05
// cta_group::2): each keeps half of the query rows resident and loads half of the keys of every
// 256-key tile.  Per instruction an SM reads 8 KB of operands for 128 cycles of math where the
// one-CTA form reads 12 KB, a key tile crosses from L2 to the SMs once per pair instead of once
// per CTA, and twice the query rows stay resident, so that half as many CTAs read each key tile.
// Bound by the tensor pipe and the board's power: L = 1M, 1024 rows per kv head, single calls on a cool
// board 1414 us = 1.56 PFLOP/s (one-CTA kernel 1568 us = 1.40), at the power cap of a long run 1470 to
// 1540 us = 1.43 to 1.49.
struct PairTail {
  uint64_t q_full;                   // q_full, k_full and acc_empty: used in the first CTA only
  uint64_t k_full[kMaxUnits];
  uint64_t k_empty[kMaxUnits];       // both CTAs
  uint64_t acc_full[2];              // both CTAs
  uint64_t acc_empty[2];
  uint32_t tmem_base;
  int abort_flag;
};
static_assert(sizeof(PairTail) <= kSmemTailBytes, "tail too large");

// TMA producer of one CTA: its 128 keys of every key tile in units of 64 channels, and its half of
// the query rows once.  Both CTAs' bytes are counted on the first CTA's barriers, whose producer
// announces the sum.  The keys are the caller's and final since before this launch, so a ring's
// worth of them is on its way before the wait for the kernel that packs the query.
template <int MT>
__device__ __forceinline__ void pair_producer_loop(const CUtensorMap* tmapK, const CUtensorMap* tmapQ,
                                                   const QkParams& p, const CtaItem& it, bool wait_for_query,
                                                   PairTail* tail, uint32_t rank, uint32_t q_s, uint32_t k_s) {
  volatile int* abort_flag = &tail->abort_flag;
  const int units = p.stages, n_units = 2 * it.n_tiles;
  int s = 0;
  uint32_t phase = 0;
  auto load_unit = [&](int n) -> bool {
    if (!mbar_wait(smem_u32(&tail->k_empty[s]), phase ^ 1u, abort_flag, p.status, kDevWaitKEmpty))
      return false;
    const uint32_t kf = smem_u32(&tail->k_full[s]);
    if (rank == 0) mbar_arrive_expect_tx(kf, 2 * kUnitBytes);
    const int row = it.tile_down(n >> 1) * kPairTileKeys + static_cast<int>(rank) * kTileKeys;
    tma_load_2d_pair(k_s + s * kUnitBytes, tmapK, it.g * 128 + (n & 1) * 64, row, cluster_addr(kf, 0));
    if (++s == units) { s = 0; phase ^= 1u; }
    return true;
  };
  const int ahead = min(units, n_units);
  int n = 0;
  bool ok = true;
  for (; n < ahead && ok; ++n) ok = load_unit(n);
  if (wait_for_query) grid_dep_wait();
  grid_dep_launch();                       // the next kernel's CTAs may come in as SMs fall free
  if (!ok) return;
  const uint32_t qf = smem_u32(&tail->q_full);
  if (rank == 0) mbar_arrive_expect_tx(qf, 2u * MT * 128 * 256);
  for (int kb = 0; kb < 2; ++kb)
    for (int mt = 0; mt < MT; ++mt)
    {
      const int row = (it.group % p.n_rb) * p.rb_rows + (static_cast<int>(rank) * MT + mt) * 128;
      const uint32_t dst = q_s + kb * (MT * 16384) + mt * 16384;
      if (p.group > 0) tma_load_3d_pair(dst, tmapQ, kb * 64, it.g * p.group, row / p.group, cluster_addr(qf, 0));
      else tma_load_2d_pair(dst, tmapQ, kb * 64, it.g * p.kv_rows + row, cluster_addr(qf, 0));
    }
  for (; n < n_units && ok; ++n) ok = load_unit(n);
  // The releases of the last units, which no load waits for, arrive in both CTAs' barriers: this CTA must
  // not leave before they have.
  for (int j = 0; j < units && ok; ++j) {
    ok = mbar_wait(smem_u32(&tail->k_empty[s]), phase ^ 1u, abort_flag, p.status, kDevWaitKEmpty);
    if (++s == units) { s = 0; phase ^= 1u; }
  }
}

// One of the two MMA-issuing threads of a pair (first CTA, warps 1 and 2), one per accumulator:
// tcgen05.mma holds its issuing thread until the tensor pipe takes the instruction, so the waits
// and commits of one thread overlap the MMAs of the other.  With several row tiles per CTA each
// thread issues every other one and both release a key tile; with one row tile they take the key
// tiles in turn.
template <int MT>
__device__ __forceinline__ void pair_issue_loop(const QkParams& p, const CtaItem& it, PairTail* tail,
                                                uint32_t tmem_base, uint32_t q_s, uint32_t k_s,
                                                uint32_t mine) {
  volatile int* abort_flag = &tail->abort_flag;
  constexpr uint32_t idesc = umma_idesc_bf16(256, 256);
  bool ok = mbar_wait(smem_u32(&tail->q_full), 0, abort_flag, p.status, kDevWaitQFull);
  tc_fence_after();
  uint32_t u = 0;
  int s = 0;
  uint32_t kphase = 0;
#pragma unroll 1
  for (int i = 0; i < it.n_tiles && ok; ++i) {
    const int s0 = s;
    const uint32_t ph0 = kphase;
    if (++s == p.stages) { s = 0; kphase ^= 1u; }
    const int s1 = s;
    const uint32_t ph1 = kphase;
    if (++s == p.stages) { s = 0; kphase ^= 1u; }
    if (MT == 1 && ((static_cast<uint32_t>(i) & 1u) != mine)) { ++u; continue; }
    ok = mbar_wait(smem_u32(&tail->k_full[s0]), ph0, abort_flag, p.status, kDevWaitKFull) &&
         mbar_wait(smem_u32(&tail->k_full[s1]), ph1, abort_flag, p.status, kDevWaitKFull);
    if (!ok) break;
    const uint64_t kd[2] = {umma_desc_sw128(k_s + s0 * kUnitBytes), umma_desc_sw128(k_s + s1 * kUnitBytes)};
#pragma unroll 1
    for (int mt = 0; mt < MT; ++mt, ++u) {
      const uint32_t b = u & 1u, use = u >> 1;
      if (b != mine) continue;
      ok = mbar_wait(smem_u32(&tail->acc_empty[b]), (use & 1u) ^ 1u, abort_flag, p.status, kDevWaitAccEmpty);
      if (!ok) break;
      tc_fence_after();
      const uint64_t qd = umma_desc_sw128(q_s + mt * 16384);
#pragma unroll
      for (int kb = 0; kb < 2; ++kb)
#pragma unroll
        for (int ks = 0; ks < 4; ++ks)
          umma_bf16_pair(tmem_base + b * 256, kd[kb] + ((ks * 32) >> 4),
                         qd + ((kb * (MT * 16384) + ks * 32) >> 4), idesc, (kb | ks) != 0);
      umma_commit_pair(smem_u32(&tail->acc_full[b]));
    }
    umma_commit_pair(smem_u32(&tail->k_empty[s0]));
    umma_commit_pair(smem_u32(&tail->k_empty[s1]));
  }
}

// D is 256 keys (128 in each CTA) by 256 query rows (columns 0..127 from the first CTA's row tile
// nh, 128..255 from the second's); consumer warpgroup w of a CTA takes columns [64 w, 64 w + 64) of
// its 128 keys.  MT: row tiles of 128 in each CTA.
template <int MT>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kPairThreads, 1)
scores_pair_kernel(const __grid_constant__ CUtensorMap tmapK,
                   const __grid_constant__ CUtensorMap tmapQ, const QkParams p, const MergeParams mp) {
  extern __shared__ __align__(1024) uint8_t smem[];
  const uint32_t smem_base = smem_u32(smem);
  const uint32_t q_s = smem_base;
  const uint32_t k_s = smem_base + MT * 128 * 256;
  PairTail* tail = reinterpret_cast<PairTail*>(smem + MT * 128 * 256 + p.stages * kUnitBytes);
  float* nl = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(tail) + kSmemTailBytes);
  volatile int* abort_flag = &tail->abort_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const CtaItem it = decode_item(p, blockIdx.x >> 1);

  if (threadIdx.x == 32) {
    tma_prefetch_desc(&tmapK);
    tma_prefetch_desc(&tmapQ);
  }
  if (threadIdx.x == 0) {
    tail->abort_flag = 0;
    if (smem_base & 1023u) {                       // swizzled tiles need 1024-byte alignment
      tail->abort_flag = 1;
      atomicCAS(p.status, 0, kDevSmemAlign);
    }
    mbar_init(smem_u32(&tail->q_full), 1);
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(smem_u32(&tail->k_full[s]), 1);
      mbar_init(smem_u32(&tail->k_empty[s]), (MT >= 2) ? 2 : 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&tail->acc_full[b]), 1);
      mbar_init(smem_u32(&tail->acc_empty[b]), 2 * kPairConsumerWarps);
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
  const bool run = (it.n_tiles > 0) && (*abort_flag == 0);

  if (warp == 0) {
    // A packed query was made by the kernel before the statistics kernel, which had completed before
    // the statistics kernel let this one start.  A launch without the statistics kernel waits.
    if (lane == 0 && run)
      pair_producer_loop<MT>(&tmapK, &tmapQ, p, it, p.group == 0 && mp.n_ext > 0, tail, rank, q_s, k_s);
  } else if (warp == 1 || warp == 2) {
    if (lane == 0 && run && rank == 0)
      pair_issue_loop<MT>(p, it, tail, tmem_base, q_s, k_s, static_cast<uint32_t>(warp - 1));
  } else if (warp >= 4) {
    // merge the per-key-chunk statistics of the pair's rows (see the one-CTA kernel)
    grid_dep_wait();
    for (int i = threadIdx.x - 128; i < p.rb_rows; i += kPairConsumerWarps * 32)
      nl[i] = merged_neg_lse2(mp, it.g, (it.group % p.n_rb) * p.rb_rows + i, it.chunk == 0 && rank == 0);
    asm volatile("bar.sync 2, %0;" ::"r"(kPairConsumerWarps * 32) : "memory");
    const int wg = (warp - 4) >> 2;
    const int quad = warp & 3;
    const float c2 = p.c2;
    const uint32_t full_bar = smem_u32(&tail->acc_full[0]);
    const uint32_t empty_bar = cluster_addr(smem_u32(&tail->acc_empty[0]), 0);
    const uint32_t taddr = tmem_base + (static_cast<uint32_t>(quad * 32) << 16) + wg * 64;
    // columns 64 wg ..: rows of CTA wg / 2 of the pair
    const float4* nl4 = reinterpret_cast<const float4*>(nl + (wg >> 1) * (MT * 128) + (wg & 1) * 64);
    bool ok = run;
    uint32_t u = 0;
    for (int i = 0; i < it.n_tiles && ok; ++i) {
      float b0 = -INFINITY, b1 = -INFINITY, b2 = -INFINITY, b3 = -INFINITY;
#pragma unroll 1
      for (int nh = 0; nh < MT; ++nh, ++u) {
        const uint32_t b = u & 1u;
        ok = mbar_wait(full_bar + 8 * b, (u >> 1) & 1u, abort_flag, p.status, kDevWaitAccFull);
        if (!ok) break;
        tc_fence_after();
        float va[32], vb[32];
        tmem_ld32(taddr + b * 256, va);
        tmem_ld32(taddr + b * 256 + 32, vb);
        tmem_ld_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(empty_bar + 8 * b);     // the arithmetic runs under the next MMAs
#pragma unroll
        for (int j = 0; j < 32; j += 4) {
          const float4 n4 = nl4[nh * 32 + (j >> 2)];
          b0 = fmaxf(b0, fmaf(va[j], c2, n4.x));
          b1 = fmaxf(b1, fmaf(va[j + 1], c2, n4.y));
          b2 = fmaxf(b2, fmaf(va[j + 2], c2, n4.z));
          b3 = fmaxf(b3, fmaf(va[j + 3], c2, n4.w));
        }
#pragma unroll
        for (int j = 0; j < 32; j += 4) {
          const float4 n4 = nl4[nh * 32 + 8 + (j >> 2)];
          b0 = fmaxf(b0, fmaf(vb[j], c2, n4.x));
          b1 = fmaxf(b1, fmaf(vb[j + 1], c2, n4.y));
          b2 = fmaxf(b2, fmaf(vb[j + 2], c2, n4.z));
          b3 = fmaxf(b3, fmaf(vb[j + 3], c2, n4.w));
        }
      }
      const long long t = static_cast<long long>(it.tile_down(i)) * kPairTileKeys +
                          static_cast<int>(rank) * kTileKeys + quad * 32 + lane;
      if (ok && t < p.L) atomicMax(p.enc + t, float_to_ordered(fmaxf(fmaxf(b0, b1), fmaxf(b2, b3))));
    }
  }
  // Neither CTA may leave while the other can still signal its barriers or read its operands (every commit
  // has been waited for, by the consumers or by the loading thread).
  tc_fence_before();
  __syncwarp();
  cluster_sync_all();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, 512);
  }
}

// ---------------------------------------------------------------------------------------
// small kernels around the two passes
// ---------------------------------------------------------------------------------------

// Packs the query rows of every kv head contiguously, zero-padded to kv_rows (head groups whose rows a
// TMA box cannot collect from the caller's array),
// and clears the per-run state (encoded scores, empty bitmap, selection
// state).
__global__ void prepare_kernel(const uint4* q, uint4* qp, PrepParams p) {
  // The run before this one may still use the buffers, and whatever was before it may have written the
  // query: no read through the non-coherent path.
  grid_dep_wait();
  grid_dep_launch();                     // the next kernel sets itself up meanwhile
  const long long tid = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  const long long nthreads = static_cast<long long>(gridDim.x) * blockDim.x;
  // packed query: 16 x uint4 per 128-element row
  const long long n_pack = static_cast<long long>(p.n_kv) * p.kv_rows * 16;
  for (long long e = tid; e < n_pack; e += nthreads) {
    const int part = static_cast<int>(e & 15);
    const long long prow = e >> 4;
    const int g = static_cast<int>(prow / p.kv_rows), rg = static_cast<int>(prow % p.kv_rows);
    uint4 val = make_uint4(0, 0, 0, 0);
    if (rg < p.group_size * p.q_len) {
      const int i = rg / p.group_size, j = rg % p.group_size;
      val = __ldcg(q + (static_cast<long long>(i) * p.n_q + g * p.group_size + j) * 16 + part);
    }
    qp[e] = val;
  }
  if (p.clear) clear_state(p, tid, nthreads);
}

// ---------------------------------------------------------------------------------------
// host-side launchers
// ---------------------------------------------------------------------------------------
size_t row_stats_smem_bytes(int rb_rows, int stages) {
  return static_cast<size_t>(rb_rows) * 256 + static_cast<size_t>(stages) * kStageBytes +
         kSmemTailBytes;
}
size_t scores_smem_bytes(int rb_rows, int stages) {
  return row_stats_smem_bytes(rb_rows, stages) + static_cast<size_t>(rb_rows) * sizeof(float);
}

template <int MT>
static cudaError_t launch_row_stats_mt(const CUtensorMap& tk, const CUtensorMap& tq, const CUtensorMap& tq32,
                                       const QkParams& p, const PrepParams& pp, cudaStream_t st) {
  const size_t smem = row_stats_smem_bytes(MT * 128, p.stages);
  auto kernel = row_stats_kernel<MT, kRowStatsPolyPairs, false>;
  if constexpr (MT > 1)
    if (p.tail) kernel = row_stats_kernel<MT, kRowStatsPolyPairs, true>;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  return launch_after_previous(kernel, p.n_groups * p.cpg, kStatsThreads<MT>, smem, st, tk, tq, tq32, p, pp);
}

cudaError_t launch_row_stats(const CUtensorMap& tk, const CUtensorMap& tq, const CUtensorMap& tq32, const QkParams& p,
                             const PrepParams& pp, cudaStream_t st) {
  switch ((p.rb_rows + 127) / 128) {
    case 1: return launch_row_stats_mt<1>(tk, tq, tq32, p, pp, st);
    case 2: return launch_row_stats_mt<2>(tk, tq, tq32, p, pp, st);
    case 3: return launch_row_stats_mt<3>(tk, tq, tq32, p, pp, st);
    case 4: return launch_row_stats_mt<4>(tk, tq, tq32, p, pp, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_export_stats(const MergeParams& p, float2* out, cudaStream_t st) {
  const int n = p.n_kv * p.group_size * p.q_len;
  export_stats_kernel<<<(n + 127) / 128, 128, 0, st>>>(p, out);
  return cudaGetLastError();
}

cudaError_t launch_decode_scores(const uint32_t* enc, float* out, long long L, cudaStream_t st) {
  decode_scores_kernel<<<static_cast<unsigned>((L + 255) / 256), 256, 0, st>>>(enc, out, L);
  return cudaGetLastError();
}

template <int MT>
static cudaError_t launch_scores_pair_mt(const CUtensorMap& tk, const CUtensorMap& tq, QkParams p,
                                         const MergeParams& mp, cudaStream_t st) {
  constexpr int kFixed = MT * 128 * 256 + kSmemTailBytes + MT * 256 * static_cast<int>(sizeof(float));
  constexpr int kUnits = (kMaxDynSmem - kFixed) / kUnitBytes < kMaxUnits ? (kMaxDynSmem - kFixed) / kUnitBytes
                                                                         : kMaxUnits;
  // the issuing threads take the tiles of two units in turn with one row tile; see scores_ring_stages
  static_assert(MT > 1 || kUnits % 4 == 0, "a ring unit must always meet the same issuing thread");
  p.stages = kUnits;
  const size_t smem = static_cast<size_t>(kFixed) + static_cast<size_t>(p.stages) * kUnitBytes;
  cudaError_t e = cudaFuncSetAttribute(scores_pair_kernel<MT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  return launch_after_previous(scores_pair_kernel<MT>, 2 * p.n_groups * p.cpg, kPairThreads, smem, st, tk, tq, p, mp);
}

cudaError_t launch_scores(const CUtensorMap& tk, const CUtensorMap& tq, const QkParams& p,
                          const MergeParams& mp, cudaStream_t st) {
  if (p.pair) {
    switch (p.rb_rows / 256) {
      case 1: return launch_scores_pair_mt<1>(tk, tq, p, mp, st);
      case 2: return launch_scores_pair_mt<2>(tk, tq, p, mp, st);
      case 3: return launch_scores_pair_mt<3>(tk, tq, p, mp, st);
      case 4: return launch_scores_pair_mt<4>(tk, tq, p, mp, st);
      default: return cudaErrorInvalidValue;
    }
  }
  const size_t smem = scores_smem_bytes(p.rb_rows, p.stages);
  cudaError_t e = cudaFuncSetAttribute(scores_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  return launch_after_previous(scores_kernel, p.n_groups * p.cpg, kQkThreads, smem, st, tk, tq, p, mp);
}

cudaError_t launch_prepare(const void* q, void* qp, const PrepParams& p, int n_sm,
                           cudaStream_t st) {
  return launch_after_previous(prepare_kernel, n_sm * 4, 256, 0, st, static_cast<const uint4*>(q),
                               static_cast<uint4*>(qp), p);
}

}  // namespace ilre
