// Algorithm 1 ("Context Allocation") on the device, as ONE kernel, a thread-block cluster or a cooperative
// grid, whose CTAs meet at barriers between the phases:
//
//   A  MaxPooling(size = stride = m), once per distinct m > 1;
//   B  the stride-1 window pooling (average or max) of every (m, n) combination, up to kPoolGroup
//      windows of one m from one load of the cells, and a histogram of the pooled values in
//      kHistBins logarithmic bins;
//   (A and B take A^C[t] = exp2(max_r log2 p_rt) from the scores pass' encoded maxima, Eq. 5, as they
//   read them;)
//   C  every CTA finds, for each combination it scans, the bin that holds the K_m-th largest value
//      and how many values lie in the bins above each bin;
//   D  one scan gathers the candidates, the cells of that bin and of the bins above it, sorted by
//      bin: the place of a cell is the number of values in higher bins plus a counter of its own
//      bin.  The threshold bin brings a few cells more than K_m; only when it brings more than
//      kCandSlack of them (a plateau of equal values, mostly) does the combination take the long
//      way: a radix select of the K_m-th value in two more histogram passes over the array, then the
//      ties in cell order (the tiles are in cell order, so a count of the holders per tile plus an
//      ordered rank inside the tile settle which cells win);
//   E  ranking (value descending, cell ascending): a candidate is compared with the candidates of
//      its own bin only (a crowded bin's are dealt out first), spread over the grid;
//   F  one CTA walks the combinations in loop order: maps cells back to tokens, skips tokens
//      already allocated, stops each combination at its quota B_c, then writes the allocated
//      positions in ascending order.
//
// Work of phase B is cut into tiles of cells of one group of windows, work of phase D into tiles of
// kSelTile cells of one combination; every CTA owns a contiguous run of tiles.
//
// Bound by the chain of its phases: barriers, one CTA's walk, code met cold in the instruction cache
// (everything it reads is in L2).  Hence `unroll 1` on loops of few turns: the compiler's fourfold copies with
// their remainders are lines fetched for one turn (the kernel between its own time stamps, with the compiler's choice
// 128K positions 33.1 us, so 28.9; 1M 71, 64).  The stage by itself, events around it after an L2 flush, with a
// selection inside the threshold bin, one window per pooling tile and scattered candidates -> as it
// stands: 4K positions 39 -> 24 us, 32K 52 -> 31, 128K 59 -> 36, 512K 89 -> 55, 1M 117..131 -> 68, 1M with
// 48 combinations 270..280 -> 188.
#include <atomic>

#include "select_kernels.cuh"
#include "sm100_ptx.cuh"

namespace ilre {

__device__ __forceinline__ unsigned long long make_key(float w, uint32_t cell) {
  return (static_cast<unsigned long long>(float_to_ordered(w)) << 32) | (0xFFFFFFFFu - cell);
}

__device__ __forceinline__ void pass_bits(int pass, int& shift, int& bits) {
  const int sh[kSelectPasses] = {53, 42, 32};
  const int bt[kSelectPasses] = {11, 11, 10};
  shift = sh[pass];
  bits = bt[pass];
}

enum : uint8_t { kFirstDigitKnown = 1, kAllPasses = 2 };       // SelShared::mode

struct SelShared {
  alignas(8) uint32_t hist[kHistBins];     // (the ranking's scratch after the scans)
  uint32_t above[kHistBins + 1];           // of one combination: [b + 1] values in the bins above bin b; [0] all
  uint32_t scan[32];
  int flag;                                // of the grid barrier: written and read there only
  int list;                                // ranking: the combination that this CTA serves
  int threshold;                           // the bin of its K_m-th largest value
  int plateau;                             // it brings too many cells: full-scan passes
  uint32_t n_listed;                       // candidates of this CTA listed in shared memory
  unsigned long long prefix[kMaxCombos];   // full-scan passes, per combination: radix prefix found so far,
  uint32_t state[kMaxCombos];              // 1: the K_m-th value is settled, 2: the first pass is left out,
  uint32_t krem[kMaxCombos];               // and the keys still wanted inside the prefix
  uint8_t mode[kMaxCombos];                // 0, or how the combination takes the full-scan passes
  uint32_t tot[2][32];                     // warp totals of the one-barrier block scan
  // quota walk, per combination: (m, quota, ranked cells, kind of cells); an indexed read of the kernel's
  // parameters costs hundreds of cycles in the walk's dependent chain
  int4 walk[kMaxCombos];
};

// Grid-wide barrier (all CTAs are co-resident: cooperative launch).  The arrival counter is
// zero when the kernel starts and only grows: the k-th barrier completes when it reaches
// k * gridDim.x.  One thread per CTA arrives with a release at device scope (cumulative over the
// CTA's writes, which the block barrier before it orders) and polls with acquire loads; no
// value comes back from the arrival, so a barrier costs one trip to the L2 instead of two.
// The wait is bounded; a CTA that gives up records it and leaves the kernel.
// kCluster: the whole grid is one thread-block cluster (short contexts): the hardware cluster
// barrier takes the place of the counter, with release / acquire ordering at cluster scope.
template <bool kCluster>
__device__ __forceinline__ bool grid_sync(const SelectParams& p, SelShared* sh, uint32_t& epoch) {
  if constexpr (kCluster) {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    return true;
  }
  ++epoch;
  __syncthreads();
  if (threadIdx.x == 0) {
    int ok = 1;
    const uint32_t target = epoch * (gridDim.x + static_cast<uint32_t>(p.barrier_extra));
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p.barrier) : "memory");
    const long long t0 = clock64();
    for (uint32_t it = 1;; ++it) {
      uint32_t arrived;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(arrived) : "l"(p.barrier) : "memory");
      if (arrived >= target) break;
      if ((it & 0xFF) == 0 && clock64() - t0 > p.wait_limit) {
        atomicCAS(p.status, 0, kDevGridBarrier);
        ok = 0;
        break;
      }
    }
    sh->flag = ok;
  }
  __syncthreads();
  return sh->flag != 0;
}

// Exclusive prefix sum over the block of kSelThreads threads; *total receives the block sum.
// Begins with a barrier, and none follows the last reads of sh_warp: its next writer is the next call's, behind that
// barrier.  Not inlined: the kernel meets its code cold, and every phase after the first use finds this one warm.
__device__ __noinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t* sh_warp,
                                                         uint32_t* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if (lane >= o) incl += t;
  }
  __syncthreads();                       // protects sh_warp from the previous call's readers
  if (lane == 31) sh_warp[warp] = incl;
  __syncthreads();
  const uint32_t w = sh_warp[lane];      // every warp adds up the warps' totals itself
  *total = __reduce_add_sync(0xFFFFFFFFu, w);
  return __reduce_add_sync(0xFFFFFFFFu, lane < warp ? w : 0u) + incl - v;
}

// Adds one digit per thread (0xFFFFFFFF = none) to the shared histogram, one atomic per
// distinct digit of the warp: plateaus of equal pooled values are the common case.
__device__ __forceinline__ void hist_add(uint32_t* hist, uint32_t digit) {
  if (!__any_sync(0xFFFFFFFFu, digit != 0xFFFFFFFFu)) return;
  const uint32_t peers = __match_any_sync(0xFFFFFFFFu, digit);
  if (digit != 0xFFFFFFFFu && (threadIdx.x & 31) == __ffs(peers) - 1)
    atomicAdd(&hist[digit], __popc(peers));
}

// Adds the shared histogram to the global one and clears it.
__device__ __forceinline__ void hist_drain(uint32_t* sh_hist, uint32_t* gh) {
  for (int b = threadIdx.x; b < kHistBins; b += kSelThreads) {
    const uint32_t v = sh_hist[b];
    if (v) { atomicAdd(&gh[b], v); sh_hist[b] = 0u; }
  }
}
__device__ __forceinline__ void hist_flush(uint32_t* sh_hist, uint32_t* gh) {
  __syncthreads();
  hist_drain(sh_hist, gh);
  __syncthreads();
}

// Combination that owns `tile`.  Tiles are visited in increasing order, so the search resumes
// from the previous answer (`cur`, 0 at first).
__device__ __forceinline__ int combo_of_tile(const ComboTable& tbl, int tile, int& cur) {
#pragma unroll 1
  while (cur + 1 < tbl.n_comb && tile >= tbl.tile_begin[cur + 1]) ++cur;
  return cur;
}

static constexpr int kTilePer = kSelTile / kSelThreads;
static constexpr int kMaxWalkWarps = kSelThreads / 32;
static constexpr int kScanGroup = 4;      // tiles whose loads are issued together (long way)
static constexpr int kGatherGroup = 4;    // the same in the gather

// Pooled values of one tile, kTilePer per thread, all loads in flight together.
__device__ __forceinline__ void fetch_tile(const ComboTable& tbl, const SelectParams& p, int tile,
                                           int& cur, const uint32_t* skip, float (&wv)[kTilePer]) {
  const int combo = combo_of_tile(tbl, tile, cur);
  if (skip && skip[combo]) return;
  const float* w = p.pooled + static_cast<long long>(combo) * p.pooled_stride;
  const int c0 = (tile - tbl.tile_begin[combo]) * kSelTile, n = cells_from(tbl.len[combo], c0, kSelTile);
#pragma unroll
  for (int k = 0; k < kTilePer; ++k) {
    const int i = k * kSelThreads + threadIdx.x;
    wv[k] = (i < n) ? __ldcg(&w[c0 + i]) : 0.f;
  }
}

// Score of position t (Eq. 5).
__device__ __forceinline__ float score_at(const SelectParams& p, long long t) {
  return p.scores_given ? __ldcg(&p.scores[t]) : exp2f(ordered_to_float(__ldcg(&p.enc[t])));
}

// Phase A for one tile of source `src`: cells of MaxPooling(size = stride = m), a shorter
// last cell where m does not divide the length.  The tokens are read coalesced into `buf`
// (kSrcTileTokens words), all loads in flight together; of encoded scores the maximum is taken before
// they are decoded (their order is the scores'), one exponential per cell.
__device__ __forceinline__ void maxpool_tile(const ComboTable& tbl, const SelectParams& p, int src,
                                             int tile_in_src, uint32_t* buf) {
  const int m = tbl.src_m[src], len = tbl.src_len[src];
  const long long Lp = p.L - p.n_sink;
  const uint32_t* a = (p.scores_given ? reinterpret_cast<const uint32_t*>(p.scores) : p.enc) + p.n_sink;
  const int cells_per_tile = kSrcTileTokens / m;
  const int c0 = tile_in_src * cells_per_tile;
  const int n_cells = min(cells_per_tile, len - c0);
  const long long t0 = static_cast<long long>(c0) * m;
  const int n_tok = static_cast<int>(min(static_cast<long long>(n_cells) * m, Lp - t0));
  constexpr int kLd = kSrcTileTokens / kSelThreads;
  const uint32_t pad = p.scores_given ? __float_as_uint(-INFINITY) : 0u;        // below every score
  uint32_t v[kLd];
#pragma unroll
  for (int k = 0; k < kLd; ++k) {
    const int i = k * kSelThreads + threadIdx.x;
    v[k] = (i < n_tok) ? __ldcg(a + t0 + i) : pad;
  }
#pragma unroll
  for (int k = 0; k < kLd; ++k) buf[k * kSelThreads + threadIdx.x] = v[k];
  __syncthreads();
  float* out = p.maxpooled + static_cast<long long>(src) * p.maxpooled_stride;
  for (int c = threadIdx.x; c < n_cells; c += kSelThreads) {
    if (p.scores_given) {                  // as floats: a NaN does not win
      float acc = __uint_as_float(buf[c * m]);
      for (int j = 1; j < m; ++j) acc = fmaxf(acc, __uint_as_float(buf[c * m + j]));
      out[c0 + c] = acc;
    } else {
      uint32_t acc = buf[c * m];
      for (int j = 1; j < m; ++j) acc = max(acc, buf[c * m + j]);
      out[c0 + c] = exp2f(ordered_to_float(acc));
    }
  }
  __syncthreads();
}

// A pooled value as it is stored: no NaN, since the histogram, the gather and the ranking must agree on
// where every cell belongs (a cell counted and not found leaves a hole in the candidate list).  A NaN (of
// given scores, or of positions that a scores pass which gave up never reached) ranks below every score.
__device__ __forceinline__ float ranked_value(float v) { return (v == v) ? v : -0.f; }

// Counts the bin of one cell per lane (-1: none).  Neighbouring cells of a window maximum are often
// equal: the first lane of a run of equal bins adds the whole run.
__device__ __forceinline__ void count_bins(uint32_t* hist, int bin) {
  const int lane = threadIdx.x & 31;
  const int left = __shfl_up_sync(0xFFFFFFFFu, bin, 1);
  const bool leader = lane == 0 || left != bin;
  const uint32_t leaders = __ballot_sync(0xFFFFFFFFu, leader);
  if (leader && bin >= 0) {
    const uint32_t after = (lane == 31) ? 0u : leaders >> (lane + 1);
    atomicAdd(&hist[bin], after ? static_cast<uint32_t>(__ffs(after)) : static_cast<uint32_t>(32 - lane));
  }
}

// Phase B for one tile: cells [c0, c0 + n_out) of every combination of group `grp` from their common
// source (the scores themselves for m = 1), written to p.pooled; the bins of the cells are counted in
// the group's histograms.  `buf0` / `buf1` hold the tile and the widest window's margin; hists[k] belongs
// to the group's k-th combination (ascending window sizes).
__device__ __forceinline__ void pool_tile(const ComboTable& tbl, const SelectParams& p, int grp, int c0, int n_out,
                                          float* buf0, float* buf1, uint32_t* hist0, uint32_t* hist1) {
  const int first = tbl.grp_first[grp], n_win = tbl.grp_first[grp + 1] - first;
  const int some = tbl.grp_combo[first];
  const int n_max = tbl.n[tbl.grp_combo[first + n_win - 1]], len = tbl.len[some];
  const int source = tbl.src[some];
  // the cells: pooled ones, given scores, or encoded ones, which are decoded here
  const bool encoded = source < 0 && !p.scores_given;
  const uint32_t* a = source >= 0 ? reinterpret_cast<const uint32_t*>(p.maxpooled + static_cast<long long>(source) * p.maxpooled_stride)
                                  : (encoded ? p.enc : reinterpret_cast<const uint32_t*>(p.scores)) + p.n_sink;
  const int lo = c0 - n_max / 2;
  const int span = n_out + n_max - 1;
  const float pad = (p.win_op == 0) ? 0.f : -INFINITY;
  const int in_begin = -lo, in_end = cells_from(len, c0, span) + n_max / 2;      // of the tile and its margins, what lies inside
#pragma unroll 1
  for (int base = 0; base < span; base += 4 * kSelThreads) {
    uint32_t raw[4];                                       // all loads in flight together
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int idx = base + k * kSelThreads + threadIdx.x;
      raw[k] = (idx >= in_begin && idx < min(span, in_end)) ? __ldcg(a + lo + idx) : 0u;
    }
#pragma unroll 1
    for (int k = 0; k < 4; ++k) {
      const int idx = base + k * kSelThreads + threadIdx.x;
      if (idx >= span) break;
      buf0[idx] = (idx < in_begin || idx >= in_end) ? pad : encoded ? exp2f(ordered_to_float(raw[0])) : __uint_as_float(raw[0]);
      raw[0] = raw[1]; raw[1] = raw[2]; raw[2] = raw[3];
    }
  }
  __syncthreads();
  if (p.win_op != 0) {
    // Window maximum by doubling: after the step of width w, src[i] = max of cells [i, i + w);
    // a window of n cells is then the maximum of two overlapping runs of width w <= n < 2w.
    float *src = buf0, *dst = buf1;
    int w = 1;
#pragma unroll 1
    for (int k = 0; k < n_win; ++k) {
      const int combo = tbl.grp_combo[first + k], n = tbl.n[combo];
#pragma unroll 1
      for (; 2 * w <= n; w *= 2) {
        const int cnt = span - 2 * w + 1;
#pragma unroll 1
        for (int i = threadIdx.x; i < cnt; i += kSelThreads) dst[i] = fmaxf(src[i], src[i + w]);
        __syncthreads();
        float* t = src; src = dst; dst = t;
      }
      float* out = p.pooled + static_cast<long long>(combo) * p.pooled_stride + c0;
      uint32_t* hist = (k == 0) ? hist0 : hist1 + (k - 1) * kHistBins;
      const float* s0 = src + (n_max / 2 - n / 2);
#pragma unroll 1
      for (int base = 0; base < n_out; base += kSelThreads) {
        const int i = base + threadIdx.x;
        int bin = -1;
        if (i < n_out) {
          const float acc = ranked_value(fmaxf(s0[i], s0[i + n - w]));
          out[i] = acc;
          bin = bin_of_bits(__float_as_int(acc), p.scores_given != 0);
        }
        count_bins(hist, bin);
      }
      // the next doubling step writes the other buffer, which everyone has left at its last barrier
    }
    __syncthreads();
  } else {
    // Window averages: the sum of n cells from cell u on is the sum of n - 1 cells from u on plus one,
    // added left to right as in the definition, so one pass serves all windows that start at u.
#pragma unroll 1
    for (int base = 0; base < span; base += kSelThreads) {
      const int i = base + threadIdx.x;
      float acc = 0.f;
      int j = 0;
#pragma unroll 1
      for (int k = 0; k < n_win; ++k) {
        const int combo = tbl.grp_combo[first + k], n = tbl.n[combo];
        if (i + n <= span) {
#pragma unroll 4
          for (int jj = j; jj < n; ++jj) acc += buf0[i + jj];
        }
        j = n;
        const int c = i - (n_max / 2 - n / 2);             // cell of the window that starts here
        int bin = -1;
        if (c >= 0 && c < n_out) {
          const float avg = ranked_value(acc / static_cast<float>(n));
          p.pooled[static_cast<long long>(combo) * p.pooled_stride + c0 + c] = avg;
          bin = bin_of_bits(__float_as_int(avg), p.scores_given != 0);
        }
        count_bins((k == 0) ? hist0 : hist1 + (k - 1) * kHistBins, bin);
      }
    }
    __syncthreads();
  }
}

// Phase C for one combination: the bin of its K_m-th largest value, and for every bin the number of
// values in the bins above it.  Every CTA does this for the combinations whose tiles it scans, from the
// same global histogram, so all of them reach the same answer.
__device__ __forceinline__ void find_threshold(const SelectParams& p, const ComboTable& tbl, int combo, SelShared* sh) {
  const uint32_t* gh = p.hist + static_cast<long long>(combo) * kHistBins;
  const uint32_t k = static_cast<uint32_t>(tbl.k_m[combo]);
  static_assert(kHistBins == 2 * kSelThreads, "two bins per thread");
  const int hi = kHistBins - 1 - 2 * threadIdx.x;           // bins in descending order
  const uint2 h = __ldcg(reinterpret_cast<const uint2*>(gh + hi - 1));      // (lower, higher) bin
  uint32_t grand;
  const uint32_t excl = block_exclusive_scan(h.x + h.y, sh->scan, &grand);   // begins with a barrier
  if (threadIdx.x == 0) sh->n_listed = 0u;
  sh->above[hi + 1] = excl;
  sh->above[hi] = excl + h.y;
  if (threadIdx.x == 0) sh->above[0] = grand;
  if (excl < k && k <= excl + h.x + h.y) {
    const bool in_hi = k <= excl + h.y;
    const uint32_t total = in_hi ? excl + h.y : excl + h.x + h.y;
    sh->threshold = in_hi ? hi : hi - 1;
    sh->plateau = total > k + static_cast<uint32_t>(kCandSlack);
    if (total > k + static_cast<uint32_t>(kCandSlack)) {
      p.cand_count[kMaxCombos + combo] = 1u;
      p.cand_count[3 * kMaxCombos] = 1u;
    } else {
      p.cand_count[combo] = total;                          // the same from every CTA
    }
  }
  __syncthreads();
}

// Where the long way begins for a combination whose threshold bin is known (one thread): the bin settles the
// first digit of the K_m-th value's key, so that pass is left out (1048576 given scores in [1/2, 1), 3 windows:
// 58 -> 48 us of long way).  A bin with several first digits (the first one, of the values below zero among
// others): all passes.
__device__ __noinline__ uint8_t start_long_way(uint32_t k, bool given, uint32_t* all_passes, int combo, SelShared* sh) {
  const int digit = bin_digit(sh->threshold, given);
  if (digit < 0) {
    sh->prefix[combo] = 0ull;
    sh->krem[combo] = k;
    *all_passes = 1u;
    return kAllPasses;
  }
  sh->prefix[combo] = static_cast<unsigned long long>(digit) << 53;
  sh->krem[combo] = k - sh->above[last_bin_of_digit(digit, given) + 1];
  return kFirstDigitKnown;
}

// Phase D for the tiles [tile0, tile1) of one combination: the cells of its threshold bin and of the bins
// above, sorted by bin.  Four consecutive cells per thread and tile; few of them are candidates, and
// those come in runs, so they are listed in shared memory first and then placed a cell per thread
// (one after another in the thread that found them, each waited for its counter: up to 3 us).
__device__ __forceinline__ void gather_combination(const SelectParams& p, const ComboTable& tbl, int combo, int tile0,
                                                   int tile1, SelShared* sh, int* list) {
  const float* w = p.pooled + static_cast<long long>(combo) * p.pooled_stride;
  unsigned long long* cand = p.cand + static_cast<long long>(combo) * p.cand_stride;
  uint32_t* seg = p.cand_seg + static_cast<long long>(combo) * p.cand_stride;
  uint32_t* slots = p.hist + static_cast<long long>(tbl.n_comb + combo) * kHistBins;
  const int len = tbl.len[combo], threshold = sh->threshold;
  const float lowest = (threshold == 0) ? -INFINITY : __int_as_float(bin_floor_bits(threshold, p.scores_given != 0));
  auto place = [&](int cell) {
    const float value = __ldcg(w + cell);
    const uint32_t o = float_to_ordered(value);
    const int bin = bin_of_bits(__float_as_int(value), p.scores_given != 0);
    const uint32_t start = sh->above[bin + 1], count = sh->above[bin] - start;
    const uint32_t at = start + atomicAdd(&slots[bin], 1u);
    if (at < static_cast<uint32_t>(p.cand_stride)) {
      cand[at] = (static_cast<unsigned long long>(o) << 32) | (0xFFFFFFFFu - static_cast<uint32_t>(cell));
      seg[at] = start | (count << 16);
    }
  };
#pragma unroll 1
  for (int tile = tile0; tile < tile1; tile += kGatherGroup) {
    const int first = (tile - tbl.tile_begin[combo]) * kSelTile, i0 = 4 * static_cast<int>(threadIdx.x);
    const int n = cells_from(len, first, min(kGatherGroup, tile1 - tile) * kSelTile);
    float4 v[kGatherGroup];
#pragma unroll
    for (int g = 0; g < kGatherGroup; ++g) {
      v[g] = make_float4(NAN, NAN, NAN, NAN);
      if (i0 + g * kSelTile < n) v[g] = __ldcg(reinterpret_cast<const float4*>(w + first + i0 + g * kSelTile));
    }
    uint32_t found = 0;
#pragma unroll
    for (int g = 0; g < kGatherGroup; ++g)
      found |= ((v[g].x >= lowest ? 1u : 0u) | (v[g].y >= lowest ? 2u : 0u) | (v[g].z >= lowest ? 4u : 0u) |
                (v[g].w >= lowest ? 8u : 0u)) << (4 * g);
    if (!found) continue;
    int at = static_cast<int>(atomicAdd(&sh->n_listed, static_cast<uint32_t>(__popc(found))));
#pragma unroll 1
    while (found) {
      const int e = __ffs(found) - 1;
      found &= found - 1;
      const int i = i0 + (e >> 2) * kSelTile + (e & 3);
      if (at < kSelWorkBytes / 4) list[at++] = (i < n) ? first + i : -1;
      else if (i < n) place(first + i);                      // more than the list holds
    }
  }
  __syncthreads();
  const int n = static_cast<int>(min(sh->n_listed, static_cast<uint32_t>(kSelWorkBytes / 4)));
#pragma unroll 1
  for (int i = threadIdx.x; i < n; i += kSelThreads)
    if (list[i] >= 0) place(list[i]);
}

// One pass of the long way: locates the digit of pass `pass` that holds the k-th largest key of `combo`
// among those that match the prefix so far and extends the prefix.  The state lives in shared memory.
// A combination is settled (state = 1) when every key of the chosen digit is wanted: then
// "key >= prefix" selects exactly K_m keys.
__device__ __forceinline__ void bin_search(const SelectParams& p, const uint32_t* gh, int combo, int pass,
                                           SelShared* sh) {
  int shift, bits;
  pass_bits(pass, shift, bits);
  const unsigned long long prefix = sh->prefix[combo];
  const uint32_t k_rem = sh->krem[combo];
  constexpr int kPer = kHistBins / kSelThreads;
  uint32_t h[kPer];
  uint32_t total = 0;
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    h[j] = __ldcg(&gh[kHistBins - 1 - (kPer * threadIdx.x + j)]);   // bins in descending order
    total += h[j];
  }
  uint32_t grand;
  const uint32_t excl = block_exclusive_scan(total, sh->scan, &grand);
  if (excl < k_rem && k_rem <= excl + total) {
    uint32_t cum = excl;
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
      if (k_rem > cum && k_rem <= cum + h[j]) {
        const uint32_t bin = kHistBins - 1 - (kPer * threadIdx.x + j);
        const uint32_t new_k = k_rem - cum;
        sh->prefix[combo] = prefix | (static_cast<unsigned long long>(bin) << shift);
        sh->krem[combo] = new_k;
        sh->state[combo] = (h[j] == new_k) ? 1u : 0u;
      }
      cum += h[j];
    }
  }
  if (threadIdx.x == 0 && (k_rem > grand || k_rem == 0))
    sh->state[combo] = 1u;                                 // fewer keys than asked: take all
  __syncthreads();
}

// Phase E: ranks the candidates [lo, hi) of `combo`, which are sorted by bin: the rank of a candidate is
// where its bin's segment begins plus the keys of the segment above its own (keys are distinct).  The
// segments that the range touches (`unsorted`, after the long way: all is one segment) are staged in
// shared memory, kRankChunk keys at a time; several
// threads share a candidate when there are threads to spare.  Ranks past K_m are not wanted.
//
// A bin may hold thousands of candidates (scores that lie close together, ties), and one CTA may have all
// of them: the early combinations want few cells and get one CTA, and the threshold bin brings up to
// kCandSlack.  Comparing them all costs 20 us per million comparisons and CTA, so from kRankDense
// comparisons on, the keys of the range's segments are first dealt out to kRankBuckets value ranges
// between as many sampled keys (taken at even strides, ranked among themselves), and a candidate is compared
// with its own range only.  The line: 4096 positions in [1/2, 1), 3 windows, 12.3 us compared, 9.1 dealt
// out; 131072 positions that took the long way 16.7 and 11.6.  Phase E with everything compared -> as it
// stands: 4096 positions within 0.1 % of each other, 3 windows, 127 -> 17 us; 131072 in [1/2, 1), 48
// combinations, 472 -> 27; log-normal scores 4.3 and 7.2 us -> 4.6 and 4.7 (the CTA's list is found by all threads).
static constexpr int kRankChunk = 8192;
static constexpr int kRankBuckets = 256;
static constexpr int kRankDense = 150000;

struct RankScratch {
  unsigned long long samp[kRankBuckets];
  unsigned long long spl[kRankBuckets];    // the samples in descending order; the last entry is unused
  uint32_t rank[kRankBuckets];
  uint32_t count[kRankBuckets];
  uint32_t start[kRankBuckets + 1];
};
static_assert(sizeof(RankScratch) <= sizeof(SelShared::hist), "the scratch takes the histogram's place");

// Ranks the keys [lo, hi) of cand[0 .. n), kRankBuckets <= n <= kRankChunk; ranks from `limit` on are not wanted.
__device__ __noinline__ void rank_dense(const unsigned long long* cand, int* ranked, int n, int lo, int hi, int limit,
                                        unsigned long long* grouped, SelShared* sh) {
  RankScratch* rs = reinterpret_cast<RankScratch*>(sh->hist);
  constexpr int kLd = kRankChunk / kSelThreads;
  const int tid = threadIdx.x;
  unsigned long long v[kLd];
#pragma unroll
  for (int k = 0; k < kLd; ++k) {
    const int i = k * kSelThreads + tid;
    v[k] = (i < n) ? __ldcg(&cand[i]) : 0ull;
  }
  if (tid < kRankBuckets) {                                 // (the caller's vote freed the scratch and the chunk)
    rs->samp[tid] = __ldcg(&cand[tid * n / kRankBuckets]);
    rs->rank[tid] = 0;
    rs->count[tid] = 0;
  }
  __syncthreads();
  {                                                         // rank the samples among themselves
    constexpr int kPer = kRankBuckets / (kSelThreads / kRankBuckets);
    const int si = tid % kRankBuckets, j0 = (tid / kRankBuckets) * kPer;
    const unsigned long long mine = rs->samp[si];
    uint32_t above = 0;
#pragma unroll 8
    for (int j = 0; j < kPer; ++j) above += (rs->samp[j0 + j] > mine) ? 1u : 0u;
    if (above) atomicAdd(&rs->rank[si], above);
  }
  __syncthreads();
  if (tid < kRankBuckets) rs->spl[rs->rank[tid]] = rs->samp[tid];
  __syncthreads();
  uint32_t where[kLd];                                      // bucket << 16 | slot inside the bucket
#pragma unroll
  for (int k = 0; k < kLd; ++k) {
    const int i = k * kSelThreads + tid;
    if (i < n) {
      int b = 0;                                            // samples above the key, the last one left out
#pragma unroll
      for (int step = kRankBuckets / 2; step >= 1; step >>= 1)
        if (rs->spl[b + step - 1] > v[k]) b += step;
      where[k] = (static_cast<uint32_t>(b) << 16) | atomicAdd(&rs->count[b], 1u);
    }
  }
  __syncthreads();
  uint32_t total;
  const uint32_t before = block_exclusive_scan(tid < kRankBuckets ? rs->count[tid] : 0u, sh->scan, &total);
  if (tid <= kRankBuckets) rs->start[tid] = before;
  __syncthreads();
#pragma unroll
  for (int k = 0; k < kLd; ++k) {
    const int i = k * kSelThreads + tid;
    if (i < n) grouped[rs->start[where[k] >> 16] + (where[k] & 0xFFFFu)] = v[k];
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < kLd; ++k) {
    const int i = k * kSelThreads + tid;
    if (i < lo || i >= hi) continue;
    const int first = static_cast<int>(rs->start[where[k] >> 16]), last = static_cast<int>(rs->start[(where[k] >> 16) + 1]);
    int rank = first;
#pragma unroll 4
    for (int j = first; j < last; ++j) rank += (grouped[j] > v[k]) ? 1 : 0;
    if (rank < limit) ranked[rank] = static_cast<int>(0xFFFFFFFFu - static_cast<uint32_t>(v[k] & 0xFFFFFFFFull));
  }
}

__device__ __forceinline__ void rank_range(const SelectParams& p, const ComboTable& tbl, int combo, int n, int lo, int hi,
                                           bool unsorted, unsigned long long* chunk, SelShared* sh) {
  const unsigned long long* cand = p.cand + static_cast<long long>(combo) * p.cand_stride;
  const uint32_t* seg = p.cand_seg + static_cast<long long>(combo) * p.cand_stride;
  int* ranked = p.ranked + static_cast<long long>(combo) * p.cand_stride;
  const int k_m = tbl.k_m[combo];
#pragma unroll 1
  for (int c0 = lo; c0 < hi; c0 += kSelThreads) {
    const int nc = min(kSelThreads, hi - c0);
    int g = 1;                                              // threads per candidate
#pragma unroll 1
    while (g < 32 && 2 * g * nc <= kSelThreads) g <<= 1;
    const int local = threadIdx.x / g, sub = threadIdx.x % g;
    const bool active = local < nc;
    const uint32_t whole = static_cast<uint32_t>(n) << 16;  // start | length << 16
    const uint32_t s_first = unsorted ? whole : __ldcg(&seg[c0]);
    const uint32_t s_last = unsorted ? whole : __ldcg(&seg[c0 + nc - 1]);
    const uint32_t s_mine = (active && !unsorted) ? __ldcg(&seg[c0 + local]) : whole;
    const unsigned long long key = active ? __ldcg(&cand[c0 + local]) : ~0ull;
    const int begin = static_cast<int>(s_first & 0xFFFFu);
    const int end = static_cast<int>((s_last & 0xFFFFu) + (s_last >> 16));
    const int first = static_cast<int>(s_mine & 0xFFFFu), last = first + static_cast<int>(s_mine >> 16);
    // the vote is also the barrier behind the previous users of the chunk
    if (__syncthreads_or(active && (last - first) * (hi - c0) > kRankDense)) {
      const uint32_t s_end = unsorted ? whole : __ldcg(&seg[hi - 1]);
      const int len = static_cast<int>((s_end & 0xFFFFu) + (s_end >> 16)) - begin;
      if (len >= kRankBuckets && len <= kRankChunk) {       // uniform
        rank_dense(cand + begin, ranked + begin, len, c0 - begin, hi - begin, k_m - begin, chunk, sh);
        return;
      }
    }
    int above = 0;
#pragma unroll 1
    for (int base = begin; base < end; base += kRankChunk) {
      const int cnt = min(kRankChunk, end - base);
      if (base > begin) __syncthreads();                    // previous users of the chunk
#pragma unroll 1
      for (int i = threadIdx.x; i < cnt; i += kSelThreads) chunk[i] = __ldcg(&cand[base + i]);
      __syncthreads();
      if (active) {
        const int j1 = min(last, base + cnt) - base;
#pragma unroll 4
        for (int j = max(first, base) - base + sub; j < j1; j += g) above += (chunk[j] > key) ? 1 : 0;
      }
    }
#pragma unroll 1
    for (int d = 1; d < g; d <<= 1) above += __shfl_xor_sync(0xFFFFFFFFu, above, d);
    if (active && sub == 0 && first + above < k_m)
      ranked[first + above] = static_cast<int>(0xFFFFFFFFu - static_cast<uint32_t>(key & 0xFFFFFFFFull));
  }
}

// Shared memory of the allocation phase: the bitmap lies behind the work area of the other phases, which
// the output list reuses.
__device__ __forceinline__ uint32_t* smem_bitmap(uint8_t* dyn_smem) {
  return reinterpret_cast<uint32_t*>(dyn_smem + kSelWorkBytes);
}

// Bitmap word access of the quota walk.  The bitmap lives in shared memory on the common path;
// naming the address space spares the generic-address forms.
template <bool kSmem>
__device__ __forceinline__ uint32_t bitmap_word(const uint32_t* bm, int w) {
  if constexpr (kSmem) {
    uint32_t v;
    asm volatile("ld.volatile.shared.u32 %0, [%1];" : "=r"(v) : "r"(smem_u32(bm + w)) : "memory");
    return v;
  } else {
    return *reinterpret_cast<const volatile uint32_t*>(bm + w);
  }
}
// Sets bits where there are any: a predicated atomic, since a branch around each costs more than it saves.
template <bool kSmem>
__device__ __forceinline__ void bitmap_set(uint32_t* bm, int w, uint32_t bits) {
  if constexpr (kSmem) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %1, 0;\n\t@p red.shared.or.b32 [%0], %1;\n\t}"
                 ::"r"(smem_u32(bm + w)), "r"(bits) : "memory");
  } else {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %1, 0;\n\t@p red.global.or.b32 [%0], %1;\n\t}"
                 ::"l"(__cvta_generic_to_global(bm + w)), "r"(bits) : "memory");
  }
}

// The bitmap of allocated tokens covers the context without its sink part: bit t = token t, t < Lp; the
// bits past the end are set from the start, so that they never look free.
__device__ __forceinline__ uint32_t empty_bitmap_word(int w, int Lp) {
  const int left = Lp - 32 * w;
  return (left >= 32) ? 0u : (left <= 0) ? 0xFFFFFFFFu : 0xFFFFFFFFu << left;
}

// How the cells of a combination lie in the bitmap words.
enum : int {
  kCellsAligned = 0,      // m divides 32: inside one word
  kCellsShort = 1,        // m <= 32: in at most two words (one funnel shift)
  kCellsLong = 2          // m <= 64: in at most three words
};
__device__ __forceinline__ int cells_kind(int m) {
  return (m & (m - 1)) == 0 && m <= 32 ? kCellsAligned : m <= 32 ? kCellsShort : kCellsLong;
}

// Tokens of cell `cell` (size m) that are not allocated yet, as a bit mask (bit j = token j).  Positions
// fit 32 bits (L < 2^31).  Up to two words past the bitmap's end may be read (kSelBitmapSlackWords of
// memory lie behind it) but their bits are masked.
template <int kCells, bool kSmem>
__device__ __forceinline__ auto fresh_tokens(const uint32_t* bm, int cell, int m, int Lp) {
  const int t0 = cell * m;
  const int w0 = t0 >> 5, sh = t0 & 31;
  if constexpr (kCells == kCellsAligned) {
    return (~bitmap_word<kSmem>(bm, w0) >> sh) & (0xFFFFFFFFu >> (32 - m));
  } else if constexpr (kCells == kCellsShort) {
    const uint32_t taken = __funnelshift_r(bitmap_word<kSmem>(bm, w0), bitmap_word<kSmem>(bm, w0 + 1), sh);
    return ~taken & (0xFFFFFFFFu >> (32 - min(m, Lp - t0)));
  } else {
    unsigned long long taken = bitmap_word<kSmem>(bm, w0);
    taken |= static_cast<unsigned long long>(bitmap_word<kSmem>(bm, w0 + 1)) << 32;
    taken >>= sh;
    if (sh) taken |= static_cast<unsigned long long>(bitmap_word<kSmem>(bm, w0 + 2)) << (64 - sh);
    return ~taken & (~0ull >> (64 - min(m, Lp - t0)));
  }
}

// Marks the fresh tokens `f` of a cell that starts at token t0 and may lie in several words.
template <int kCells, bool kSmem, class Mask>
__device__ __forceinline__ void mark_tokens(uint32_t* bm, int t0, Mask f) {
  const int w0 = t0 >> 5, sft = t0 & 31;
  if constexpr (kCells == kCellsShort) {
    bitmap_set<kSmem>(bm, w0, f << sft);
    bitmap_set<kSmem>(bm, w0 + 1, __funnelshift_l(f, 0u, sft));
  } else {
    const unsigned long long shifted = f << sft;
    bitmap_set<kSmem>(bm, w0, static_cast<uint32_t>(shifted));
    bitmap_set<kSmem>(bm, w0 + 1, static_cast<uint32_t>(shifted >> 32));
    bitmap_set<kSmem>(bm, w0 + 2, sft ? static_cast<uint32_t>(f >> (64 - sft)) : 0u);
  }
}

// One round of the quota walk over a combination: kWalkCells consecutive ranks per lane, r0 on, a warp those of
// its lanes in turn; c: their cells.  The cells of a combination are disjoint, so all of a round's
// cells are counted before any is marked, and a round's marks do not change another round's counts: one
// barrier per round, `tot`: the warps' counts, two buffers that the rounds use in turn.  `taken`: tokens of
// the combination's rounds before (kept up to date when another round follows; in warp 0 always).
//
// What a round costs is the instructions that each warp has to fetch and issue (about three cycles each) and
// the chain of its steps (B200, cycles: shuffle 40, warp reduction 52, block barrier 35 with one warp and 104
// with 32; several lanes' atomics on one word 31 per lane; a divergent branch about 50).  So only the warp in which
// the quota ends looks at the order of its lanes, warps behind it mark nothing, and a lane's
// neighbouring cells mark a bitmap word together (a plateau's cells are ranked one behind the other).
// The walk of 3 / 4 / 5 / 48 combinations (4K, 128K, 1M, 200003 positions), one cell after another in each lane
// and lists copied to shared memory a step ahead -> as it stands: 4.6, 10, 13, 66 -> 2.8, 6.2, 8.5, 42 us.
template <int kCells, bool kSmem, class Barrier>
__device__ __forceinline__ void walk_round(const SelectParams& p, const int (&c)[kWalkCells], int r0, int K, int m,
                                           uint32_t quota, uint32_t* bm, uint32_t* tot, uint32_t& taken, bool last_round,
                                           int n_walk, Barrier walk_barrier) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int Lp = static_cast<int>(p.L - p.n_sink);
  auto count = [](auto f) -> uint32_t {
    if constexpr (kCells == kCellsLong) return __popcll(f); else return __popc(f);
  };
  decltype(fresh_tokens<kCells, kSmem>(bm, 0, m, Lp)) f[kWalkCells];
  uint32_t mine = 0, sum = 0;                                  // of this lane, of the warp
  if (r0 - kWalkCells * lane < K) {                            // uniform
#pragma unroll
    for (int j = 0; j < kWalkCells; ++j) {
      f[j] = fresh_tokens<kCells, kSmem>(bm, (r0 + j < K) ? c[j] : 0, m, Lp);
      if (r0 + j >= K) f[j] = 0;
      mine += count(f[j]);
    }
    sum = __reduce_add_sync(0xFFFFFFFFu, mine);
  }
  if (lane == 0) tot[warp] = sum;
  walk_barrier();
  const uint32_t wt = (lane < n_walk / 32) ? tot[lane] : 0u;
  const uint32_t before = taken + __reduce_add_sync(0xFFFFFFFFu, lane < warp ? wt : 0u);
  if (!last_round || warp == 0) taken += __reduce_add_sync(0xFFFFFFFFu, wt);
  if (before >= quota || sum == 0) return;                     // uniform
  if (before + sum > quota) {                                  // the quota ends inside this warp
    uint32_t incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= o) incl += t;
    }
    const uint32_t ord = before + incl - mine;
    uint32_t room = ord < quota ? quota - ord : 0u;
    auto end = f[0];                                           // the cell in which the quota ends
    uint32_t end_room = 0;
    int end_cell = 0;
#pragma unroll
    for (int j = 0; j < kWalkCells; ++j) {
      const uint32_t n_new = count(f[j]);
      const bool all = n_new <= room;
      if (!all && room) { end = f[j]; end_room = room; end_cell = c[j]; }
      f[j] = all ? f[j] : 0;
      room = all ? room - n_new : 0;
    }
    if (end_room) {                                            // its lowest tokens
      auto rest = end;
#pragma unroll 1
      for (uint32_t k = 0; k < end_room; ++k) rest &= rest - 1;
      const int t0 = end_cell * m;
      if constexpr (kCells == kCellsAligned) bitmap_set<kSmem>(bm, t0 >> 5, (end ^ rest) << (t0 & 31));
      else mark_tokens<kCells, kSmem>(bm, t0, end ^ rest);
    }
  }
  if constexpr (kCells == kCellsAligned) {
    uint32_t bits = 0;
#pragma unroll
    for (int j = 0; j < kWalkCells; ++j) {
      const int t0 = c[j] * m;
      bits |= f[j] << (t0 & 31);
      const bool goes_on = j + 1 < kWalkCells && (c[(j + 1) % kWalkCells] * m) >> 5 == t0 >> 5;
      bitmap_set<kSmem>(bm, t0 >> 5, goes_on ? 0u : bits);
      bits = goes_on ? bits : 0u;
    }
  } else {
#pragma unroll
    for (int j = 0; j < kWalkCells; ++j) mark_tokens<kCells, kSmem>(bm, c[j] * m, f[j]);
  }
}

// Writes the positions of one bitmap word per lane (`bits` of word `w`, its first position at `place`).  A
// lane writes its word's positions itself where they are few, the warp together, a lane each, those of
// a word with more: quoted passages fill whole words, and a lane by itself takes 32 steps for one.
__device__ __forceinline__ void emit_words(const SelectParams& p, uint32_t bits, int w, uint32_t place, uint32_t cap) {
  constexpr uint32_t kAlone = 4;
  const uint32_t lane = threadIdx.x & 31, n = __popc(bits);
  const int pos0 = p.n_sink + w * 32;
  uint32_t together = __ballot_sync(0xFFFFFFFFu, n > kAlone);
#pragma unroll 1
  while (together) {
    const int a = __ffs(together) - 1;                         // two words per turn
    together &= together - 1;
    const int b = together ? __ffs(together) - 1 : a;
    together &= together - 1;                                  // (0 stays 0)
    const uint32_t bits_a = __shfl_sync(0xFFFFFFFFu, bits, a), bits_b = __shfl_sync(0xFFFFFFFFu, bits, b);
    const uint32_t place_a = __shfl_sync(0xFFFFFFFFu, place, a), place_b = __shfl_sync(0xFFFFFFFFu, place, b);
    const int pos_a = __shfl_sync(0xFFFFFFFFu, pos0, a), pos_b = __shfl_sync(0xFFFFFFFFu, pos0, b);
    const uint32_t lt = (1u << lane) - 1u;
    const uint32_t at_a = place_a + __popc(bits_a & lt), at_b = place_b + __popc(bits_b & lt);
    if (((bits_a >> lane) & 1u) && at_a < cap) p.out_idx[at_a] = pos_a + lane;
    if (((bits_b >> lane) & 1u) && at_b < cap) p.out_idx[at_b] = pos_b + lane;
  }
  if (n <= kAlone) {
#pragma unroll 1
    while (bits) {
      const int k = __ffs(bits) - 1;
      bits &= bits - 1;
      if (place < cap) p.out_idx[place] = pos0 + k;
      ++place;
    }
  }
}

// Exclusive prefix sum over the block with a single barrier: every warp scans the 32 warp
// totals itself.  `slot` alternates between calls (two buffers), which keeps a call's readers
// apart from the next call's writers.
__device__ __forceinline__ uint32_t block_exclusive_scan_1(uint32_t v, uint32_t (*tot)[32],
                                                           int slot, uint32_t* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) tot[slot][warp] = incl;
  __syncthreads();
  const uint32_t w = tot[slot][lane];
  uint32_t wi = w;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, wi, o);
    if (lane >= o) wi += t;
  }
  *total = __shfl_sync(0xFFFFFFFFu, wi, 31);
  return __shfl_sync(0xFFFFFFFFu, wi - w, warp) + incl - v;
}

// Phase F (one CTA): quota walk over the ranked cells of every combination, then the
// ascending list of allocated positions.  The bitmap lives in shared memory when it fits
// (cleared at the start of the kernel, beside the memory of the other phases), else in global
// memory.
template <bool kBitmapInSmem>
__device__ __forceinline__ void allocate(const ComboTable& tbl, const SelectParams& p,
                                         uint8_t* dyn_smem, SelShared* sh) {
  // Two instantiations, so that the compiler knows the bitmap's address space on the common
  // path (shared memory) instead of going through generic loads and atomics.
  uint32_t* bm = kBitmapInSmem ? smem_bitmap(dyn_smem) : p.bitmap;
  __shared__ uint32_t warp_totals[2][kMaxWalkWarps];
  const int n_walk = p.walk_threads;                       // multiple of 32, <= kSelThreads
  // The walk is a chain of short dependent rounds, at least one per combination: walk_threads threads walk
  // (kWalkCells ranked cells each for the longest list, as long as there are so many threads), the others
  // wait for the output pass.  A thread fetches its cells of a round while it walks the one before.
  if (static_cast<int>(threadIdx.x) < n_walk) {
    auto walk_barrier = [&] { asm volatile("bar.sync 1, %0;" ::"r"(n_walk) : "memory"); };
    const int n_comb = tbl.n_comb, first = kWalkCells * static_cast<int>(threadIdx.x);
    static_assert(kWalkCells == 4, "one 16-byte load per round");
    auto fetch = [&](int combo, int r0, int K) -> int4 {
      return (r0 < K) ? __ldcg(reinterpret_cast<const int4*>(p.ranked + static_cast<long long>(combo) * p.cand_stride + r0))
                      : make_int4(0, 0, 0, 0);
    };
    int4 entry = n_comb > 0 ? sh->walk[0] : make_int4(1, 0, 0, 0);
    int4 next = fetch(0, first, entry.z);
    uint32_t round = 0;
#pragma unroll 1
    for (int combo = 0; combo < n_comb; ++combo) {
      const int m = entry.x, K = entry.z, kind = entry.w;
      const uint32_t quota = static_cast<uint32_t>(entry.y);
      entry = combo + 1 < n_comb ? sh->walk[combo + 1] : make_int4(1, 0, 0, 0);
      uint32_t taken = 0;
      int base = 0;
#pragma unroll 1
      for (;;) {
        const int c[kWalkCells] = {next.x, next.y, next.z, next.w};
        const int r0 = base + first;
        uint32_t* tot = warp_totals[round++ & 1u];
        base += kWalkCells * n_walk;
        const bool last_round = base >= K;
        next = last_round ? fetch(combo + 1, first, entry.z) : fetch(combo, base + first, K);
        if (kind == kCellsAligned)
          walk_round<kCellsAligned, kBitmapInSmem>(p, c, r0, K, m, quota, bm, tot, taken, last_round, n_walk, walk_barrier);
        else if (kind == kCellsShort)
          walk_round<kCellsShort, kBitmapInSmem>(p, c, r0, K, m, quota, bm, tot, taken, last_round, n_walk, walk_barrier);
        else
          walk_round<kCellsLong, kBitmapInSmem>(p, c, r0, K, m, quota, bm, tot, taken, last_round, n_walk, walk_barrier);
        if (last_round) break;
        if (taken >= quota) {                                  // met before the list's end: the wrong cells were fetched
          next = fetch(combo + 1, first, entry.z);
          break;
        }
      }
      if (threadIdx.x == 0 && taken < quota) atomicCAS(p.status, 0, kDevQuota);
      walk_barrier();                                          // bitmap updates visible
    }
  }
  // The bits past the end, which had to look taken, stand for nothing from here on.
  const int Lp = static_cast<int>(p.L - p.n_sink), n_quads = (Lp + 127) / 128;     // bitmap words by fours
  if (threadIdx.x < 4) {
    const int w = Lp / 32 + static_cast<int>(threadIdx.x);
    const uint32_t keep = (threadIdx.x == 0) ? (1u << (Lp & 31)) - 1u : 0u;
    if (w < 4 * n_quads) bm[w] = bitmap_word<kBitmapInSmem>(bm, w) & keep;
  }
  __syncthreads();

  // Ascending output.  One SM does this, so what counts is the number of instructions it has to issue (with 32
  // warps a shuffle takes 6 cycles of a scheduler, a vote 3.6, a population count 2.7) and that it meets
  // them cold (a line that is not in its cache costs some 300 cycles).  The sink part is the identity.
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t cap = static_cast<uint32_t>(p.n_sink + p.budget);
#pragma unroll 1
  for (int j = threadIdx.x; j < p.n_sink; j += kSelThreads) p.out_idx[j] = j;
  uint32_t total;
  if (4 * n_quads <= kSelThreads) {
    // up to 32K positions: a lane per bitmap word, the words shared out evenly over the warps (32K: 3.5 -> 2.4 us)
    const int per = (4 * n_quads + kMaxWalkWarps - 1) / kMaxWalkWarps, w = warp * per + lane;
    const uint32_t bits = (lane < per && w < 4 * n_quads) ? bitmap_word<kBitmapInSmem>(bm, w) : 0u;
    const uint32_t before = block_exclusive_scan(__popc(bits), sh->scan, &total);
    emit_words(p, bits, w, p.n_sink + before, cap);
    if (threadIdx.x == 0 && total != static_cast<uint32_t>(p.budget)) atomicCAS(p.status, 0, kDevQuota);
    return;
  }
  // Longer contexts: every warp takes an equal run of the bitmap and counts the words that are not empty (a few in a
  // hundred, neighbours for the most part) and their positions; with the sums of the warps' before it, it goes
  // through the run again and enters the words, in order, in the block's list.  Then it writes the positions of
  // its own words, a lane per word.  But passages may lie anywhere, all of them in one warp's run too: where a
  // warp would have a round of words more than an equal share of the list, all take equal shares, which
  // costs two barriers and another sum.  (Own words always / shares always / as it stands, us: allocation, budget 4096,
  // chosen from one 32nd of the context, 131072 positions 45.1 / 39.0 / 39.0, 524288 80.4 / 64.7 / 65.2, 4000000
  // 143 / 102 / 103, spread out, 524288 91.5 / 92.2 / 91.9; recalls of 81690 positions, budget 1024, 118.6 / 120.2 / 118.8.)
  const int per = ((n_quads + kMaxWalkWarps - 1) / kMaxWalkWarps + 31) & ~31;
  const int q_begin = min(n_quads, warp * per), q_end = min(n_quads, q_begin + per);
  auto load_quad = [&](int q) -> uint4 {
    if (q >= q_end) return make_uint4(0u, 0u, 0u, 0u);
    if constexpr (kBitmapInSmem) return reinterpret_cast<const uint4*>(bm)[q];
    else return __ldcg(reinterpret_cast<const uint4*>(bm) + q);
  };
  uint32_t mine = 0;                                             // positions | words << 16
#pragma unroll 1
  for (int q = q_begin; q < q_end; q += 32) {
    const uint4 v = load_quad(q + lane);
    if (__any_sync(0xFFFFFFFFu, (v.x | v.y | v.z | v.w) != 0u))
      mine += __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w) +
              (((v.x ? 1u : 0u) + (v.y ? 1u : 0u) + (v.z ? 1u : 0u) + (v.w ? 1u : 0u)) << 16);
  }
  constexpr uint32_t kList = kSelWorkBytes / 4;
  static_assert(kList >= kMaxKm && kMaxKm < 65536, "the list holds a word per position, a count fits 16 bits");
  int* list = reinterpret_cast<int*>(dyn_smem);
  uint32_t at = block_exclusive_scan(mine, sh->scan, &total);
  at = __shfl_sync(0xFFFFFFFFu, at, 0);
  if (threadIdx.x == 0 && (total & 0xFFFFu) != static_cast<uint32_t>(p.budget)) atomicCAS(p.status, 0, kDevQuota);
  const int n_listed = static_cast<int>(min(total >> 16, kList)), share = (n_listed + kMaxWalkWarps - 1) / kMaxWalkWarps;
  const bool own = __reduce_max_sync(0xFFFFFFFFu, sh->scan[lane] >> 16) <= static_cast<uint32_t>(share + 32);   // the same for all
  uint32_t to = at >> 16;
  int e_begin = min(static_cast<int>(to), n_listed);
#pragma unroll 1
  for (int q = q_begin; q < q_end; q += 32) {
    const uint4 v = load_quad(q + lane);
    const uint32_t full = (v.x ? 1u : 0u) | (v.y ? 2u : 0u) | (v.z ? 4u : 0u) | (v.w ? 8u : 0u);
    if (!__any_sync(0xFFFFFFFFu, full != 0u)) continue;
    // a word's place in the list: behind the words of the lanes before, by votes, and those of its own lane
    const uint32_t lt = (1u << lane) - 1u;
    uint32_t place = to;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint32_t votes = __ballot_sync(0xFFFFFFFFu, (full >> k) & 1u);
      place += __popc(votes & lt);
      to += __popc(votes);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if ((full >> k) & 1u) {
        if (place < kList) list[place] = 4 * (q + lane) + k;     // never past it unless a quota was overrun
        ++place;
      }
  }
  int e_end = min(static_cast<int>(to), n_listed);
  at = p.n_sink + (at & 0xFFFFu);
  if (own) {
    __syncwarp();
  } else {
    __syncthreads();
    e_begin = min(n_listed, warp * share);
    e_end = min(n_listed, e_begin + share);
    mine = 0;
#pragma unroll 1
    for (int e = e_begin + lane; e < e_end; e += 32) mine += __popc(bitmap_word<kBitmapInSmem>(bm, list[e]));
    at = p.n_sink + block_exclusive_scan(mine, sh->scan, &total);
    at = __shfl_sync(0xFFFFFFFFu, at, 0);
  }
#pragma unroll 1
  for (int e = e_begin; e < e_end; e += 32) {
    const int w = (e + lane < e_end) ? list[e + lane] : 0;
    const uint32_t bits = (e + lane < e_end) ? bitmap_word<kBitmapInSmem>(bm, w) : 0u, n = __popc(bits);
    uint32_t incl = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= o) incl += t;
    }
    emit_words(p, bits, w, at + incl - n, cap);
    at += __shfl_sync(0xFFFFFFFFu, incl, 31);
  }
}

// The long way, for the combinations whose threshold bin is a plateau: the K_m-th value, then the ties and
// the gather.  Out of line, as it is hardly ever needed and the kernel meets its code cold: recalls of 4096
// tokens in a row 46.3 us with it inline, 45.3 so (it costs the long way itself 2 to 8 us).  tbl and p are
// references into the kernel's parameters (__grid_constant__; a copy in local memory took 60 us).
// Returns the barrier's epoch, kGaveUp when a barrier gave up.
static constexpr uint32_t kGaveUp = 0xFFFFFFFFu;
template <bool kCluster>
__device__ __noinline__ uint32_t long_way(const ComboTable& tbl, const SelectParams& p, SelShared* sh, int t_begin,
                                      int t_end, int c_lo, int c_hi, uint32_t epoch) {
  uint32_t* pass_hist = p.hist + 2ll * tbl.n_comb * kHistBins;
  const long long n_hist = static_cast<long long>(kSelectPasses) * tbl.n_comb * kHistBins;
  const int first_pass = __ldcg(&p.cand_count[3 * kMaxCombos + 1]) != 0u ? 0 : 1;       // the same for every CTA
  for (long long i = static_cast<long long>(blockIdx.x) * kSelThreads + threadIdx.x; i < n_hist;
       i += static_cast<long long>(gridDim.x) * kSelThreads)
    pass_hist[i] = 0u;
  for (int combo = c_lo + threadIdx.x; combo <= c_hi; combo += kSelThreads) {
    // nothing left to do for those that do not go the long way
    sh->state[combo] = sh->mode[combo] == 0 ? 1u : (sh->mode[combo] == kFirstDigitKnown && first_pass == 0) ? 2u : 0u;
  }
  if (!grid_sync<kCluster>(p, sh, epoch)) return kGaveUp;
  for (int pass = first_pass; pass < kSelectPasses; ++pass) {
    if (pass == 1) {
      for (int combo = c_lo + threadIdx.x; combo <= c_hi; combo += kSelThreads)
        if (sh->state[combo] == 2u) sh->state[combo] = 0u;
      __syncthreads();
    }
    int shift, bits;
    pass_bits(pass, shift, bits);
    const uint32_t mask = (1u << bits) - 1u;
    uint32_t* hist_pass = pass_hist + static_cast<long long>(pass) * tbl.n_comb * kHistBins;
    int cur = -1, load_cursor = 0, cursor = 0;
    for (int t0 = t_begin; t0 < t_end; t0 += kScanGroup) {
      float wv[kScanGroup][kTilePer];
#pragma unroll
      for (int g = 0; g < kScanGroup; ++g)
        if (t0 + g < t_end) fetch_tile(tbl, p, t0 + g, load_cursor, sh->state, wv[g]);
#pragma unroll
      for (int g = 0; g < kScanGroup; ++g) {
        const int tile = t0 + g;
        if (tile >= t_end) break;
        const int combo = combo_of_tile(tbl, tile, cursor);
        if (sh->state[combo]) continue;
        if (combo != cur && cur >= 0)
          hist_flush(sh->hist, hist_pass + static_cast<long long>(cur) * kHistBins);
        cur = combo;
        const unsigned long long prefix = sh->prefix[combo];
        const int c0 = (tile - tbl.tile_begin[combo]) * kSelTile, n = cells_from(tbl.len[combo], c0, kSelTile);
#pragma unroll
        for (int k = 0; k < kTilePer; ++k) {
          const int i = k * kSelThreads + threadIdx.x;
          uint32_t digit = 0xFFFFFFFFu;                    // sentinel: does not take part
          if (i < n) {
            const unsigned long long key = make_key(wv[g][k], static_cast<uint32_t>(c0 + i));
            if (pass == 0 || ((key ^ prefix) >> (shift + bits)) == 0ull)
              digit = static_cast<uint32_t>(key >> shift) & mask;
          }
          hist_add(sh->hist, digit);
        }
      }
    }
    if (cur >= 0) hist_flush(sh->hist, hist_pass + static_cast<long long>(cur) * kHistBins);
    if (!grid_sync<kCluster>(p, sh, epoch)) return kGaveUp;
    for (int combo = c_lo; combo <= c_hi; ++combo)
      if (sh->state[combo] == 0u)
        bin_search(p, hist_pass + static_cast<long long>(combo) * kHistBins, combo, pass, sh);
  }

  // ---- D: ties at the K_m-th value, then the gather ----
  // A combination that is not settled by now has its K_m-th value v (upper half of the
  // prefix) and wants krem of the cells that hold exactly v: the ones with the lowest index.
  {
    int load_cursor = 0, cursor = 0;
    for (int t0 = t_begin; t0 < t_end; t0 += kScanGroup) {
      float wv[kScanGroup][kTilePer];
#pragma unroll
      for (int g = 0; g < kScanGroup; ++g)
        if (t0 + g < t_end) fetch_tile(tbl, p, t0 + g, load_cursor, sh->state, wv[g]);
#pragma unroll
      for (int g = 0; g < kScanGroup; ++g) {
        const int tile = t0 + g;
        if (tile >= t_end) break;
        const int combo = combo_of_tile(tbl, tile, cursor);
        if (sh->state[combo]) continue;
        const uint32_t v_star = static_cast<uint32_t>(sh->prefix[combo] >> 32);
        const int c0 = (tile - tbl.tile_begin[combo]) * kSelTile, n = cells_from(tbl.len[combo], c0, kSelTile);
        int mine = 0;
#pragma unroll
        for (int k = 0; k < kTilePer; ++k) {
          const int i = k * kSelThreads + threadIdx.x;
          mine += (i < n && float_to_ordered(wv[g][k]) == v_star) ? 1 : 0;
        }
        const int holders = __syncthreads_count(mine & 1) + 2 * __syncthreads_count(mine & 2) +
                            4 * __syncthreads_count(mine & 4);
        if (threadIdx.x == 0) p.tile_ties[tile] = holders;
      }
    }
  }
  if (!grid_sync<kCluster>(p, sh, epoch)) return kGaveUp;
  {
    const int lane = threadIdx.x & 31;
    int load_cursor = 0, cursor = 0;
    for (int t0 = t_begin; t0 < t_end; t0 += kScanGroup) {
      float wv[kScanGroup][kTilePer];
#pragma unroll
      for (int g = 0; g < kScanGroup; ++g)
        if (t0 + g < t_end) fetch_tile(tbl, p, t0 + g, load_cursor, nullptr, wv[g]);
#pragma unroll
      for (int g = 0; g < kScanGroup; ++g) {
        const int tile = t0 + g;
        if (tile >= t_end) break;
        const int combo = combo_of_tile(tbl, tile, cursor);
        if (!sh->mode[combo]) continue;                       // gathered in the first scan
        const bool settled = sh->state[combo] != 0u;
        const unsigned long long threshold = sh->prefix[combo];
        const uint32_t v_star = static_cast<uint32_t>(threshold >> 32);
        const uint32_t wanted = sh->krem[combo];
        unsigned long long* cand = p.cand + static_cast<long long>(combo) * p.cand_stride;
        const int c0 = (tile - tbl.tile_begin[combo]) * kSelTile, n = cells_from(tbl.len[combo], c0, kSelTile);
        // holders of v in the earlier tiles of this combination (tiles are in cell order)
        uint32_t before = 0;
        bool ties_here = false;
        if (!settled) {
          ties_here = __ldcg(&p.tile_ties[tile]) > 0;      // uniform
          if (ties_here) {
            uint32_t part = 0;
            for (int t = tbl.tile_begin[combo] + threadIdx.x; t < tile; t += kSelThreads)
              part += static_cast<uint32_t>(__ldcg(&p.tile_ties[t]));
            block_exclusive_scan_1(part, sh->tot, 0, &before);
            __syncthreads();
          }
        }
#pragma unroll
        for (int k = 0; k < kTilePer; ++k) {
          const int i = k * kSelThreads + threadIdx.x;
          unsigned long long key = 0ull;
          bool take = false, holder = false;
          if (i < n) {
            key = make_key(wv[g][k], static_cast<uint32_t>(c0 + i));
            const uint32_t v = static_cast<uint32_t>(key >> 32);
            if (settled) take = key >= threshold;
            else { take = v > v_star; holder = v == v_star; }
          }
          if (ties_here) {                                 // uniform
            uint32_t in_row;
            const uint32_t rank = before + block_exclusive_scan_1(holder ? 1u : 0u, sh->tot, 1, &in_row);
            __syncthreads();
            if (holder && rank < wanted) take = true;
            before += in_row;
          }
          const uint32_t votes = __ballot_sync(0xFFFFFFFFu, take);
          if (votes) {
            uint32_t slot = 0;
            if (lane == __ffs(votes) - 1) slot = atomicAdd(&p.cand_count[combo], __popc(votes));
            slot = __shfl_sync(0xFFFFFFFFu, slot, __ffs(votes) - 1) +
                   __popc(votes & ((1u << lane) - 1u));
            if (take && slot < static_cast<uint32_t>(tbl.k_m[combo])) cand[slot] = key;
          }
        }
      }
    }
  }
  return epoch;
}

template <bool kCluster>
__global__ void __launch_bounds__(kSelThreads, 1)
select_kernel(const __grid_constant__ ComboTable tbl, const __grid_constant__ SelectParams p) {
  extern __shared__ __align__(16) uint8_t dyn_smem[];
  __shared__ SelShared sh;
  const int n_tiles = tbl.tile_begin[tbl.n_comb];
  const int t_begin = static_cast<int>(static_cast<long long>(blockIdx.x) * n_tiles / gridDim.x);
  const int t_end = static_cast<int>(static_cast<long long>(blockIdx.x + 1) * n_tiles / gridDim.x);
  for (int b = threadIdx.x; b < kHistBins; b += kSelThreads) sh.hist[b] = 0u;
  if (blockIdx.x == 0 && p.bitmap_in_smem) {               // for phase F: empty
    uint32_t* bm = smem_bitmap(dyn_smem);
    const int n_words = static_cast<int>((p.L + 31) / 32), Lp = static_cast<int>(p.L - p.n_sink);
#pragma unroll 1
    for (int w = threadIdx.x; w < n_words; w += kSelThreads) bm[w] = empty_bitmap_word(w, Lp);
  }
  uint32_t epoch = 0;
  grid_dep_wait();       // the kernel before this one (scores, state cleared for this run) is done

  // ---- A: strided max-pool arrays, one per distinct m > 1 ----
  if (tbl.n_src > 0) {
    const int n_st = tbl.src_tile_begin[tbl.n_src];
    const int s_begin = static_cast<int>(static_cast<long long>(blockIdx.x) * n_st / gridDim.x);
    const int s_end = static_cast<int>(static_cast<long long>(blockIdx.x + 1) * n_st / gridDim.x);
    int src = 0;
#pragma unroll 1
    for (int tile = s_begin; tile < s_end; ++tile) {
#pragma unroll 1
      while (src + 1 < tbl.n_src && tile >= tbl.src_tile_begin[src + 1]) ++src;
      maxpool_tile(tbl, p, src, tile - tbl.src_tile_begin[src], reinterpret_cast<uint32_t*>(dyn_smem));
    }
    if (!grid_sync<kCluster>(p, &sh, epoch)) return;
  }

  // ---- B: window pooling of every combination + histograms ----
  {
    uint32_t* hist1 = reinterpret_cast<uint32_t*>(dyn_smem);          // of the group's combinations after the first
    float* buf0 = reinterpret_cast<float*>(hist1 + (kPoolGroup - 1) * kHistBins);
    float* buf1 = buf0 + (kPoolTileMax + kMaxWin);
    for (int i = threadIdx.x; i < (kPoolGroup - 1) * kHistBins; i += kSelThreads) hist1[i] = 0u;
    __syncthreads();
    const int n_pt = tbl.grp_tile_begin[tbl.n_grp], per = tbl.pool_tile;
    const int p_begin = static_cast<int>(static_cast<long long>(blockIdx.x) * n_pt / gridDim.x);
    const int p_end = static_cast<int>(static_cast<long long>(blockIdx.x + 1) * n_pt / gridDim.x);
    int grp = 0;
#pragma unroll 1
    for (int tile = p_begin; tile < p_end; ++tile) {
#pragma unroll 1
      while (grp + 1 < tbl.n_grp && tile >= tbl.grp_tile_begin[grp + 1]) ++grp;
      const int c0 = (tile - tbl.grp_tile_begin[grp]) * per, first = tbl.grp_first[grp];
      pool_tile(tbl, p, grp, c0, min(per, tbl.len[tbl.grp_combo[first]] - c0), buf0, buf1, sh.hist, hist1);
      if (tile + 1 == p_end || tile + 1 == tbl.grp_tile_begin[grp + 1]) {      // the CTA's last tile of this group
#pragma unroll 1
        for (int k = 0; first + k < tbl.grp_first[grp + 1]; ++k)               // (which ended with a barrier)
          hist_drain((k == 0) ? sh.hist : hist1 + (k - 1) * kHistBins,
                     p.hist + static_cast<long long>(tbl.grp_combo[first + k]) * kHistBins);
        __syncthreads();
      }
    }
  }
  if (!grid_sync<kCluster>(p, &sh, epoch)) return;

  // ---- C, D: the threshold bin of every combination this CTA scans, and the gather ----
  int c_lo = 0, c_hi = -1;
  if (t_begin < t_end) {
    int cursor = 0;
    c_lo = combo_of_tile(tbl, t_begin, cursor);
    c_hi = combo_of_tile(tbl, t_end - 1, cursor);
  }
#pragma unroll 1
  for (int combo = c_lo; combo <= c_hi; ++combo) {
    find_threshold(p, tbl, combo, &sh);
    if (threadIdx.x == 0) {
      sh.mode[combo] = sh.plateau ? start_long_way(static_cast<uint32_t>(tbl.k_m[combo]), p.scores_given != 0,
                                                   p.cand_count + 3 * kMaxCombos + 1, combo, &sh)
                                  : 0;
    }
    if (!sh.plateau)                                         // uniform
      gather_combination(p, tbl, combo, max(t_begin, tbl.tile_begin[combo]), min(t_end, tbl.tile_begin[combo + 1]), &sh,
                         reinterpret_cast<int*>(dyn_smem));
    __syncthreads();                                         // readers of the threshold words
  }
  if (!grid_sync<kCluster>(p, &sh, epoch)) return;

  // The long way, for the combinations whose threshold bin is a plateau.  The flag is the same for every CTA.
  if (__ldcg(&p.cand_count[3 * kMaxCombos]) != 0u) {
    epoch = long_way<kCluster>(tbl, p, &sh, t_begin, t_end, c_lo, c_hi, epoch);
    if (epoch == kGaveUp) return;
    if (!grid_sync<kCluster>(p, &sh, epoch)) return;
  }

  // ---- E: ranking ----
  {
    unsigned long long* chunk = reinterpret_cast<unsigned long long*>(dyn_smem);
    const int grid = static_cast<int>(gridDim.x), bid = static_cast<int>(blockIdx.x);
#pragma unroll 1
    for (int combo = threadIdx.x; combo < tbl.n_comb; combo += kSelThreads) {
      const uint32_t n = min(__ldcg(&p.cand_count[combo]), static_cast<uint32_t>(p.cand_stride));
      sh.state[combo] = n;
      sh.mode[combo] = static_cast<uint8_t>(__ldcg(&p.cand_count[kMaxCombos + combo]));     // came the long way
      sh.walk[combo] = make_int4(tbl.m[combo], tbl.quota[combo],
                                 min(static_cast<int>(min(n, static_cast<uint32_t>(kMaxKm))), tbl.k_m[combo]),
                                 cells_kind(tbl.m[combo]));
      const int b0 = tbl.rank_cta_begin[combo], share = tbl.rank_cta_begin[combo + 1] - b0;
      if (tbl.rank_by_list && bid >= b0 && bid < b0 + share) {
        sh.list = combo;
        sh.krem[0] = n * static_cast<uint32_t>(bid - b0) / static_cast<uint32_t>(share);
        sh.krem[1] = n * static_cast<uint32_t>(bid - b0 + 1) / static_cast<uint32_t>(share);
      }
    }
    __syncthreads();
    // Enough CTAs: each serves one combination only (a CTA that met two would stage and split both lists,
    // and the whole grid would wait for it).  The host has dealt the CTAs out: combination c has
    // [rank_cta_begin[c], rank_cta_begin[c + 1]).  Fewer CTAs than lists: every CTA takes a contiguous run
    // of all candidates.
    const int only = tbl.rank_by_list ? sh.list : -1;
    long long n_cand = 0;
#pragma unroll 1
    for (int combo = 0; combo < tbl.n_comb && only < 0; ++combo) n_cand += sh.state[combo];
    const int i_begin = static_cast<int>(static_cast<long long>(bid) * n_cand / grid);
    const int i_end = static_cast<int>(static_cast<long long>(bid + 1) * n_cand / grid);
    int first = 0;
#pragma unroll 1
    for (int combo = max(only, 0); combo < (only < 0 ? tbl.n_comb : only + 1); ++combo) {
      const int n = static_cast<int>(sh.state[combo]);
      const int lo = only < 0 ? max(i_begin, first) - first : static_cast<int>(sh.krem[0]);
      const int hi = only < 0 ? min(i_end, first + n) - first : static_cast<int>(sh.krem[1]);
      if (lo < hi) rank_range(p, tbl, combo, n, lo, hi, sh.mode[combo] != 0, chunk, &sh);
      first += n;
    }
  }
  if (!grid_sync<kCluster>(p, &sh, epoch)) return;

  // ---- F: allocation and ascending output (one CTA); the others write the scores if asked ----
  if (p.user_scores && (blockIdx.x != 0 || gridDim.x == 1)) {
    const long long writers = gridDim.x == 1 ? 1 : gridDim.x - 1, mine = gridDim.x == 1 ? 0 : blockIdx.x - 1;
#pragma unroll 1
    for (long long t = mine * kSelThreads + threadIdx.x; t < p.L; t += writers * kSelThreads)
      p.user_scores[t] = score_at(p, t);
  }
  if (blockIdx.x != 0) return;
  if (p.bitmap_in_smem) {
    allocate<true>(tbl, p, dyn_smem, &sh);
  } else {
    allocate<false>(tbl, p, dyn_smem, &sh);
  }
}

// ---------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------
cudaError_t select_max_grid(int n_sm, int* max_grid, bool* wide_cluster) {
  cudaError_t e = cudaFuncSetAttribute(select_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kSelMaxDynSmemBytes);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(select_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           kSelMaxDynSmemBytes);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, select_kernel<false>, kSelThreads,
                                                    kSelMaxDynSmemBytes);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorLaunchOutOfResources;
  *max_grid = n_sm;                      // one CTA per SM is plenty for these phases
  // A cluster of more than 8 CTAs is the device's to grant.  The answer is kept, since asking takes 0.2 ms.
  const bool allowed = n_sm > kSelClusterWide &&
      cudaFuncSetAttribute(select_kernel<true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
  static std::atomic<int> granted[64];             // per device: 0 not asked yet, 1 no, 2 yes
  int dev = 0;
  e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  int known = dev < 64 ? granted[dev].load() : 0;
  if (known == 0) {
    int n = 0;
    if (allowed) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(kSelClusterWide);
      cfg.blockDim = dim3(kSelThreads);
      cfg.dynamicSmemBytes = kSelMaxDynSmemBytes;
      cudaLaunchAttribute attr;
      attr.id = cudaLaunchAttributeClusterDimension;
      attr.val.clusterDim.x = kSelClusterWide;
      attr.val.clusterDim.y = 1;
      attr.val.clusterDim.z = 1;
      cfg.attrs = &attr;
      cfg.numAttrs = 1;
      if (cudaOccupancyMaxActiveClusters(&n, select_kernel<true>, &cfg) != cudaSuccess) n = 0;
    }
    known = n > 0 ? 2 : 1;
    if (dev < 64) granted[dev].store(known);
  }
  *wide_cluster = allowed && known == 2;
  cudaGetLastError();
  return cudaSuccess;
}

// Deals the CTAs of the grid out to the combinations for the ranking phase: each list gets
// its share of the grid by candidates, at least one CTA, never past what the lists after it
// still need.  With fewer CTAs than lists the kernel splits the candidates evenly instead.
static void assign_ranking(ComboTable* t, int grid) {
  long long n_cand = 0;
  int n_lists = 0;
  for (int c = 0; c < t->n_comb; ++c) {
    n_cand += t->k_m[c];
    n_lists += t->k_m[c] > 0 ? 1 : 0;
  }
  t->rank_by_list = (n_lists > 0 && grid >= n_lists) ? 1 : 0;
  long long before = 0;
  int b0 = 0, lists_left = n_lists;
  for (int c = 0; c < t->n_comb; ++c) {
    t->rank_cta_begin[c] = b0;
    if (!t->rank_by_list || t->k_m[c] <= 0) continue;
    --lists_left;
    before += t->k_m[c];
    int b1 = static_cast<int>((before * grid + n_cand / 2) / n_cand);
    if (b1 < b0 + 1) b1 = b0 + 1;
    if (b1 > grid - lists_left) b1 = grid - lists_left;
    if (lists_left == 0) b1 = grid;
    b0 = b1;
  }
  t->rank_cta_begin[t->n_comb] = b0;
}

cudaError_t launch_select(const ComboTable& table, const SelectParams& p, int grid, size_t smem,
                          cudaStream_t st) {
  ComboTable tbl = table;
  assign_pooling(&tbl, grid);
  assign_ranking(&tbl, grid);
  // Short contexts need few CTAs: up to kSelClusterMax of them, or kSelClusterWide, run as one thread-block cluster,
  // whose hardware barrier costs a fraction of a trip to the L2 (not with the self test's
  // barrier that cannot complete: that one is the counter's).  Longer ones: a cooperative
  // launch (every CTA resident: they wait on one another).  Either way the launch may overlap
  // the end of the kernel before it in the stream; the kernel waits before it reads anything.
  const bool cluster = p.cluster != 0 && p.barrier_extra == 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kSelThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  if (cluster) {
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = grid;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
  } else {
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
  }
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cluster ? cudaLaunchKernelEx(&cfg, select_kernel<true>, tbl, p)
                 : cudaLaunchKernelEx(&cfg, select_kernel<false>, tbl, p);
}

}  // namespace ilre
