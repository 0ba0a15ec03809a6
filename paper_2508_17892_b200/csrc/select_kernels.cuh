// Parameters and launcher of the Algorithm 1 kernel: pooling, ranked top-K_m per combination,
// quota allocation with de-duplication, ascending output.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <cstring>

namespace ilre {

static constexpr int kMaxCombos = 64;
static constexpr int kHistBins = 2048;
// Histogram bins of the pooled values, from their bit patterns (values below zero: the first bin).
// Probabilities from the scores pass: 32 bins per power of two from 2^-63 to 2.  Given scores may have any
// scale: 32 per power of two from 2^-35, below which hardly a selected probability lies, to 2^8, 2 below and
// 4 above.  (With the first rule log-normal scores scaled to 1e4 all share a bin: allocation of 131072
// positions 77 us, so 48; with 4 bins from 2 on, 32768 raw logits 72, so 40; with 8 bins per power of two
// throughout, one rank's part of a sharded recall of 1M tokens 620 us, so 600.)
static constexpr int kFineExponent = 92, kFineEnd = 135;      // biased exponents of 2^-35 and of 2^8
static constexpr int kFineBin = 2 * kFineExponent, kCoarseBin = kFineBin + 32 * (kFineEnd - kFineExponent);
static_assert(kCoarseBin + 4 * (255 - kFineEnd) < kHistBins, "infinity has a bin of its own");
__host__ __device__ constexpr int bin_of_bits(int bits, bool given) {
  const int u = bits < 0 ? 0 : bits;
  if (!given) {
    const int b = (u >> 18) - (64 << 5);
    return b < 0 ? 0 : b < kHistBins ? b : kHistBins - 1;
  }
  return u < (kFineExponent << 23) ? u >> 22
       : u < (kFineEnd << 23) ? (u >> 18) - (kFineExponent << 5) + kFineBin : (u >> 21) - (kFineEnd << 2) + kCoarseBin;
}
// Bit pattern of the lowest value of bin b > 0.
__host__ __device__ constexpr int bin_floor_bits(int b, bool given) {
  if (!given) return (b + (64 << 5)) << 18;
  return b < kFineBin ? b << 22
       : b < kCoarseBin ? (b - kFineBin + (kFineExponent << 5)) << 18 : (b - kCoarseBin + (kFineEnd << 2)) << 21;
}
// The last bin with values of a first digit of the long way (the upper 11 of a positive value's 32 key bits).
__host__ __device__ constexpr int last_bin_of_digit(int digit, bool given) {
  return bin_of_bits(((digit & 0x3FF) << 21) | 0x1FFFFF, given);
}
// That digit of all values of bin b; -1: the bin, or the digit's last one, holds several.
__host__ __device__ constexpr int bin_digit(int b, bool given) {
  const int digit = (bin_floor_bits(b, given) >> 21) | 0x400;
  return b == 0 || (given && b < kFineBin) || last_bin_of_digit(digit, given) == kHistBins - 1 ? -1 : digit;
}
static constexpr int kMaxWin = 1024;        // largest stride-1 window size
static constexpr int kMaxMaxSize = 64;      // largest strided max-pool size
static constexpr int kMaxKm = 16384;        // largest K_m (bounds the candidate lists)
static constexpr int kSelectPasses = 3;     // long way: 32 value bits of the key in 11/11/10-bit digits
static constexpr int kSelThreads = 1024;    // threads per CTA of the selection kernel
static constexpr int kSelTile = 4096;       // cells of one combination per work tile of the gather
static constexpr int kPoolGroup = 5;        // window sizes of one strided max-pool that are pooled together
static constexpr int kPoolTileMax = 3072;   // cells of a group of windows per work tile, at most
static constexpr int kSrcTileTokens = 8192; // tokens per work tile of the strided max-pool
static constexpr int kSelClusterMax = 8;     // grids up to this size run as one thread-block cluster
static constexpr int kSelClusterWide = 16;   // and those of this size where select_grid says so
static constexpr int kCandSlack = 4096;      // candidates past K_m that the threshold bin may bring
static constexpr int kWalkCells = 4;         // ranked cells per thread and round of the quota walk
static constexpr int kMinWalkers = 64;       // fewest threads that walk
static constexpr int kSelBitmapSmemBytes = 136 * 1024;   // bitmap kept in shared memory up to this
static constexpr int kSelBitmapSlackWords = 4;           // behind the bitmap
// Work area in front of the bitmap: pooling tiles, the keys of a ranking list and the list of the output
// pass, one after another.
static constexpr int kSelWorkBytes = 64 * 1024;
static_assert(kSelWorkBytes >= (kPoolGroup - 1) * kHistBins * 4 + 2 * (kPoolTileMax + kMaxWin) * 4 && kSelWorkBytes >= kSrcTileTokens * 4,
              "work area too small");
static constexpr int kSelMaxDynSmemBytes = kSelWorkBytes + kSelBitmapSmemBytes + 4 * kSelBitmapSlackWords;

// One entry per (m_i, n_j) combination, in Algorithm 1's loop order.
struct ComboTable {
  int n_comb;
  int m[kMaxCombos];       // strided max-pool size
  int n[kMaxCombos];       // window size
  int len[kMaxCombos];     // number of cells = ceil((L - n_sink) / m)
  int k_m[kMaxCombos];     // candidates ranked for this combination
  int quota[kMaxCombos];   // B_c
  int tile_begin[kMaxCombos + 1];   // first work tile of each combination (prefix sums)
  // Distinct strided max-pool sizes m > 1 ("sources"): their pooled arrays are computed once
  // and shared by every window size.  src[c] = source of combination c, -1 = the scores.
  int n_src;
  int src[kMaxCombos];
  int src_m[kMaxCombos];
  int src_len[kMaxCombos];
  int src_tile_begin[kMaxCombos + 1];   // tiles of kSrcTileTokens / m cells each
  // Groups of combinations of one source (up to kPoolGroup, ascending window sizes) that are pooled
  // together, and their work tiles of pool_tile cells (filled in by assign_pooling).
  int n_grp, pool_tile;
  int grp_first[kMaxCombos + 1];        // first entry of each group in grp_combo
  int grp_combo[kMaxCombos];
  int grp_tile_begin[kMaxCombos + 1];
  // Ranking phase (filled in by launch_select): with rank_by_list, combination c is ranked by
  // the CTAs [rank_cta_begin[c], rank_cta_begin[c + 1]).
  int rank_by_list;
  int rank_cta_begin[kMaxCombos + 1];
};

// Of a combination's cells, those from `first` on, at most `most`.  (Lengths go up to 2^31 - 257: the end of a work tile
// may not fit an int, and where a cell lies in its tile is compared instead.)
__host__ __device__ constexpr int cells_from(int len, int first, int most) { return len - first < most ? len - first : most; }

// The combinations of Algorithm 1 in its loop order (max sizes outer, window sizes inner) over Lp positions.
inline void make_combinations(long long Lp, int budget, const int32_t* max_sizes, int n_max, const int32_t* win_sizes,
                              int n_win, ComboTable* t) {
  std::memset(t, 0, sizeof(*t));
  t->n_comb = (budget > 0) ? n_max * n_win : 0;
  long long allocated_before = 0;
  for (int i = 0, c = 0; i < n_max && t->n_comb; ++i)
    for (int j = 0; j < n_win; ++j, ++c) {
      const int m = max_sizes[i];
      const long long len = (Lp + m - 1) / m;
      long long km = budget / m + 1 + ((Lp % m) != 0 ? 1 : 0);
      if (km > len) km = len;
      t->m[c] = m;
      t->n[c] = win_sizes[j];
      t->len[c] = static_cast<int>(len);
      t->quota[c] = budget / t->n_comb + (c < budget % t->n_comb ? 1 : 0);
      // Algorithm 1 ranks K_m cells, but the quota walk of this combination cannot go further
      // than quota cells that bring a new token plus the cells made up entirely of tokens the
      // earlier combinations took (at most allocated / m full cells and the partial tail
      // cell).  Ranking only that many gives the same walk and, for all but the last
      // combinations, far fewer candidates to select and order.
      long long reach = t->quota[c] + allocated_before / m + ((Lp % m) != 0 ? 1 : 0);
      if (reach < 1) reach = 1;
      if (km > reach) km = reach;
      t->k_m[c] = static_cast<int>(km);
      allocated_before += t->quota[c];
      t->tile_begin[c + 1] = t->tile_begin[c] + static_cast<int>((len + kSelTile - 1) / kSelTile);
      // the strided max-pool of size m is shared by all window sizes
      t->src[c] = -1;
      if (m > 1) {
        int s = 0;
        while (s < t->n_src && t->src_m[s] != m) ++s;
        if (s == t->n_src) {
          const int cells_per_tile = kSrcTileTokens / m;
          t->src_m[s] = m;
          t->src_len[s] = static_cast<int>(len);
          t->src_tile_begin[s + 1] =
              t->src_tile_begin[s] + static_cast<int>((len + cells_per_tile - 1) / cells_per_tile);
          ++t->n_src;
        }
        t->src[c] = s;
      }
    }
}

// Groups the combinations for the pooling phase and cuts the groups into tiles: equal shares of the
// grid's CTAs, rounded up to whole warps.
inline void assign_pooling(ComboTable* t, int grid) {
  t->n_grp = 0;
  int n = 0;
  long long cells = 0;
  for (int src = -1; src < t->n_src; ++src) {
    int list[kMaxCombos], cnt = 0;
    for (int c = 0; c < t->n_comb; ++c)
      if (t->src[c] == src) list[cnt++] = c;
    for (int i = 1; i < cnt; ++i)                           // by window size
      for (int j = i; j > 0 && t->n[list[j]] < t->n[list[j - 1]]; --j) {
        const int x = list[j]; list[j] = list[j - 1]; list[j - 1] = x;
      }
    const int n_groups = (cnt + kPoolGroup - 1) / kPoolGroup;
    for (int g = 0; g < n_groups; ++g) {                    // groups of even size
      t->grp_first[t->n_grp++] = n;
      for (int i = g * cnt / n_groups; i < (g + 1) * cnt / n_groups; ++i) t->grp_combo[n++] = list[i];
      cells += t->len[list[0]];
    }
  }
  t->grp_first[t->n_grp] = n;
  const long long rounds = (cells + static_cast<long long>(grid) * kPoolTileMax - 1) / (static_cast<long long>(grid) * kPoolTileMax);
  const long long workers = static_cast<long long>(grid) * (rounds < 1 ? 1 : rounds);
  long long tile = ((cells + workers - 1) / workers + 31) & ~31ll;
  t->pool_tile = static_cast<int>(tile < 256 ? 256 : (tile > kPoolTileMax ? kPoolTileMax : tile));
  t->grp_tile_begin[0] = 0;
  for (int g = 0; g < t->n_grp; ++g)
    t->grp_tile_begin[g + 1] = t->grp_tile_begin[g] +
        static_cast<int>((static_cast<long long>(t->len[t->grp_combo[t->grp_first[g]]]) + t->pool_tile - 1) / t->pool_tile);
}

struct SelectParams {
  const uint32_t* enc;     // [L] order-preserving uint of max_r log2 p_rt (scores pass output)
  const float* scores;     // A^C [L], with scores_given
  float* user_scores;      // A^C [L] for the caller, or null
  int scores_given;        // 1: `scores` holds A^C (else it comes from `enc`)
  long long L;
  int n_sink;
  int win_op;              // 0 average, 1 max
  float* maxpooled;        // [n_src][maxpooled_stride] strided max-pool of the scores
  long long maxpooled_stride;
  float* pooled;           // [n_comb][pooled_stride]
  long long pooled_stride;
  uint32_t* hist;          // [2 + kSelectPasses][n_comb][kHistBins]: values per bin and candidates placed per
                           // bin, zero on entry; then the passes of the long way
  int* tile_ties;          // [work tiles]: cells of a tile that hold the K_m-th value
  unsigned long long* cand;   // [n_comb][cand_stride] 64-bit keys of the candidates, sorted by bin
  uint32_t* cand_seg;      // [n_comb][cand_stride] start | length << 16 of a candidate's bin
  int cand_stride;         // at least K_m + kCandSlack, a multiple of 4, below 2^16
  uint32_t* cand_count;    // [4 * kMaxCombos]: candidates gathered per combination; then, at
                           // kMaxCombos, whether the combination took the long way, and at
                           // 3 kMaxCombos two flag words (some combination did; one of them takes
                           // all passes); zero on entry
  int* ranked;             // [n_comb][cand_stride] cell ids in rank order (cand_stride: multiple of 4)
  uint32_t* bitmap;        // [ceil(L/32)] in global memory, used when it does not fit shared memory
  int bitmap_in_smem;
  int cluster;             // the grid runs as one thread-block cluster
  int walk_threads;        // threads that walk the combinations in the allocation phase
  int* out_idx;            // [n_sink + budget]
  int budget;
  uint32_t* barrier;       // grid barrier arrival counter, zero when the kernel starts
  int* status;
  // Failure-detection self test (see ilre_recall_selftest_wait): spin budget of a grid
  // barrier in SM cycles, and how many CTAs more than the grid has the barrier waits for
  // (0 in normal operation).
  long long wait_limit;
  int barrier_extra;
};

// Dynamic shared memory the kernel needs for a context of L positions.  Also fills p->bitmap_in_smem and p->walk_threads.
inline size_t select_smem_bytes(long long L, int max_km, SelectParams* p) {
  // the bitmap, when it fits, lies behind the work area
  const size_t words = (static_cast<size_t>((L + 31) / 32) + 3) & ~size_t(3);
  p->bitmap_in_smem = words * sizeof(uint32_t) <= static_cast<size_t>(kSelBitmapSmemBytes) ? 1 : 0;
  int walkers = ((max_km + kWalkCells - 1) / kWalkCells + 31) & ~31;
  p->walk_threads = walkers < kMinWalkers ? kMinWalkers : (walkers > kSelThreads ? kSelThreads : walkers);
  return kSelWorkBytes + (p->bitmap_in_smem ? (words + kSelBitmapSlackWords) * sizeof(uint32_t) : 0);
}
// Grid of the selection kernel.
struct SelectGrid {
  int ctas;
  bool cluster;            // one thread-block cluster, else a cooperative grid
};

// Enough CTAs for the scan tiles and for the ranking (about a hundred candidates per CTA), but no more, since every
// barrier pays for them.  Up to kSelClusterMax CTAs, or kSelClusterWide where the device grants that, run as one
// thread-block cluster: it starts under the end of the scores pass, and its barriers cost half of the counter's, which a
// larger cooperative grid gains back on many cells, many candidates to rank, or many combinations.  Whole recalls in a
// row (16 query tokens), us, cluster of 8 / cluster of 16 / cooperative (of 16, or of as many as are worth having):
//   9 to 16 CTAs worth having: 3 windows, budget 512: 4K positions 29.3 / 29.2 / 32.9, 8K 31.6 / 31.2 / 34.5, 16K 39.1 / 35.4 /
//   39.0, 20K 41.6 / 37.9 / 41.1; 5 windows 12K 42.1 / 37.6 / 40.8; 12 combinations (m = 1, 2, 4), 4K 50.3 / 42.6 / 46.8
//   the same on fewer than 12288 cells: 2301 positions, 5 windows 43.4 / 44.4 / --, 2060, 3 windows 43.5 / 44.2 / --; but with more
//   lists to rank than 8 CTAs: 1000 positions, 12 combinations 42.6 / 35.3 / 39.1
//   more: 3 windows, 24K positions, budget 512 44.3 / 40.7 / 43.6, 2048 48.6 / 44.1 / 45.1; 32K, 512 52.0 / 47.0 / 48.0; 40K
//   60.4 / 54.2 / 53.9; one window, budget 2048, 8K 31.3 / 30.7 / 33.2, 40K 53.8 / 50.1 / 53.4
//   more candidates than 5120: 3 windows, budget 4096, 12K 47.9 / 44.0 / 41.4; 5 windows, budget 2048, 6K 48.4 / 44.0 / 39.0
inline SelectGrid select_grid(const ComboTable& t, int max_ctas, bool wide_granted) {
  long long cells = 0, cand = 0;
  for (int c = 0; c < t.n_comb; ++c) { cells += t.len[c]; cand += t.k_m[c]; }
  long long want = t.tile_begin[t.n_comb];
  if (cand / 96 > want) want = cand / 96;
  if (want < 1) want = 1;
  if (want > kSelClusterMax && want <= kSelClusterWide)
    want = wide_granted && (cells >= 12288 || t.n_comb > kSelClusterMax) ? kSelClusterWide : kSelClusterMax;
  else if (want > kSelClusterWide && wide_granted && t.n_comb <= 8 && cand <= 5120 && cells + 5 * cand <= 95000)
    want = kSelClusterWide;
  if (want > max_ctas) want = max_ctas;
  return {static_cast<int>(want), want <= kSelClusterMax || (want == kSelClusterWide && wide_granted)};
}
// Largest grid that is co-resident on the device (the kernel's CTAs wait on one another), and whether it takes a
// cluster of kSelClusterWide CTAs.
cudaError_t select_max_grid(int n_sm, int* max_grid, bool* wide_cluster);
// One launch: A^C from the encoded maxima, then all of Algorithm 1.
cudaError_t launch_select(const ComboTable& tbl, const SelectParams& p, int grid, size_t smem,
                          cudaStream_t st);

}  // namespace ilre
