// Parameters and launchers of the query-context attention kernels (Eq. 4, Eq. 5).
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace ilre {

static constexpr int kHeadDim = 128;
static constexpr int kTileKeys = 128;              // keys per K tile (one TMA stage)
static constexpr int kStageBytes = kTileKeys * kHeadDim * 2;
static constexpr int kMaxStages = 6;
static constexpr int kMaxRbRows = 512;             // query rows resident in shared memory
static constexpr int kQkThreads = 384;             // scores: warp 0 TMA, warps 1-2 MMA, warps 4..11 consumers
static constexpr int kConsumerWarps = 8;
// Row statistics: warp 0 TMA, warp 1 MMA, kStatsWarpgroups consumer warpgroups of four
// warps (one per TMEM lane quadrant), perhaps a second MMA warp; accumulator buffer u belongs to warpgroup
// u % kStatsWarpgroups.
static constexpr int kStatsWarpgroups = 4;
// A warpgroup's first accumulator must be one of the first four (the number of TMEM buffers):
// a parity wait on a buffer that has not completed its first phase yet would pass at once.
static_assert(kStatsWarpgroups >= 1 && kStatsWarpgroups <= 4, "at most one warpgroup per TMEM buffer");
static constexpr int kStatsConsumerWarps = 4 * kStatsWarpgroups;
// Issuing threads (warp 1 and the warp after the consumers): one with a single row tile, where the key
// tiles arrive more slowly than one thread issues (a second one: 4K keys 10.8 -> 12.1 us).
template <int MT> constexpr int kStatsIssuers = MT > 1 ? 2 : 1;
template <int MT> constexpr int kStatsThreads = 32 * (1 + kStatsIssuers<MT> + kStatsConsumerWarps);
static constexpr int kSmemTailBytes = 256;
static constexpr int kMaxDynSmem = 232448;         // 227 KB per CTA on sm_100
// Paired scores pass: two CTAs of a cluster share every tensor-core tile of 256 keys x 256 rows.
static constexpr int kPairTileKeys = 256;          // keys per key tile, 128 in each CTA
static constexpr int kUnitBytes = kTileKeys * 64 * 2;    // ring unit: 128 keys x 64 channels
static constexpr int kMaxUnits = 12;
static constexpr int kMaxPairRows = 1024;          // query rows resident in a pair
static constexpr int kPairConsumerWarps = 16;
static constexpr int kPairThreads = 640;           // warp 0 TMA, warps 1-2 MMA, warps 4..19 consumers

// Row statistics: how many of every 16 logit pairs take 2^x from the FMA-pipe polynomial
// instead of the special-function unit (0 = none).  Balances the two pipes.
static constexpr int kRowStatsPolyPairs = 4;

// Scores by single CTAs: row halves of 256 (accumulators per key tile) of row block `block`, whose rows past
// those of its kv head are left out, in steps of 32.
__host__ __device__ constexpr int scores_block_rows(int rb_rows, int rows_per_kv, int block) {
  const int left = rows_per_kv - block * rb_rows;
  return ((left < rb_rows ? left : rb_rows) + 31) & ~31;
}
__host__ __device__ constexpr int scores_row_halves(int block_rows) { return (block_rows + 255) / 256; }
// ... and the stages of the ring that such a block uses.  With one row half the two issuing threads take the
// key tiles in turn.  A parity wait is only sound for a thread that has seen the stage's phase before, so
// there a stage must always meet the same thread: an even ring.  A last block of few rows beside full
// ones, whose ring may be odd, has at most half of their work, so the stage it gives up costs nothing
// (1190 rows per kv head, 16384 keys: 29.4 us; all blocks with two row halves and three stages 29.1).
__host__ __device__ constexpr int scores_ring_stages(int stages, int row_halves) {
  return row_halves == 1 ? stages & ~1 : stages;
}

// Statistics pass: copies of the rows of a block's last live row tile.  A tile's rows lie in the four lane
// quadrants of tensor memory, each read by the warps of one scheduler: 20 rows are one scheduler's work, as long
// as 128 rows are, while the others wait.  So a tile of up to 32 rows is loaded four times, one of up to
// 64 twice, and each copy takes its share of the key tile's columns (148 rows, 1M keys: 521 -> 468 us).
__host__ __device__ constexpr int stats_tail_rows(int live_rows) { return (live_rows - 1) % 128 + 1; }
__host__ __device__ constexpr int stats_tail_copies(int live_rows) {
  return stats_tail_rows(live_rows) <= 32 ? 4 : stats_tail_rows(live_rows) <= 64 ? 2 : 1;
}
// Rows that a TMA box collects for such a tile: those of whole tokens.  (Head groups of more than 32: no copies.)
__host__ __device__ constexpr int stats_box_rows(int group_size) {
  return 128 % group_size == 0 && group_size > 32 ? 128 : 32;
}

// Geometry of one pass.
struct QkParams {
  long long L;
  int pair;          // 1: scores by CTA pairs
  int n_tiles;       // key tiles of kTileKeys keys (pair: of kPairTileKeys)
  int n_groups;      // n_kv_heads * n_rb
  int n_rb;          // row blocks per kv head
  int rb_rows;       // rows per block: multiple of 128 up to kMaxRbRows (statistics: of 32; pair: of 256 up to
                     // kMaxPairRows)
  int kv_rows;       // rows of one kv head in the packed query (>= n_rb * rb_rows)
  int rows_per_kv;   // those that are not padding
  int group;         // query heads per kv head when the query is loaded from the caller's array (a
                     // box of 128 rows = `group` heads of 128 / group tokens); 0: from the packed copy
  int cpg;           // key chunks (CTAs or CTA pairs) per group
  int tail;          // statistics: a block's last row tile is loaded in copies where it is short (stats_tail_copies)
  int stages;        // ring depth in key tiles (pair: in units, set by the launcher)
  float c2;          // log2(e) / sqrt(d)
  float* partial;    // [n_groups][cpg][rb_rows][2]: (max * c2, sum-exp) per key chunk
  uint32_t* enc;     // [L]: order-preserving uint of max_r log2 p_rt
  int* status;
  // When non-null, CTA 0 of the row-statistics kernel stores how long it ran in SM cycles and
  // in nanoseconds of the global timer: their ratio is the SM clock the kernel really ran at
  // (under the power cap it is well below what the driver reports).
  unsigned long long* clk;
  // Failure-detection self test (see ilre_recall_selftest_wait): spin budget of the
  // row-statistics kernel's waits in SM cycles, and how many of its last key tiles the
  // producer leaves out (0 in normal operation).
  long long wait_limit;
  int skip_tiles;
};

struct PrepParams {
  int n_kv, n_q, group_size, q_len, kv_rows;   // kv_rows = 0: no query to pack
  int clear;                // the state of the run is to be cleared
  long long L;
  int n_sink;
  uint32_t* enc;
  uint32_t* bitmap;
  uint32_t* hist;
  long long hist_words;     // words of the radix histograms to clear
  uint32_t* cand_count;     // per-run state words of the selection kernel, cleared here
  int sel_state_words;
  uint32_t* grid_barrier;   // arrival counter of the selection kernel's grid barrier
};

struct MergeParams {
  int n_kv, n_rb, rb_rows, cpg, group_size, q_len, n_q;    // n_rb, rb_rows, cpg: the statistics pass's
  const float* partial;
  float* row_lse;    // [q_len][n_q] natural-log lse
  // Key-range sharding: when n_ext > 0 the statistics come from ext_stats
  // [n_ext][q_len * n_q] (max in log2 units, sum) -- one entry per shard, rows in the
  // caller's order i * n_q + h -- instead of this launch's own partials.
  const float2* ext_stats;
  int n_ext;
};

size_t row_stats_smem_bytes(int rb_rows, int stages);
size_t scores_smem_bytes(int rb_rows, int stages);

cudaError_t launch_prepare(const void* q, void* qp, const PrepParams& p, int n_sm, cudaStream_t st);
// Where no prepare kernel was launched before it, this one clears the run's state (pp.clear).
// tq32: the query in boxes of 32 rows, read with p.tail.
cudaError_t launch_row_stats(const CUtensorMap& tk, const CUtensorMap& tq, const CUtensorMap& tq32, const QkParams& p,
                             const PrepParams& pp, cudaStream_t st);
// (max in log2 units, sum of exponentials) of every query row over the keys of this launch,
// rows in the caller's order i * n_q + h.
cudaError_t launch_export_stats(const MergeParams& p, float2* out, cudaStream_t st);
// out[t] = exp2 of the encoded maxima (the scores of Eq. 5 for a key shard)
cudaError_t launch_decode_scores(const uint32_t* enc, float* out, long long L, cudaStream_t st);
cudaError_t launch_scores(const CUtensorMap& tk, const CUtensorMap& tq, const QkParams& p,
                          const MergeParams& mp, cudaStream_t st);

}  // namespace ilre
