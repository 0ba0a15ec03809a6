// How the two passes over the key cache are split over the SMs (host side).
#pragma once
#include "qk_kernels.cuh"

namespace ilre {

static constexpr int kPairMinRows = 192;   // query rows per kv head above which the paired scores pass is used
static constexpr int kTailMinTiles = 14;   // key tiles per CTA from which short row tiles are loaded in copies
static constexpr int kPairMinTiles = 32;   // accumulators per CTA pair from which the paired scores pass is used

struct PassGeometry {
  int pair, n_rb, rb_rows, n_groups, cpg, n_tiles, stages;
};
struct Geometry {
  int group_size, kv_rows;             // kv_rows: rows of one kv head in the packed query
  PassGeometry stats, scores;
  bool stats_tail;                     // statistics: the last row tile of a full block is short; short ones are loaded in copies
};

// Splits the rows of one kv head into blocks of at most max_rows, padded to a multiple of `unit`.
inline void split_rows(int rows, int max_rows, int unit, PassGeometry* g) {
  g->n_rb = (rows + max_rows - 1) / max_rows;
  const int per = (rows + g->n_rb - 1) / g->n_rb;
  g->rb_rows = ((per + unit - 1) / unit) * unit;
}

// Upper bound of the packed rows of one kv head, for any query of up to q_len tokens.
inline int rows_padded_bound(int group_size, int q_len) {
  const long long rg = static_cast<long long>(group_size) * q_len;
  const long long n_rb = (rg + kMaxRbRows - 1) / kMaxRbRows, n_pair = (rg + kMaxPairRows - 1) / kMaxPairRows;
  const long long stats = 128 * (n_rb + 1), pair = 256 * (n_pair + 1);     // paddings
  return static_cast<int>(rg + (stats > pair ? stats : pair));
}

inline Geometry make_geometry(int n_kv_heads, int n_q_heads, int n_sm, long long L, int q_len) {
  Geometry g;
  g.group_size = n_q_heads / n_kv_heads;
  const int rg = g.group_size * q_len;
  auto padded = [](int rows) { return (rows + 127) & ~127; };          // a query tile in shared memory has 128 rows
  auto finish = [&](PassGeometry* p, int tile_keys, int workers) {
    p->n_groups = n_kv_heads * p->n_rb;
    p->n_tiles = static_cast<int>((L + tile_keys - 1) / tile_keys);
    p->cpg = workers / p->n_groups;
    if (p->cpg < 1) p->cpg = 1;
    if (p->cpg > p->n_tiles) p->cpg = p->n_tiles;
    const long long fixed = static_cast<long long>(padded(p->rb_rows)) * 256 + kSmemTailBytes +
                            static_cast<long long>(padded(p->rb_rows)) * 4;
    p->stages = static_cast<int>((kMaxDynSmem - fixed) / kStageBytes);
    if (p->stages > kMaxStages) p->stages = kMaxStages;
  };
  // Statistics: where blocks of even size to 32 rows, instead of to 128, end in a tile short enough for copies
  // (stats_tail_copies), they do, behind a full one and from kTailMinTiles key tiles per CTA on.  Statistics pass
  // after an L2 flush, without / with copies, us: 148 rows, 8K keys 17.7 / 18.6, 16K 22.2 / 22.8, 32K (14 tiles per
  // CTA) 30.4 / 29.1, 128K 81.2 / 72.2, 1M 521 / 468; 276 rows, 16K 27.1 / 29.1, 32K 39.3 / 39.5, 128K
  // 117 / 106; 540 rows, 16K 39.3 / 37.1, 128K 209 / 187; 800 rows, 128K 268 / 256; one tile of 64 rows, 32K
  // 25.8 / 26.9, 1M 338 / 349 (bound by the key stream).
  g.stats.pair = 0;
  split_rows(rg, kMaxRbRows, stats_box_rows(g.group_size), &g.stats);
  finish(&g.stats, kTileKeys, n_sm);
  g.stats_tail = stats_box_rows(g.group_size) == 32 && rg > 128 && stats_tail_copies(rg < g.stats.rb_rows ? rg : g.stats.rb_rows) > 1 &&
                 g.stats.n_tiles >= kTailMinTiles * g.stats.cpg;
  if (!g.stats_tail) {
    split_rows(rg, kMaxRbRows, 128, &g.stats);
    finish(&g.stats, kTileKeys, n_sm);
  }
  PassGeometry single;
  single.pair = 0;
  split_rows(rg, kMaxRbRows, 128, &single);
  finish(&single, kTileKeys, n_sm);
  // Scores by CTA pairs, which pad the rows of a kv head to a multiple of 256 (single CTAs: to 32), where
  // there are more than kPairMinRows rows, and where a pair has at least kPairMinTiles accumulators to
  // compute, which pay for the cluster launch.  Scores pass, pairs / single CTAs, us:
  //   rows, 128K keys: 148: 53.4 / 49.0; 192: 53.5 / 50.0; 256: 53.7 / 56.1; 280: 93.7 / 100.6;
  //   400: 94.6 / 101.7; 560: 129.7 / 194.8; 800: 169 / 189 (a second tile of few rows starves the two
  //   issuing threads of the single form); L = 1M, 1024 rows: 1414 / 1568 (single calls).
  //   accumulators: 57 (32K keys, 1024 rows) 55.2 / 56.4; 28 (32K, 512) 37.9 / 37.7; 14 (8K, 1024)
  //   24.4 / 23.4.
  PassGeometry pair;
  split_rows(rg, kMaxPairRows, 256, &pair);
  pair.pair = 1;
  finish(&pair, kPairTileKeys, n_sm / 2);
  pair.stages = 2;                       // the launcher sizes the ring
  const long long accumulators = static_cast<long long>(pair.n_tiles) * (pair.rb_rows / 256);
  const bool use_pair = rg > kPairMinRows && accumulators >= static_cast<long long>(kPairMinTiles) * pair.cpg;
  g.scores = use_pair ? pair : single;
  const int a = (g.stats.n_rb - 1) * g.stats.rb_rows + padded(g.stats.rb_rows), b = g.scores.n_rb * g.scores.rb_rows;
  g.kv_rows = a > b ? a : b;
  return g;
}

}  // namespace ilre
