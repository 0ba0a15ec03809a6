"""Host-side launch rules, compiled from the library's headers with the host compiler and checked over
ranges of sizes.  No GPU."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2508_17892_b200", "csrc")
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


def _run(tmp_path, body, *flags):
    src, exe = tmp_path / "check.cpp", tmp_path / "check"
    src.write_text(body)
    subprocess.check_call(["g++", "-std=c++17", "-O1", *flags, "-I", CSRC, "-I", os.path.join(CUDA, "include"),
                           "-x", "c++", str(src), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout[-2000:]
    return r.stdout


RINGS = r"""
#include <cstdio>
#include <cstring>
#include "qk_geometry.cuh"
using namespace ilre;
int main() {
  const int heads[][2] = {{8, 32}, {4, 28}, {8, 64}, {2, 16}, {4, 16}, {1, 7}, {2, 8}, {7, 7}};
  const long long lengths[] = {1, 129, 1000, 4096, 9001, 16384, 24001, 49001, 131072, 1048576};
  long long blocks = 0, in_turn = 0, short_last = 0, bad = 0;
  for (const auto& h : heads)
    for (long long L : lengths)
      for (int q_len = 1; q_len <= 640; ++q_len) {
        const Geometry g = make_geometry(h[0], h[1], 148, L, q_len);
        if (g.scores.pair) continue;
        const int rows = g.group_size * q_len;
        int covered = 0;
        for (int b = 0; b < g.scores.n_rb; ++b, ++blocks) {
          const int block_rows = scores_block_rows(g.scores.rb_rows, rows, b);
          const int halves = scores_row_halves(block_rows);
          const int ring = scores_ring_stages(g.scores.stages, halves);
          covered += block_rows;
          bool ok = block_rows > 0 && block_rows <= g.scores.rb_rows && halves <= 2 && ring >= 2 &&
                    ring <= g.scores.stages;
          if (halves == 1) {             // tile i: issuing thread i % 2, stage i % ring
            ++in_turn;
            short_last += g.scores.rb_rows > 256;
            for (int i = 0; i < 4 * ring; ++i) ok = ok && ((i % ring) & 1) == (i & 1);
          }
          if (!ok && bad++ < 5)
            std::printf("heads %d/%d L %lld q_len %d block %d: %d rows, ring %d\n", h[0], h[1], L, q_len, b,
                        block_rows, ring);
        }
        if (covered < rows && bad++ < 5) std::printf("rows not covered: %d of %d\n", covered, rows);
      }
  std::printf("%lld blocks, %lld in turn, %lld of them short last blocks\n", blocks, in_turn, short_last);
  return bad || !in_turn || !short_last;
}
"""


def test_a_ring_stage_always_meets_the_same_issuing_thread(tmp_path):
    """Single-CTA scores pass: where the two issuing threads take the key tiles in turn, a stage must not
    change hands (a parity wait is only sound for a thread that has seen the phase before), in every
    row block of a launch: the last one may have few live rows beside full ones."""
    _run(tmp_path, RINGS)


WALK = r"""
#include <cstdio>
#include "select_kernels.cuh"
using namespace ilre;
int main() {
  int bad = 0;
  long long past_end = 0;
  for (long long L = 1; L <= 5000; L += (L < 1100 ? 1 : 97))
    for (int n_sink = 0; n_sink < 5 && n_sink < L; n_sink += 4) {
      SelectParams p;
      const size_t bytes = select_smem_bytes(L, 1, &p);
      const int Lp = static_cast<int>(L) - n_sink;
      if (!p.bitmap_in_smem || bytes > static_cast<size_t>(kSelMaxDynSmemBytes)) ++bad;
      for (int m = 1; m <= kMaxMaxSize; ++m) {
        int last = 0;                    // last bitmap word that the walk reads for any cell
        for (int t0 = 0; t0 < Lp; t0 += m) {
          const int w = (t0 >> 5) + (32 % m == 0 ? 0 : m <= 32 ? 1 : (t0 & 31) ? 2 : 1);
          last = w > last ? w : last;
        }
        past_end += last >= (L + 31) / 32;
        if (kSelWorkBytes + 4 * static_cast<size_t>(last + 1) > bytes && bad++ < 5)
          std::printf("L %lld sink %d m %d: word %d read, %zu bytes\n", L, n_sink, m, last, bytes);
      }
    }
  std::printf("%lld cases read past the bitmap\n", past_end);
  return bad || !past_end;
}
"""


def test_the_quota_walk_reads_inside_its_shared_memory(tmp_path):
    """A cell of more than 32 tokens is read as three bitmap words, the last of which may lie behind the
    bitmap: the launch asks for that memory too."""
    _run(tmp_path, WALK)


BINS = r"""
#include <cstdio>
#include <cstring>
#include "select_kernels.cuh"
using namespace ilre;
static int bits_of(float f) { int b; std::memcpy(&b, &f, 4); return b; }
int main() {
  int bad = 0;
  for (int given = 0; given < 2; ++given) {
    const bool r = given;
    const int last = bin_of_bits(0x7F800000, r);         // infinity
    bad += bin_of_bits(0, r) != 0 || bin_of_bits(bits_of(-0.0f), r) != 0 || bin_of_bits(bits_of(-3.0f), r) != 0;
    bad += last >= kHistBins || (given && last == kHistBins - 1);
    // a bin begins where the one before it ends
    for (int b = 1; b <= last; ++b)
      if (bin_of_bits(bin_floor_bits(b, r), r) != b || bin_of_bits(bin_floor_bits(b, r) - 1, r) != b - 1)
        if (bad++ < 5) std::printf("given %d: bin %d begins at %08x\n", given, b, bin_floor_bits(b, r));
    // a digit's bins hold that digit only, and none of it lies above the last of them
    for (int b = 0; b <= last; ++b) {
      const int digit = bin_digit(b, r);
      if (digit < 0) { bad += b != 0 && b >= (given ? kFineBin : 1) && (given || b < kHistBins - 8); continue; }
      const int top = last_bin_of_digit(digit, r);
      bad += top < b || bin_digit(top, r) != digit;
      bad += top < last && bin_digit(top + 1, r) == digit;
      const int end = top < kHistBins - 1 ? bin_floor_bits(top + 1, r) - 1 : 0x7F800000;
      bad += ((end >> 21) | 0x400) != digit;
    }
  }
  // 32 bins per power of two for probabilities
  float v = 1.0f;
  for (int e = 0; e < 62; ++e, v *= 0.5f)
    bad += bin_of_bits(bits_of(v), false) - bin_of_bits(bits_of(v * 0.5f), false) != 32;
  return bad;
}
"""


def test_histogram_bins_cover_every_value_in_order(tmp_path):
    _run(tmp_path, BINS)


LONGEST = r"""
#include <algorithm>
#include <cstdio>
#include <cstring>
#include "select_kernels.cuh"
using namespace ilre;
int main() {
  int bad = 0;
  for (long long L : {2147483647LL - 256, 2147483647LL - 256 - 2 * kPoolTileMax, 2147479553LL, 2147479552LL, 5000LL, 1LL})
    for (int m : {1, 2, 64})
      for (int grid : {1, 8, 148}) {
        ComboTable t;
        std::memset(&t, 0, sizeof(t));
        t.n_comb = 2;
        t.n_src = m > 1;
        const int len = static_cast<int>((L + m - 1) / m);
        for (int c = 0; c < 2; ++c) { t.m[c] = m; t.n[c] = c ? kMaxWin : 1; t.len[c] = len; t.src[c] = m > 1 ? 0 : -1; }
        assign_pooling(&t, grid);
        const long long end = static_cast<long long>(t.grp_tile_begin[1]) * t.pool_tile;
        bool ok = t.n_grp == 1 && t.pool_tile <= kPoolTileMax && end >= len && end - t.pool_tile < len;
        // the last tiles of the pooling and of the gather hold the last cell and nothing behind it
        for (int size : {t.pool_tile, kSelTile, kSelTile * 4}) {
          const int first = (len - 1) / size * size;
          ok = ok && first + static_cast<long long>(cells_from(len, first, size)) == len;
          ok = ok && (first == 0 || cells_from(len, first - size, size) == size);
        }
        // and of a tile with its margins, idx < cells_from(..) + margin are the cells of the context
        for (int c0 : {0, std::max(0, len - 1), std::max(0, len / 2)}) {
          const int span = std::min(t.pool_tile, len - c0) + kMaxWin - 1, margin = kMaxWin / 2;
          const long long inside = std::min<long long>(span, static_cast<long long>(len) - c0 + margin);
          ok = ok && std::min(span, cells_from(len, c0, span) + margin) == inside;
        }
        if (!ok && bad++ < 5) std::printf("L %lld m %d grid %d: tiles end at %lld\n", L, m, grid, end);
      }
  return bad;
}
"""


def test_tiles_of_the_longest_contexts_end_where_the_context_does(tmp_path):
    """Lengths go up to 2^31 - 257, where the end of a tile may not fit 32 bits with a sign."""
    _run(tmp_path, LONGEST, "-fsanitize=signed-integer-overflow", "-fno-sanitize-recover")


GRIDS = r"""
#include <cstdio>
#include "select_kernels.cuh"
using namespace ilre;
static SelectGrid grid_of(long long L, int budget, int n_max, const int32_t* max_sizes, int n_win, const int32_t* win_sizes,
                          int n_sink, bool granted, ComboTable* t) {
  make_combinations(L - n_sink, budget, max_sizes, n_max, win_sizes, n_win, t);
  return select_grid(*t, 148, granted);
}
int main() {
  int bad = 0;
  ComboTable t;
  // {L, budget, n_sink, number of max sizes, max sizes .., number of window sizes, window sizes ..}, one cluster of 16
  const int32_t wide[][32] = {%s};
  for (const auto& w : wide) {
    const int32_t* ms = w + 4;
    const int32_t* ws = ms + w[3] + 1;
    const SelectGrid g = grid_of(w[0], w[1], w[3], ms, ms[w[3]], ws, w[2], true, &t);
    const SelectGrid no = grid_of(w[0], w[1], w[3], ms, ms[w[3]], ws, w[2], false, &t);
    if ((!g.cluster || g.ctas != kSelClusterWide || (no.cluster && no.ctas > kSelClusterMax)) && bad++ < 5)
      std::printf("L %%d budget %%d: %%d CTAs, cluster %%d\n", w[0], w[1], g.ctas, g.cluster);
  }
  const int32_t sizes[] = {1, 2, 4, 8, 16, 32}, wins[] = {1, 3, 7, 9, 15, 31, 47, 63};
  int seen[4] = {0, 0, 0, 0};
  for (long long L = 1; L < 5000000; L += 1 + L / 7)
    for (int budget = 0; budget <= L && budget <= 16382; budget += 1 + budget)
      for (int n_max = 1; n_max <= 6; ++n_max)
        for (int n_win = 1; n_win <= 8; ++n_win)
          for (int granted = 0; granted < 2; ++granted) {
            const SelectGrid g = grid_of(L, budget, n_max, sizes, n_win, wins, 0, granted, &t);
            long long cand = 0;
            for (int c = 0; c < t.n_comb; ++c) cand += t.k_m[c];
            bool ok = g.ctas >= 1 && g.ctas <= 148;
            // a cluster is one that the device takes, and nothing of one cluster's size runs as a cooperative grid
            ok = ok && (!g.cluster || g.ctas <= kSelClusterMax || (granted && g.ctas == kSelClusterWide));
            ok = ok && (g.cluster || g.ctas > kSelClusterMax) && (g.cluster || !granted || g.ctas > kSelClusterWide);
            // sixteen CTAs are not given the ranking of more candidates than they were measured with
            ok = ok && (g.ctas != kSelClusterWide || cand <= 5120);
            ++seen[g.cluster ? (g.ctas == kSelClusterWide ? 2 : 1) : 3];
            if (!ok && bad++ < 5)
              std::printf("L %%lld budget %%d %%d x %%d: %%d CTAs, cluster %%d\n", L, budget, n_max, n_win, g.ctas, g.cluster);
          }
  std::printf("%%d small clusters, %%d wide, %%d cooperative\n", seen[1], seen[2], seen[3]);
  return bad || !seen[1] || !seen[2] || !seen[3];
}
"""


def test_which_grid_the_selection_takes(tmp_path):
    from test_gpu_walk import WIDE_CASES
    rows = ",\n".join("{%d, %d, %d, %d, %s, %d, %s}" % (L, budget, n_sink, len(ms), ", ".join(map(str, ms)), len(ws),
                                                        ", ".join(map(str, ws)))
                      for L, budget, ms, ws, n_sink in WIDE_CASES)
    _run(tmp_path, GRIDS % rows)
