"""How the statistics pass splits the query rows of a kv head, compiled from the library's header with
the host compiler.  No GPU."""
from test_launch_plan import _run

SPLIT = r"""
#include <cstdio>
#include <cstring>
#include "qk_geometry.cuh"
using namespace ilre;
int main() {
  long long bad = 0, copied = 0, uneven = 0;
  for (int group : {1, 2, 3, 4, 7, 8, 32, 64, 128})
    for (int n_kv : {1, 4, 8, 16})
      for (long long L : {100LL, 16129LL, 40000LL, 1000000LL})
        for (int q_len = 1; q_len < 700; ++q_len) {
          const Geometry g = make_geometry(n_kv, n_kv * group, 148, L, q_len);
          const int rows = group * q_len, rb = g.stats.rb_rows, n_rb = g.stats.n_rb;
          bool ok = rb <= kMaxRbRows && (n_rb - 1) * rb < rows && n_rb * rb >= rows && g.stats.stages >= 2;
          ok = ok && g.scores.rb_rows % 128 == 0 && g.kv_rows <= rows_padded_bound(group, q_len);
          // a box starts at a whole token and no tile reads past the packed rows of its kv head
          ok = ok && (128 % group != 0 || rb % group == 0 || n_rb == 1) && (n_rb - 1) * rb + ((rb + 127) & ~127) <= g.kv_rows;
          if (g.stats_tail) {
            ++copied;
            uneven += rb % 128 != 0;
            for (int live = 1; live <= rb; ++live) {
              const int copies = stats_tail_copies(live), tail = stats_tail_rows(live);
              ok = ok && tail <= 128 / copies && (copies == 4 || tail > 128 / (2 * copies)) && copies * (128 / copies) == 128;
            }
            ok = ok && stats_box_rows(group) == 32;
            ok = ok && rows > 128 && g.stats.n_tiles >= kTailMinTiles * g.stats.cpg;
          } else {
            ok = ok && rb % 128 == 0;
          }
          if (!ok && bad++ < 5)
            std::printf("group %d kv %d L %lld q_len %d: %d blocks of %d\n", group, n_kv, L, q_len, n_rb, rb);
        }
  std::printf("%lld with copied tiles, %lld of them in blocks that are no multiple of 128\n", copied, uneven);
  return bad || !copied || !uneven;
}
"""


def test_row_blocks_cover_the_query_and_stay_inside_its_packed_copy(tmp_path):
    _run(tmp_path, SPLIT)
