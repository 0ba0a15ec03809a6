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


FORMS = r"""
#include <cstdio>
#include "qk_geometry.cuh"
using namespace ilre;
int main() {
  const int cases[][5] = {%s};          // kv heads, heads per kv head, query tokens, keys; loaded in copies
  int bad = 0, behind = 0;
  for (const auto& c : cases) {
    const int rows = c[1] * c[2];
    const Geometry g = make_geometry(c[0], c[0] * c[1], 148, c[3], c[2]);
    const int last = rows - (g.stats.n_rb - 1) * g.stats.rb_rows;
    behind += g.stats_tail && stats_tail_copies(last) > 1 && (last + 127) / 128 < (g.stats.rb_rows + 127) / 128;
    if (g.stats_tail != (c[4] != 0) && ++bad)
      std::printf("%%d x %%d heads, %%d tokens, %%d keys: copies %%d\n", c[0], c[1], c[2], c[3], g.stats_tail);
  }
  return bad || behind < 2;
}
"""


def test_gpu_cases_take_the_form_they_are_listed_under(tmp_path):
    """And two of them copy a tile that is not the last of its block."""
    from test_gpu_row_tails import COPIED, PLAIN
    rows = ["{%d, %d, %d, %d, %d}" % (*c, form) for form, cases in ((1, COPIED), (0, PLAIN)) for c in cases]
    _run(tmp_path, FORMS % ", ".join(rows))
