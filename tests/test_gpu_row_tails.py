"""GPU: statistics of query row counts whose last 128-row tile is short (its rows are loaded two or four
times and share the key tile's columns), with one to four row tiles and several row blocks, for head
groups that are read in place and for ones that are packed, on contexts that end inside a key tile."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
from workloads import make_inputs, small_workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_kv,group,q_len,L", [
    # few key tiles per CTA, or one row tile, or heads of more than 32 per group: no copies
    (1, 1, 1, 1), (2, 1, 31, 130), (1, 1, 33, 1000), (1, 64, 3, 300), (2, 4, 37, 1111), (1, 64, 3, 270000),
    # two tiles: 129 and 148 rows (four copies), 147 (packed), 192 (two copies); 14 tiles per CTA and more
    (8, 1, 129, 32256), (8, 4, 37, 32300), (8, 7, 21, 33000), (16, 2, 96, 17001),
    (16, 4, 69, 16200), (16, 8, 40, 17000),                     # three: 276, 320
    (16, 32, 13, 16129), (16, 7, 62, 17100),                    # four: 416, 434 (packed)
    (8, 7, 86, 16500), (16, 4, 300, 9100), (8, 1, 1057, 9999),  # blocks of 320 (301 live), 416, 384 (353)
])
def test_row_statistics_of_short_last_tiles(n_kv, group, q_len, L):
    """lse: sums in fp32 of exponentials within 2.7e-6 (relative), merged over chunks, copies and
    warpgroups: a few 1e-6 in all; 2e-5 is far below what a wrong row or column would change."""
    from paper_2508_17892_b200 import IlreRecall
    w = small_workload(L, q_len, n_kv_heads=n_kv, n_q_heads=n_kv * group, budget=min(L, 64),
                       n_spans=2 if L > 200 else 0)
    x = make_inputs(w)
    eng = IlreRecall(max_L=L, max_q_len=q_len, max_budget=64, n_kv_heads=n_kv, n_q_heads=n_kv * group)
    eng.run(x.K.cuda(), x.Q.cuda(), w.budget, w.max_sizes, w.win_sizes, w.win_op)
    torch.cuda.synchronize()
    eng.check_status()
    assert eng.check_guards() == 0
    m, z = oracle.row_stats(x.K, x.Q, range(q_len * w.n_q_heads))
    lse = eng.row_lse(q_len).cpu().numpy().reshape(-1)
    assert np.abs(lse - (m + np.log(z))).max() < 2e-5
    eng.close()
