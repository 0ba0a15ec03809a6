"""GPU: statistics of query row counts whose last 128-row tile is short (its rows are loaded two or four
times and share the key tile's columns), with one to four row tiles and several row blocks, for head
groups that are read in place and for ones that are packed, on contexts that end inside a key tile."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
import parity
from workloads import make_inputs, small_workload

pytestmark = pytest.mark.gpu


# (the host test of the row blocks checks that these are loaded in copies, and those are not)
COPIED = [
    # two tiles: 129 and 148 rows (four copies), 147 (packed), 192 (two copies); 14 tiles per CTA and more
    (8, 1, 129, 32256), (8, 4, 37, 32300), (8, 7, 21, 33000), (16, 2, 96, 17001),
    (16, 4, 69, 16200), (16, 8, 40, 17000),                     # three: 276, 320
    (16, 32, 13, 16129), (16, 7, 62, 17100),                    # four: 416, 434 (packed)
    (8, 7, 86, 16500), (16, 4, 300, 9100),                      # blocks of 320 (the last has 282 rows), 416 (368: not copied)
    # blocks of 416, the last of 289 and 292 rows: the copied tile is the third of four, the fourth is empty
    (8, 1, 1537, 7300), (8, 7, 220, 7300),
]
PLAIN = [
    # one row tile, few key tiles per CTA, heads of more than 32 per group, full blocks without a short tile
    (1, 1, 1, 1), (2, 1, 31, 130), (1, 1, 33, 1000), (1, 64, 3, 300), (2, 4, 37, 1111), (1, 64, 3, 270000), (8, 1, 1057, 9999),
]


@pytest.mark.parametrize("n_kv,group,q_len,L", COPIED + PLAIN)
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


def _reference_lse(K, Q):
    """ln of the row sums in 64 bits, [q_len, n_q]."""
    n_kv, n_q = K.shape[1], Q.shape[1]
    k, q = K.double(), Q.double()
    return torch.stack([torch.logsumexp(q[:, h] @ k[:, h * n_kv // n_q].T / 128 ** 0.5, dim=1) for h in range(n_q)], dim=1)


@pytest.mark.parametrize("n_kv,group,q_len,L", [(8, 4, 37, 32300), (8, 7, 86, 16500), (8, 1, 1537, 7300)])
def test_scores_behind_copied_tiles(n_kv, group, q_len, L):
    """The scores pass splits the rows another way than the statistics that it reads."""
    from paper_2508_17892_b200 import IlreRecall
    w = small_workload(L, q_len, n_kv_heads=n_kv, n_q_heads=n_kv * group, budget=64, n_spans=2)
    x = make_inputs(w)
    eng = IlreRecall(max_L=L, max_q_len=q_len, max_budget=64, n_kv_heads=n_kv, n_q_heads=n_kv * group)
    idx, sc = eng.run(x.K.cuda(), x.Q.cuda(), w.budget, w.max_sizes, w.win_sizes, w.win_op, want_scores=True)
    torch.cuda.synchronize()
    eng.check_status()
    parity.check_recall(x.K, x.Q, w, idx.cpu().numpy(), sc.cpu().numpy())
    eng.close()


@pytest.mark.parametrize("n_kv,group,q_len", [(8, 4, 37), (8, 7, 22)])
def test_shards_and_pieces_with_copied_tiles(n_kv, group, q_len):
    """148 and 154 rows per kv head: the exported statistics of a shard, and those of the pieces in which a
    context is uploaded, three of 65536 keys and less (28 key tiles per CTA and fewer)."""
    from paper_2508_17892_b200 import IlreRecall
    L, budget = 165000, 300
    g = torch.Generator(device="cuda").manual_seed(L + q_len)
    K = torch.randn(L, n_kv, 128, generator=g, device="cuda").to(torch.bfloat16)
    Q = torch.randn(q_len, n_kv * group, 128, generator=g, device="cuda").to(torch.bfloat16)
    ref = _reference_lse(K, Q)
    eng = IlreRecall(max_L=L, max_q_len=q_len, max_budget=budget, n_kv_heads=n_kv, n_q_heads=n_kv * group,
                     host_staging=True)
    cut = 100003
    st = torch.stack([eng.shard_stats(K[:cut], Q), eng.shard_stats(K[cut:], Q)]).double().view(2, q_len, -1, 2)
    lse = torch.logsumexp((st[..., 0] + torch.log2(st[..., 1])) * np.log(2.0), dim=0)
    assert (lse - ref).abs().max() < 2e-5               # bound: see above
    idx, sc = eng.run(K, Q, budget, (1,), (1, 7), 1, want_scores=True)
    hidx, hsc = eng.run_host(K.cpu(), Q.cpu(), budget, (1,), (1, 7), 1, out_scores=torch.empty(L))
    assert (eng.row_lse(q_len).double() - ref).abs().max() < 2e-5
    eng.check_status()
    assert eng.check_guards() == 0
    # the same logits, against row sums that were merged in another order: a few 1e-6
    assert ((hsc.cuda() - sc).abs() <= 2e-5 * sc).all()
    assert len(set(hidx.tolist()) ^ set(idx.tolist())) <= 2
    eng.close()
