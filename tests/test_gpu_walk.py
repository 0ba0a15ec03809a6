"""GPU: selection, quota walk and ascending output where their paths change.

A walking thread takes four ranked cells per round, at most 1024 threads walk: lists of more than
4096 cells take several rounds, and may meet the quota before their last one.  Cells lie in one,
two or three bitmap words.  The output pass takes a lane per bitmap word up to 32768 positions,
a list of words shared out over the warps behind, in one round or many; above 1 114 112 positions the
bitmap lives in global memory.
"""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
import parity
from workloads import make_inputs, small_workload

pytestmark = pytest.mark.gpu

# Contexts that run as one cluster of 16 CTAs (the host test of the launch rules checks that they do): the fewest
# and the most cells, few and many candidates, a strided max-pool, more than 8 combinations.
WIDE_CASES = [
    # L, budget, max sizes, window sizes, n_sink
    (4096, 512, (1,), (1, 7, 15), 0),
    (6830, 512, (1,), (1, 7, 15), 2),
    (16384, 512, (1,), (1, 7, 15), 0),
    (24001, 2040, (1,), (1, 7, 15), 3),
    (20001, 300, (1, 2), (1, 9), 0),
    (3003, 300, (1, 2, 4), (1, 4, 9, 15), 1),
]
CASES = WIDE_CASES + [
    (1, 1, (1,), (1,), 0),
    (129, 125, (1,), (3, 5), 4),
    (12289, 2047, (1,), (1, 7, 15, 31, 63), 3),
    (32768, 4097, (1,), (1, 7, 15), 0),             # a lane per word, the last such length
    (32773, 5, (2, 64), (1, 2), 5),                 # 32768 positions behind the sink part
    (32769, 16382, (1,), (1, 31), 0),               # word list; four rounds, met before the last
    (40001, 16000, (3, 1, 48), (1, 9), 1),          # cells of one, two and three words
    (131072, 12289, (1, 2, 32, 33, 64), (1, 4), 0),
    (1048576, 16000, (1,), (1, 7), 0),              # a list of many rounds per warp where spread out
    (1114113, 9000, (1, 5, 64), (1, 15), 0),        # bitmap in global memory
]


@pytest.mark.parametrize("lie", ["spread", "runs", "together"])
@pytest.mark.parametrize("L,budget,max_sizes,win_sizes,n_sink", CASES)
def test_walk_and_output(L, budget, max_sizes, win_sizes, n_sink, lie):
    """Windows take the maximum, so every value is exact on both sides: identical positions."""
    from paper_2508_17892_b200 import IlreRecall
    rng = np.random.default_rng(L + budget)
    a = (rng.random(L) ** 4).astype(np.float32)
    if lie == "runs":                               # whole runs of high and equal scores
        for p in rng.integers(0, L, size=max(1, L // 4000)):
            a[p:p + 300] = np.float32(0.5 + 0.4 * rng.random())
    elif lie == "together":                         # a third of one 32nd of the context
        part = a[5 * L // 32:6 * L // 32 + 1]
        part += np.where(rng.random(len(part)) < 0.33, 1, 0).astype(np.float32)
    eng = IlreRecall(max_L=L, max_q_len=1, max_budget=budget, n_kv_heads=1, n_q_heads=1,
                     max_combinations=len(max_sizes) * len(win_sizes))
    idx = eng.allocate(torch.from_numpy(a).cuda(), budget, max_sizes, win_sizes, 1, n_sink)
    torch.cuda.synchronize()
    eng.check_status()
    assert eng.check_guards() == 0
    ref = oracle.allocate(a.astype(np.float64), budget, max_sizes, win_sizes, 1, n_sink)
    assert np.array_equal(idx.cpu().numpy(), ref)
    eng.close()


@pytest.mark.parametrize("L,budget,max_sizes,win_sizes,n_sink", WIDE_CASES[2:5])
def test_one_cluster_of_16_behind_the_scores_pass(L, budget, max_sizes, win_sizes, n_sink):
    """Encoded scores, decoded by every CTA of the cluster, and the scores written for the caller."""
    from paper_2508_17892_b200 import IlreRecall
    w = small_workload(L, 3, n_kv_heads=2, n_q_heads=4, budget=budget, max_sizes=max_sizes, win_sizes=win_sizes,
                       win_op=1, n_sink=n_sink, n_spans=3)
    x = make_inputs(w)
    eng = IlreRecall(max_L=L, max_q_len=3, max_budget=budget, n_kv_heads=2, n_q_heads=4,
                     max_combinations=len(max_sizes) * len(win_sizes))
    idx, sc = eng.run(x.K.cuda(), x.Q.cuda(), budget, max_sizes, win_sizes, 1, n_sink, want_scores=True)
    torch.cuda.synchronize()
    eng.check_status()
    assert eng.check_guards() == 0
    parity.check_recall(x.K, x.Q, w, idx.cpu().numpy(), sc.cpu().numpy())
    eng.close()


@pytest.mark.parametrize("win_op,win_sizes", [(1, (1, 1023)), (0, (8, 64))])
def test_the_longest_context(win_op, win_sizes):
    """2^31 - 257 positions, scores above zero among the last 20000 only: what is chosen there is what a
    context that begins behind the zeros gives.  (Values are multiples of 2^-17 below 1, window sizes of the
    averages powers of two: every sum and quotient is exact.)"""
    from paper_2508_17892_b200 import IlreRecall
    L, tail, budget = 2 ** 31 - 257, 20000, 2000
    if torch.cuda.mem_get_info()[0] < 80 << 30:
        pytest.skip("needs 80 GB of free device memory")
    rng = np.random.default_rng(7)
    a = (rng.integers(1, 2 ** 17, size=tail) / 2 ** 17).astype(np.float32)
    a[:2000] = 0
    eng = IlreRecall(max_L=L, max_q_len=1, max_budget=budget, n_kv_heads=1, n_q_heads=1, max_combinations=2)
    scores = torch.zeros(L, device="cuda")
    scores[-tail:] = torch.from_numpy(a).cuda()
    idx = eng.allocate(scores, budget, (1,), win_sizes, win_op)
    torch.cuda.synchronize()
    eng.check_status()
    assert eng.check_guards() == 0
    ref = oracle.allocate(a.astype(np.float64), budget, (1,), win_sizes, win_op)
    eng.close()
    del scores
    torch.cuda.empty_cache()
    assert np.array_equal(idx.cpu().numpy(), ref + (L - tail))
