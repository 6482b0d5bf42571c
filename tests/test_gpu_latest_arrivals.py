"""Arrivals at the largest time an int64 holds: prompts that cost nothing (fully cached, or empty) are finished there and then."""
import numpy as np
import pytest
import torch

import oracle
from paper_2502_04677_b200 import workloads as W

pytestmark = pytest.mark.gpu
LAST = (1 << 63) - 1


@pytest.fixture(scope="module")
def K():
    from paper_2502_04677_b200 import binding
    return binding


@pytest.mark.parametrize("budget", [0, 100_000])
@pytest.mark.parametrize("n,late", [(1, 1), (33, 5), (64, 33), (100, 100), (300, 200)])
@pytest.mark.parametrize("policy,k", [(0, 1), (1, 1), (2, 3)])
def test_arrivals_at_the_end_of_time(K, budget, n, late, policy, k):
    prompts, _ = W.random_small_queue(7, n, vocab=3, max_len=12)
    early = n - late
    qt, qo = W.to_csr(prompts)
    arr = np.array([3 * i for i in range(early)] + [LAST] * late, dtype=np.int64)
    pt, po = W.to_csr(prompts[early:])
    tree = K.rt_create(max_nodes=8 * n + 64, max_pool_tokens=4 * qt.numel() + 64 * n + 64, budget_tokens=budget, max_clock=4 * n + 64)
    K.rt_insert(tree, pt.cuda() if pt.numel() else torch.zeros(4, dtype=torch.int32, device="cuda"), po.cuda())
    out = [torch.full((n,), -1, dtype=d, device="cuda") for d in (torch.int32, torch.int32, torch.int64, torch.int64)]
    d_qt = qt.cuda() if qt.numel() else torch.zeros(4, dtype=torch.int32, device="cuda")
    K.klpm_run(tree, d_qt, qo.cuda(), torch.from_numpy(arr).cuda(), K.make_params(policy, k), *out)
    assert K.rt_sync_status(tree) == 0
    ot = oracle.OracleTree(budget)
    ot.insert(pt.numpy(), po.numpy())
    want = oracle.schedule(qt.numpy(), qo.numpy(), arr, policy, k, 0, 1, 0, oracle.CACHE_TREE, oracle.TIER_REMATCH, ot)
    for g, w in zip(out, want):
        assert np.array_equal(g.cpu().numpy(), w)
    assert (want[2][early:] == 0).all()
