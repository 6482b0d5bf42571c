"""klpm_replay of an order that is short against its queue (only the groups it touches are looked at before the loop), on both sides of
an eighth of the queue, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2502_04677_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def K():
    from paper_2502_04677_b200 import binding
    return binding


@pytest.mark.parametrize("budget", [0, 2500])
@pytest.mark.parametrize("n_order", [1, 2, 24, 49, 50, 51, 400])
def test_short_order_over_a_queue_with_groups(K, budget, n_order):
    n = 400
    rng = np.random.RandomState(n_order)
    stems = [rng.randint(0, 50, size=120).tolist() for _ in range(6)]
    tails, arr = W.random_small_queue(3, n, vocab=2, max_len=12, max_gap=20)
    prompts = [(stems[i % 7][:int(rng.randint(1, 121))] if i % 7 < 6 else [60 + i]) + t for i, t in enumerate(tails)]
    qt, qo = W.to_csr(prompts)
    ta = np.asarray(arr, dtype=np.int64)
    order = rng.permutation(n)[:n_order].astype(np.int32)
    tree = K.rt_create(max_nodes=4 * n + 64, max_pool_tokens=2 * qt.numel() + 16 * n + 64, budget_tokens=budget, max_clock=2 * n + 64)
    ot = oracle.OracleTree(budget)
    d = qt.cuda(), qo.cuda(), torch.from_numpy(ta).cuda()
    for _ in range(2):                                       # on an empty cache, and on what that left
        unc = torch.full((n,), -7, dtype=torch.int32, device="cuda")
        ttft, done = (torch.full((n,), -7, dtype=torch.int64, device="cuda") for _ in range(2))
        K.klpm_replay(tree, torch.from_numpy(order).cuda(), *d, K.make_params(K.POLICY_KLPM, 2, 1, 3, 2), unc, ttft, done)
        assert K.rt_sync_status(tree) == 0
        want = oracle.replay(order, qt.numpy(), qo.numpy(), ta, 1, 3, 2, oracle.CACHE_TREE, ot)
        rest = np.setdiff1d(np.arange(n), order)
        for g, w in zip((unc, ttft, done), want):
            g = g.cpu().numpy()
            assert np.array_equal(g[order], w[order]) and (g[rest] == -7).all()
    st, ost = K.rt_stats(tree), ot.stats()
    for key in ("n_nodes", "tokens", "clock", "evictions"):
        assert st[key] == ost[key], key
    m = torch.zeros(n, dtype=torch.int32, device="cuda")
    K.rt_match_batch(tree, d[0], d[1], m)
    assert np.array_equal(m.cpu().numpy(), ot.match(qt.numpy(), qo.numpy()))
