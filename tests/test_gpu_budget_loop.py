"""The loop on a tree with a budget (one warp decides, another keeps the tree) in the layouts that long queues take, against the
oracle: leaf blocks of more than 32 slots, the processed bitmap in global memory, crowds of arrivals, and a given order."""
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


@pytest.mark.parametrize("max_blocks,smem_kb", [(0, 0), (4, 0), (3, 48)])
@pytest.mark.parametrize("max_gap", [0, 2, 60])
def test_budgeted_loop_layouts(K, max_blocks, smem_kb, max_gap):
    """700 prompts over a tiny alphabet with a few long shared stems, budgets that evict all the time: queries fall back out of evicted
    leaves, groups dissolve by the warp and by the CTA, several arrive at once."""
    rng = np.random.RandomState(max_gap)
    prompts, arr = W.random_small_queue(31 + max_gap, 700, vocab=2, max_len=20, max_gap=max_gap)
    stems = [rng.randint(0, 2, size=600).tolist() for _ in range(3)]
    prompts = [stems[int(rng.randint(0, 3))][:int(rng.randint(1, 601))] + p if rng.randint(0, 3) == 0 else p for p in prompts]
    qt, qo = W.to_csr(prompts)
    n = len(prompts)
    ta = np.asarray(arr, dtype=np.int64)
    try:
        K.klpm_debug_set("fast_max_blocks", max_blocks if max_blocks else -1)
        K.klpm_debug_set("fast_smem_kb", smem_kb if smem_kb else -1)
        for policy, k, budget in ((K.POLICY_KLPM, 3, 1500), (K.POLICY_LPM, 1, 900), (K.POLICY_FCFS, 1, 4000)):
            tree = K.rt_create(max_nodes=4 * n + 64, max_pool_tokens=3 * qt.numel() + 32 * n + 64, budget_tokens=budget, max_clock=2 * n + 64)
            out = [torch.full((n,), -1, dtype=d, device="cuda") for d in (torch.int32, torch.int32, torch.int64, torch.int64)]
            K.klpm_run(tree, qt.cuda(), qo.cuda(), torch.from_numpy(ta).cuda(), K.make_params(policy, k, 1, 3, 2), *out)
            assert K.rt_sync_status(tree) == 0
            ot = oracle.OracleTree(budget)
            want = oracle.schedule(qt.numpy(), qo.numpy(), ta, policy, k, 1, 3, 2, oracle.CACHE_TREE, oracle.TIER_REMATCH, ot)
            for g, w in zip(out, want):
                assert np.array_equal(g.cpu().numpy(), w), (policy, k)
            st, ost = K.rt_stats(tree), ot.stats()
            for key in ("n_nodes", "tokens", "clock", "evictions"):
                assert st[key] == ost[key], key
            assert ost["evictions"] > 0
            # the same order again, given, on the cache the first pass left
            unc, ttft = torch.zeros_like(out[1]), torch.zeros_like(out[2])
            K.klpm_replay(tree, out[0], qt.cuda(), qo.cuda(), torch.from_numpy(ta).cuda(), K.make_params(policy, k, 1, 3, 2), unc, ttft)
            assert K.rt_sync_status(tree) == 0
            wu, wt, _ = oracle.replay(want[0], qt.numpy(), qo.numpy(), ta, 1, 3, 2, oracle.CACHE_TREE, ot)
            assert np.array_equal(unc.cpu().numpy(), wu) and np.array_equal(ttft.cpu().numpy(), wt)
    finally:
        K.klpm_debug_set("fast_max_blocks", -1)
        K.klpm_debug_set("fast_smem_kb", -1)


def _stem_queue(queue_seed, seed, vocab, n=700):
    rng = np.random.RandomState(seed)
    prompts, _ = W.random_small_queue(queue_seed, n, vocab=vocab, max_len=20, max_gap=0)
    stems = [rng.randint(0, vocab, size=600).tolist() for _ in range(3)]
    return [stems[int(rng.randint(0, 3))][:int(rng.randint(1, 601))] + p if rng.randint(0, 3) == 0 else p for p in prompts]


@pytest.mark.parametrize("queue_seed,seed,vocab", [(31, 4, 2), (31, 18, 2), (31, 19, 2), (38, 7, 2), (32, 32, 3), (26, 26, 8), (29, 29, 8), (31, 31, 8)])
def test_fall_backs_out_of_a_leaf_and_the_node_above_it(K, queue_seed, seed, vocab):
    """Everybody has arrived.  In each of these queues a decision evicts a leaf together with the node above it while more than 32
    queries are parked in the leaf, matches of which end in that node: whoever counts only those that end in the leaf itself
    sees 0 to 31 of the 42 to 95 that lose tokens."""
    prompts = _stem_queue(queue_seed, seed, vocab)
    qt, qo = W.to_csr(prompts)
    n = len(prompts)
    ta = np.zeros(n, dtype=np.int64)
    tree = K.rt_create(max_nodes=4 * n + 64, max_pool_tokens=3 * qt.numel() + 32 * n + 64, budget_tokens=1500, max_clock=2 * n + 64)
    out = [torch.full((n,), -1, dtype=d, device="cuda") for d in (torch.int32, torch.int32, torch.int64, torch.int64)]
    K.klpm_run(tree, qt.cuda(), qo.cuda(), torch.from_numpy(ta).cuda(), K.make_params(K.POLICY_KLPM, 3, 1, 3, 2), *out)
    assert K.rt_sync_status(tree) == 0
    ot = oracle.OracleTree(1500)
    want = oracle.schedule(qt.numpy(), qo.numpy(), ta, K.POLICY_KLPM, 3, 1, 3, 2, oracle.CACHE_TREE, oracle.TIER_REMATCH, ot)
    for g, w in zip(out, want):
        assert np.array_equal(g.cpu().numpy(), w)
    st, ost = K.rt_stats(tree), ot.stats()
    for key in ("n_nodes", "tokens", "clock", "evictions"):
        assert st[key] == ost[key], key
    unc, ttft = torch.zeros_like(out[1]), torch.zeros_like(out[2])
    K.klpm_replay(tree, out[0], qt.cuda(), qo.cuda(), torch.from_numpy(ta).cuda(), K.make_params(K.POLICY_KLPM, 3, 1, 3, 2), unc, ttft)
    assert K.rt_sync_status(tree) == 0
    wu, wt, _ = oracle.replay(want[0], qt.numpy(), qo.numpy(), ta, 1, 3, 2, oracle.CACHE_TREE, ot)
    assert np.array_equal(unc.cpu().numpy(), wu) and np.array_equal(ttft.cpu().numpy(), wt)
