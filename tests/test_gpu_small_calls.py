"""Calls of the sizes an online scheduler makes: few queries per batched match, short queues per selection."""
import numpy as np
import pytest
import torch

import oracle
from paper_2502_04677_b200 import workloads as W

pytestmark = pytest.mark.gpu

SMS = 148                                        # the batch sizes at which a B200 takes fewer warps per query


@pytest.fixture(scope="module")
def K():
    from paper_2502_04677_b200 import binding
    return binding


def long_edges():
    """Cached prompts that cut two trunks at many depths, and queries that leave them around every comparison boundary (512 tokens per
    warp, 4,096 per CTA), inside edges and at node ends, at every 16-byte phase."""
    rng = np.random.RandomState(3)
    trunks = [rng.randint(0, 1000, size=9000).tolist() for _ in range(2)]
    cached = [trunks[0], trunks[1][:5000] + [1001] * 40]
    for cut in (1, 511, 512, 513, 3000, 4096, 4100, 8190):
        cached.append(trunks[0][:cut] + [1002] + trunks[1][:700])
    queries = [[], [2000], trunks[0], trunks[0] + [7], trunks[1], trunks[0][:512], trunks[0][:4096]]
    for d in [1, 2, 127, 128, 510, 511, 512, 513, 514, 1023, 1024, 1025, 3583, 3584, 3585, 4094, 4095, 4096, 4097, 4608, 4609, 8189, 8190, 8191,
              8192, 8193, 8999]:
        queries.append(trunks[0][:d] + [1003, 5])
        queries.append(trunks[0][:d] + [1002] + trunks[1][:d // 2] + [1003])
        queries.append(trunks[1][:d])
    return cached, queries


@pytest.mark.parametrize("budget", [0, 60_000])
@pytest.mark.parametrize("n", [1, 4 * SMS, 4 * SMS + 1, 8 * SMS + 1, 16 * SMS + 1, 32 * SMS, 32 * SMS + 1])
def test_match_of_few_queries(K, n, budget):
    cached, queries = long_edges()
    ct, co = W.to_csr(cached)
    tree = K.rt_create(max_nodes=4 * len(cached) + 16, max_pool_tokens=ct.numel() + 8 * len(cached) + 16, budget_tokens=budget,
                       max_clock=len(cached) + 16)
    K.rt_insert(tree, ct.cuda(), co.cuda())
    ot = oracle.OracleTree(budget)
    ot.insert(ct.numpy(), co.numpy())
    which = [(5 * i + 2) % len(queries) for i in range(n)]
    lens = np.array([len(queries[w]) for w in which], dtype=np.int64)
    pad = 3                                      # the first query starts off a 16-byte boundary
    off = np.zeros(n + 1, dtype=np.int64)
    off[0] = pad
    off[1:] = pad + np.cumsum(lens)
    flat = [torch.tensor(q, dtype=torch.int32) for q in queries]
    tok = torch.cat([torch.zeros(pad, dtype=torch.int32)] + [flat[w] for w in which] + [torch.zeros(8, dtype=torch.int32)]).cuda()
    m, node, at = (torch.full((n,), -7, dtype=torch.int32, device="cuda") for _ in range(3))
    K.rt_match_batch(tree, tok, torch.from_numpy(off).cuda(), m, node, at)
    assert K.rt_sync_status(tree) == 0
    qt, qo = W.to_csr(queries)
    want_m, want_at, want_depth = (np.asarray(x)[which] for x in ot.match_pos(qt.numpy(), qo.numpy()))
    assert np.array_equal(m.cpu().numpy(), want_m)
    assert np.array_equal(at.cpu().numpy(), want_at)
    assert np.array_equal((m - at).cpu().numpy(), want_depth)
    assert np.array_equal((node == 0).cpu().numpy(), want_m == 0)
    if n > 1:                                    # the records of the same match carry a whole schedule (trees without a budget use them)
        state = K.match_state_buffer(n, "cuda")
        K.rt_match_batch_ex(tree, tok, torch.from_numpy(off).cuda(), m, node, at, state)
        assert np.array_equal(m.cpu().numpy(), want_m)


@pytest.mark.parametrize("n", [16_384, 16_385])
def test_match_around_the_ordered_batches(K, n):
    """Trees without a budget: the last batch size that is taken in index order and the first that is ordered."""
    cached, queries = long_edges()
    queries = [q[:900] for q in queries]
    ct, co = W.to_csr(cached)
    tree = K.rt_build(ct.cuda(), co.cuda(), max_nodes=4 * len(cached) + 16, max_pool_tokens=ct.numel() + 8 * len(cached) + 16)
    qt, qo = W.to_csr(queries)
    want = oracle.OracleTree(0)
    want.insert(ct.numpy(), co.numpy())
    want_m = want.match_pos(qt.numpy(), qo.numpy())[0]
    reps = -(-n // len(queries))
    tok = qt.repeat(reps).cuda()
    lens = np.tile(np.diff(qo.numpy()), reps)
    off = np.concatenate([[0], np.cumsum(lens)])[:n + 1]
    m = torch.full((n,), -7, dtype=torch.int32, device="cuda")
    K.rt_match_batch(tree, tok, torch.from_numpy(off).cuda(), m)
    assert K.rt_sync_status(tree) == 0
    assert np.array_equal(m.cpu().numpy(), np.tile(want_m, reps)[:n])


@pytest.mark.parametrize("n", [0, 1, 31, 33, 1023, 1025, 8191, 8192, 8193])
def test_selection_on_both_sides_of_the_one_cta_kernel(K, n):
    """One pick and the 64 best of queues around a warp, a thread per query and the largest queue that one CTA holds: few distinct
    values (ties), negative and large arrivals, queues with fewer than 64 waiting."""
    g = torch.Generator().manual_seed(n)
    m = torch.randint(0, 7, (n,), generator=g, dtype=torch.int32)
    t = torch.randint(-2, 3, (n,), generator=g, dtype=torch.int64) * ((1 << 33) + 1)
    for waiting in (torch.ones(n, dtype=torch.uint8), (torch.randint(0, 200, (n,), generator=g) == 0).to(torch.uint8), torch.zeros(n, dtype=torch.uint8)):
        d = m.cuda(), t.cuda(), waiting.cuda()
        for policy, k, c in ((K.POLICY_KLPM, 3, 6), (K.POLICY_KLPM, 3, 7), (K.POLICY_FCFS, 1, 1), (K.POLICY_LPM, 1, 0)):
            pick, same = torch.full((1,), -7, dtype=torch.int32, device="cuda"), torch.full((1,), -7, dtype=torch.int32, device="cuda")
            K.klpm_select(*d, c, K.make_params(policy, k), pick)
            K.klpm_select_noalloc(*d, c, K.make_params(policy, k), same)
            want = oracle.select(m.numpy(), t.numpy(), waiting.numpy(), c, policy, k) if n else -1
            assert int(pick) == want and int(same) == want
        out = torch.full((64,), -7, dtype=torch.int32, device="cuda")
        K.klpm_select_topk(*d, out)
        idx = np.nonzero(waiting.numpy())[0]
        best = sorted(idx.tolist(), key=lambda i: (-int(m[i]), int(t[i]), i))[:64]
        assert out.tolist() == best + [-1] * (64 - len(best))


@pytest.mark.parametrize("budget", [0, 300, 900])
@pytest.mark.parametrize("batch", [1, 7, 100])
def test_insert_in_order_with_results(K, budget, batch):
    """Prompts stored one after the other in calls of several sizes: prompts of one call that extend, cut and repeat each other, leaves
    (and then their parents) evicted between a prompt's match and its turn, empty and fully cached prompts."""
    prompts, _ = W.random_small_queue(77 + batch, 300, vocab=2, max_len=30)
    more, _ = W.random_small_queue(78, 100, vocab=3, max_len=120)
    prompts = [p for pair in zip(prompts, more * 3) for p in pair]
    prompts += prompts[10:60] + [[]] + [p + [1, 1, 0] for p in prompts[20:40]]
    pt, po = W.to_csr(prompts)
    n = len(prompts)
    tree = K.rt_create(max_nodes=2 * n + 16, max_pool_tokens=pt.numel() + 8 * n + 16, budget_tokens=budget, max_clock=n + 16)
    new = torch.full((n,), -7, dtype=torch.int32, device="cuda")
    tok, off = pt.cuda(), po.cuda()
    for a in range(0, n, batch):
        b = min(n, a + batch)
        K.rt_insert(tree, tok, off[a:b + 1], new[a:b])
    assert K.rt_sync_status(tree) == 0
    ot = oracle.OracleTree(budget)
    assert np.array_equal(new.cpu().numpy(), ot.insert(pt.numpy(), po.numpy()))
    st, want = K.rt_stats(tree), ot.stats()
    for key in ("n_nodes", "tokens", "clock", "evictions"):
        assert st[key] == want[key], key
    qs, _ = W.random_small_queue(79, 200, vocab=2, max_len=40)
    qt, qo = W.to_csr(qs + prompts)
    m, at = (torch.zeros(len(qs) + n, dtype=torch.int32, device="cuda") for _ in range(2))
    K.rt_match_batch(tree, qt.cuda(), qo.cuda(), m, None, at)
    want_m, want_at, _ = ot.match_pos(qt.numpy(), qo.numpy())
    assert np.array_equal(m.cpu().numpy(), want_m) and np.array_equal(at.cpu().numpy(), want_at)
    # the loop goes on from the tree that the insertions left
    if budget:
        k = 40
        o = [torch.zeros(k, dtype=d, device="cuda") for d in (torch.int32, torch.int32, torch.int64)]
        q1, q2 = W.to_csr(prompts[:k])
        tree2 = K.rt_create(max_nodes=2 * (n + k) + 16, max_pool_tokens=pt.numel() + q1.numel() + 8 * (n + k) + 2 * budget + 64, budget_tokens=budget, max_clock=n + k + 16)
        K.rt_insert(tree2, tok, off, new)
        K.klpm_run(tree2, q1.cuda(), q2.cuda(), torch.zeros(k, dtype=torch.int64, device="cuda"), K.make_params(K.POLICY_KLPM, 3), *o)
        assert K.rt_sync_status(tree2) == 0
        wo, wu, wt, _ = oracle.schedule(q1.numpy(), q2.numpy(), np.zeros(k, dtype=np.int64), oracle.POLICY_KLPM, 3, 0, 1, 0, oracle.CACHE_TREE,
                                        oracle.TIER_REMATCH, ot)
        assert np.array_equal(o[0].cpu().numpy(), wo) and np.array_equal(o[1].cpu().numpy(), wu) and np.array_equal(o[2].cpu().numpy(), wt)


@pytest.mark.parametrize("n,budget", [(16_385, 0), (65_537, 60_000)])
def test_ordered_match_kernels_on_long_edges(K, n, budget):
    """The smallest batches of the ordered kernels, one without and one with a budget: the long queries at full length at every 16-byte
    phase between short ones, match length and where the match ended."""
    cached, queries = long_edges()
    ct, co = W.to_csr(cached)
    tree = K.rt_create(max_nodes=4 * len(cached) + 16, max_pool_tokens=ct.numel() + 8 * len(cached) + 16, budget_tokens=budget,
                       max_clock=len(cached) + 16)
    K.rt_insert(tree, ct.cuda(), co.cuda())
    ot = oracle.OracleTree(budget)
    ot.insert(ct.numpy(), co.numpy())
    short = [q[:9 + i % 7] for i, q in enumerate(queries)]
    both = queries + short
    which = len(queries) + np.arange(n) % len(short)
    at_long = np.random.RandomState(4).permutation(n)[:8 * len(queries)]
    which[at_long] = np.arange(8 * len(queries)) % len(queries)
    flat = [torch.tensor(q, dtype=torch.int32) for q in both]
    off = np.concatenate([[0], np.cumsum([len(both[w]) for w in which])]).astype(np.int64)
    tok = torch.cat([flat[w] for w in which]).cuda()
    m, node, at = (torch.full((n,), -7, dtype=torch.int32, device="cuda") for _ in range(3))
    K.rt_match_batch(tree, tok, torch.from_numpy(off).cuda(), m, node, at)
    assert K.rt_sync_status(tree) == 0
    qt, qo = W.to_csr(both)
    want_m, want_at, want_depth = (np.asarray(x)[which] for x in ot.match_pos(qt.numpy(), qo.numpy()))
    assert np.array_equal(m.cpu().numpy(), want_m)
    assert np.array_equal(at.cpu().numpy(), want_at)
    assert np.array_equal((m - at).cpu().numpy(), want_depth)
    assert np.array_equal((node == 0).cpu().numpy(), want_m == 0)
    assert len({int(off[i]) % 4 for i in at_long}) == 4


@pytest.mark.parametrize("budget", [0, 1200])
@pytest.mark.parametrize("n", [1, 2, 33, 1023, 1024, 1025])
def test_schedule_around_the_one_cta_set_up_of_groups(K, n, budget):
    """Queues with groups of all sizes on both sides of the longest that one CTA groups, on a cache that holds some of them, twice."""
    rng = np.random.RandomState(n)
    stems = [rng.randint(0, 9, size=80).tolist() for _ in range(5)]
    tails, _ = W.random_small_queue(n, n, vocab=2, max_len=10)
    prompts = [(stems[i % 6][:int(rng.randint(1, 81))] if i % 6 < 5 else []) + t for i, t in enumerate(tails)]
    prompts[0] = prompts[0] + [1]
    qt, qo = W.to_csr(prompts)
    arr = np.zeros(n, dtype=np.int64)
    tree = K.rt_create(max_nodes=8 * n + 64, max_pool_tokens=4 * qt.numel() + 64 * n + 2 * budget + 64, budget_tokens=budget, max_clock=4 * n + 64)
    ct, co = W.to_csr([s[:40] for s in stems])
    K.rt_insert(tree, ct.cuda(), co.cuda())
    ot = oracle.OracleTree(budget)
    ot.insert(ct.numpy(), co.numpy())
    for policy, k in ((K.POLICY_KLPM, 3), (K.POLICY_LPM, 1)):
        out = [torch.full((n,), -1, dtype=d, device="cuda") for d in (torch.int32, torch.int32, torch.int64, torch.int64)]
        K.klpm_run(tree, qt.cuda(), qo.cuda(), torch.from_numpy(arr).cuda(), K.make_params(policy, k, 1, 3, 2), *out)
        assert K.rt_sync_status(tree) == 0
        want = oracle.schedule(qt.numpy(), qo.numpy(), arr, policy, k, 1, 3, 2, oracle.CACHE_TREE, oracle.TIER_REMATCH, ot)
        for g, w in zip(out, want):
            assert np.array_equal(g.cpu().numpy(), w)
    st, ost = K.rt_stats(tree), ot.stats()
    for key in ("n_nodes", "tokens", "clock", "evictions"):
        assert st[key] == ost[key], key
