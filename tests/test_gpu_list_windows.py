"""Queues that take several windows of the list-mode loop (2,048 entries of either pick order each), with prompts that share their
continuation in twos and threes: compared with the one-decision-at-a-time loop, which the oracle checks at smaller sizes."""
import numpy as np
import pytest
import torch

from paper_2502_04677_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def K():
    from paper_2502_04677_b200 import binding
    return binding


@pytest.mark.parametrize("n", [2047, 2049, 8191, 8193, 12288])
@pytest.mark.parametrize("own", [900, 40_000])
def test_windows_against_the_one_by_one_loop(K, n, own):
    """`own` different continuations of 12 prefixes (two of one length): at 900 two thirds of the prompts share theirs with one or two others,
    more to a window than are looked at for groups of two; at 40,000 few do, and queues of 8,192 and more work them out inside the rounds."""
    rng = np.random.RandomState(n + own)
    prefixes = [rng.randint(0, 1000, size=ln).tolist() for ln in (3, 9, 17, 17, 25, 33, 40, 41, 50, 64, 80, 90)]
    prompts = [prefixes[rng.randint(12)] + [2000 + int(rng.randint(own))] + rng.randint(0, 9, size=rng.randint(0, 4)).tolist() for _ in range(n)]
    ct, co = W.to_csr([p + [1001] for p in prefixes])
    qt, qo = W.to_csr(prompts)
    arr = torch.from_numpy(np.sort(rng.randint(0, 50, size=n)).astype(np.int64)).cuda()
    prio = torch.from_numpy(rng.randint(0, 20, size=n).astype(np.int64)).cuda()
    d_qt, d_qo = qt.cuda(), qo.cuda()
    tree = K.rt_build(ct.cuda(), co.cuda(), max_nodes=2 * n + 64, max_pool_tokens=ct.numel() + qt.numel() + 8 * n + 64, max_clock=n + 64)
    K.rt_checkpoint(tree)
    for policy, k, ties, mode in ((2, 2, False, 0), (2, 4, False, 0), (2, 5, True, 1), (2, 300, False, 0), (1, 1, True, 0), (0, 1, False, 0)):
        got = []
        for one_by_one in (0, 1):
            K.rt_rollback(tree)
            out = [torch.full((n,), -1, dtype=d, device="cuda") for d in (torch.int32, torch.int32, torch.int64, torch.int64)]
            K.klpm_debug_set("run_one_by_one", one_by_one)
            try:
                K.klpm_run_ex(tree, d_qt, d_qo, arr, K.make_params(policy, k, 1, 3, 50), prio if ties else None, mode, *out)
                assert K.rt_sync_status(tree) == 0
            finally:
                K.klpm_debug_set("run_one_by_one", -1)
            got.append(out)
        for a, b in zip(*got):
            assert torch.equal(a, b), (policy, k, ties, mode)


@pytest.mark.parametrize("windows", [0, 1, 2])
@pytest.mark.parametrize("start", [50, 0])
def test_a_loop_that_gives_up_charges_nothing(K, windows, start):
    """The loop stops after that many windows of list mode: the status word says so, and the charge pass leaves the outputs of the
    decisions made there alone (the entries of `order` behind them were never written and name no prompt).  With start 0 some
    decisions come before everybody has arrived, and those stand.  A tree that is asked again gives what it always gives."""
    n = 9000
    rng = np.random.RandomState(windows)
    prompts = [[int(rng.randint(40)), 100 + int(rng.randint(3)), 1000 + i] for i in range(n)]
    ct, co = W.to_csr([[a, 100 + b, 999] for a in range(40) for b in range(3)])      # what they share is cached: no groups, every decision is a window's
    qt, qo = W.to_csr(prompts)
    d_qt, d_qo = qt.cuda(), qo.cuda()
    arr = torch.from_numpy(np.sort(rng.randint(0, 50, size=n)).astype(np.int64)).cuda()
    params = K.make_params(K.POLICY_KLPM, 3, 0, 1, start)
    got = []
    for limit in (windows, -1):
        tree = K.rt_build(ct.cuda(), co.cuda(), max_nodes=2 * n + 512, max_pool_tokens=ct.numel() + qt.numel() + 8 * n + 1024, max_clock=n + 256)
        out = [torch.full((n,), -1, dtype=d, device="cuda") for d in (torch.int32, torch.int32, torch.int64, torch.int64)]
        K.klpm_debug_set("list_max_windows", limit)
        try:
            K.klpm_run(tree, d_qt, d_qo, arr, params, *out)
            status, detail = K.rt_sync_status(tree), K.rt_status_detail(tree)
        finally:
            K.klpm_debug_set("list_max_windows", -1)
        got.append((status, detail, [o.cpu().numpy() for o in out]))
        K.rt_destroy(tree)
    (status, detail, cut), (ok, _, full) = got
    assert status == K.RT_ERR_LIMIT and detail == 118 and ok == 0
    charged = cut[1] >= 0
    before = int(charged.sum())                             # decisions made while arrivals were pending
    assert (before == 0) == (start == 50) and before < n
    assert np.array_equal(np.sort(full[0][:before]), np.flatnonzero(charged))
    assert np.array_equal(cut[0][:before], full[0][:before])
    for c, f in zip(cut[1:], full[1:]):
        assert np.array_equal(c[charged], f[charged]) and (c[~charged] == -1).all()


@pytest.mark.parametrize("smem_kb", [0, 51, 50])
@pytest.mark.parametrize("k", [2, 3, 8])
def test_changed_keys_are_looked_for_beside_a_commit(K, smem_kb, k):
    """A third of the prompts come in pairs, so a key grows every few decisions and waits in the tournament.  A step that takes such a key
    looks through its block of 32 slots while the others commit the batch before it, of which the oldest slots lie in that very block.
    In 51 KiB the bitmap of processed slots is in shared memory and that of changed keys is not, in 50 neither is."""
    n = 6000
    rng = np.random.RandomState(k)
    trunk = rng.randint(0, 30000, size=300).tolist()
    prompts = []
    while len(prompts) < n:
        m, own = rng.randint(1, 300), 100_000 + len(prompts)
        more = rng.randint(0, 30000, size=rng.randint(0, 8)).tolist()
        prompts += [trunk[:m] + [own] + more + [90_000 + i] for i in range(2 if rng.rand() < 0.2 else 1)]
    prompts = [prompts[i] for i in rng.permutation(len(prompts))[:n]]
    ct, co = W.to_csr([trunk + [7]])
    qt, qo = W.to_csr(prompts)
    d_qt, d_qo = qt.cuda(), qo.cuda()
    arr = torch.arange(n, dtype=torch.int64).cuda()
    tree = K.rt_build(ct.cuda(), co.cuda(), max_nodes=2 * n + 64, max_pool_tokens=ct.numel() + qt.numel() + 8 * n + 64, max_clock=n + 64)
    K.rt_checkpoint(tree)
    got = []
    for one_by_one in (1, 0, 0, 0):                         # (one order of the threads may go well)
        K.rt_rollback(tree)
        out = [torch.full((n,), -1, dtype=d, device="cuda") for d in (torch.int32, torch.int32, torch.int64, torch.int64)]
        K.klpm_debug_set("run_one_by_one", one_by_one)
        K.klpm_debug_set("fast_smem_kb", smem_kb)
        try:
            K.klpm_run(tree, d_qt, d_qo, arr, K.make_params(K.POLICY_KLPM, k, 0, 1, n), *out)
            assert K.rt_sync_status(tree) == 0
        finally:
            K.klpm_debug_set("run_one_by_one", -1)
            K.klpm_debug_set("fast_smem_kb", -1)
        got.append(out)
    assert K.rt_debug_counters(tree)["single_decisions"] > n // 10
    for out in got[1:]:
        for a, b in zip(got[0], out):
            assert torch.equal(a, b)
    K.rt_destroy(tree)


def paired_queue(n, low, share, seed, depth=400):
    """Match lengths spread over one cached trunk; of the prompts whose length is in the lowest part `low` a part `share` come in pairs that
    go on together for one to three tokens."""
    rng = np.random.RandomState(seed)
    trunk = rng.randint(0, 30000, size=depth).tolist()
    prompts = []
    while len(prompts) < n:
        m, own = rng.randint(1, depth), 100_000 + len(prompts)
        if m < low * depth and rng.rand() < share / (2 - share):
            more = [own] + rng.randint(0, 30000, size=rng.randint(0, 3)).tolist()
            prompts += [trunk[:m] + more + [90_000], trunk[:m] + more + [90_001]]
        else:
            prompts.append(trunk[:m] + [own])
    return trunk + [7], [prompts[i] for i in rng.permutation(len(prompts))[:n]]


@pytest.mark.parametrize("n, low, share, ks, smem_kb", [(9000, 0.25, 0.12, (2, 3), 0), (9000, 0.25, 0.1, (3, 4), 52), (20000, 0.1, 0.12, (4, 8), 0),
                                                        (20000, 0.1, 0.13, (4,), 55), (30000, 0.07, 0.13, (3, 8), 0)])
@pytest.mark.parametrize("pending", [False, True])
def test_groups_of_two_inside_the_rounds(K, n, low, share, ks, smem_kb, pending):
    """Up to 280 prompts of pairs a window: their decisions are made by the rounds.  They sit at the end of the key list, so that keys which
    have grown wait there in numbers, more at a time than the 64 that find a thread.  `pending`: a fifth of the queue is still to arrive
    as the loop starts, and the rounds go on from where that leaves the bitmaps.  With less shared memory they live in global memory."""
    trunk, prompts = paired_queue(n, low, share, n)
    ct, co = W.to_csr([trunk])
    qt, qo = W.to_csr(prompts)
    d_qt, d_qo = qt.cuda(), qo.cuda()
    late = n // 5 if pending else 0
    arr = torch.cat([torch.zeros(n - late, dtype=torch.int64), torch.arange(1, late + 1, dtype=torch.int64) // 8]).cuda()
    tree = K.rt_build(ct.cuda(), co.cuda(), max_nodes=2 * n + 64, max_pool_tokens=ct.numel() + qt.numel() + 8 * n + 64, max_clock=n + 64)
    K.rt_checkpoint(tree)
    for k in ks:
        got = []
        for one_by_one in (1, 0):
            K.rt_rollback(tree)
            out = [torch.full((n,), -1, dtype=d, device="cuda") for d in (torch.int32, torch.int32, torch.int64, torch.int64)]
            K.klpm_debug_set("run_one_by_one", one_by_one)
            K.klpm_debug_set("fast_smem_kb", smem_kb)
            try:
                K.klpm_run(tree, d_qt, d_qo, arr, K.make_params(K.POLICY_KLPM, k, 0, 1, 0), *out)
                assert K.rt_sync_status(tree) == 0
            finally:
                K.klpm_debug_set("run_one_by_one", -1)
                K.klpm_debug_set("fast_smem_kb", -1)
            got.append(out)
        for a, b in zip(*got):
            assert torch.equal(a, b), k
        c = K.rt_debug_counters(tree)
        assert c["lane_decisions"] >= 40, c
    K.rt_destroy(tree)


def replicas(n, seed, distinct):
    """n prompts of which every one is asked for several times, in random order, and the one-by-one loop's answer needs no cache."""
    rng = np.random.RandomState(seed)
    base = [rng.randint(0, 30000, size=rng.randint(20, 60)).tolist() for _ in range(distinct)]
    return [base[i] for i in rng.permutation(np.arange(n) % distinct)]


def run_both_ways(K, prompts, cached, params, settings=()):
    """The grouped loop's and the one-by-one loop's outputs, and the grouped loop's counters; everybody waits as it starts."""
    n = len(prompts)
    qt, qo = W.to_csr(prompts)
    ct, co = W.to_csr(cached)
    d_qt, d_qo, arr = qt.cuda(), qo.cuda(), torch.zeros(n, dtype=torch.int64).cuda()
    cap = dict(max_nodes=2 * (n + len(cached)) + 64, max_pool_tokens=ct.numel() + qt.numel() + 8 * (n + len(cached)) + 64, max_clock=n + len(cached) + 64)
    got = []
    for one_by_one in (1, 0):
        tree = K.rt_build(ct.cuda(), co.cuda(), **cap) if cached else K.rt_create(**cap)
        out = [torch.full((n,), -1, dtype=d, device="cuda") for d in (torch.int32, torch.int32, torch.int64, torch.int64)]
        K.klpm_debug_set("run_one_by_one", one_by_one)
        for name, value in settings:
            K.klpm_debug_set(name, value)
        try:
            K.klpm_run(tree, d_qt, d_qo, arr, params, *out)
            assert K.rt_sync_status(tree) == 0
        finally:
            K.klpm_debug_set("run_one_by_one", -1)
            for name, _ in settings:
                K.klpm_debug_set(name, -1)
        got.append(out)
        counters = K.rt_debug_counters(tree)
        K.rt_destroy(tree)
    return got[1], got[0], counters


@pytest.mark.parametrize("k", [2, 4])
def test_a_changed_key_is_taken_without_a_look_at_every_lane(K, k):
    """Queues below 8,192 have no lanes: a step that takes a key from the tournament used to go through all 128 of them per block (17,000
    to 22,000 cycles a step instead of 6,000)."""
    got, want, c = run_both_ways(K, replicas(1200, k, 300), [], K.make_params(K.POLICY_KLPM, k))
    for a, b in zip(got, want):
        assert torch.equal(a, b)
    assert c["single_decisions"] > 1000 and c["cycles_single"] < 10_000 * c["single_decisions"], c


@pytest.mark.parametrize("smem_kb", [0, 51, 50])
@pytest.mark.parametrize("policy, k", [(2, 2), (2, 4), (2, 40), (1, 1), (0, 1)])
def test_windows_are_left_where_most_decisions_are_steps(K, policy, k, smem_kb):
    """Prompts that are asked for several times each: most decisions touch a group or a changed key, and one warp makes them one after the
    other (as steps between batches of a window they took three to ten times as long).  Where such prompts are a part of the queue only,
    windows are taken up again.  51 and 50 KiB of shared memory: some, all bitmaps in global memory."""
    n = 3000
    got, want, c = run_both_ways(K, replicas(n, k, n // 4), [], K.make_params(policy, k), [("fast_smem_kb", smem_kb)])
    for a, b in zip(got, want):
        assert torch.equal(a, b)
    assert c["stretch_decisions"] > n // 2, c
    rng = np.random.RandomState(k)
    trunk = rng.randint(0, 30000, size=2000).tolist()
    plain = [trunk[:rng.randint(100, 1800)] + [100_000 + i] for i in range(5000)]
    again = [trunk[:m] + [200_000 + i, 7] for i in range(150) for m in [rng.randint(1800, 2000)] for _ in range(4)]      # first in both orders
    got, want, c = run_both_ways(K, again + plain, [trunk + [3]], K.make_params(policy, k), [("fast_smem_kb", smem_kb)])
    for a, b in zip(got, want):
        assert torch.equal(a, b)
    assert c["windows"] > 1 and c["iterated_decisions"] > 0, c


def test_windows_are_kept_where_nothing_is_grouped(K):
    """The two orders meet all the time on prompts of one match length, which is slow for one warp: without steps windows are never left."""
    prefixes = [[p] * 40 for p in range(8)]
    rng = np.random.RandomState(3)
    prompts = [prefixes[rng.randint(8)] + [1000 + i] for i in range(1000)]
    got, want, c = run_both_ways(K, prompts, [p + [999] for p in prefixes], K.make_params(K.POLICY_KLPM, 2))
    for a, b in zip(got, want):
        assert torch.equal(a, b)
    assert c["stretch_decisions"] == 0, c
