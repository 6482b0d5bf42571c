"""rt_insert one prompt after the other: long calls (several parts), inside a stream capture, and calls that end early."""
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


def some_prompts(n):
    a, _ = W.random_small_queue(5, n, vocab=2, max_len=14)
    b, _ = W.random_small_queue(6, n, vocab=40, max_len=9)
    return [x + y if i % 3 else y + x for i, (x, y) in enumerate(zip(a, b))]


def same_tree(K, tree, ot, prompts):
    st, want = K.rt_stats(tree), ot.stats()
    for key in ("n_nodes", "tokens", "clock", "evictions"):
        assert st[key] == want[key], key
    qt, qo = W.to_csr(prompts)
    m = torch.zeros(len(prompts), dtype=torch.int32, device="cuda")
    K.rt_match_batch(tree, qt.cuda(), qo.cuda(), m)
    assert np.array_equal(m.cpu().numpy(), ot.match(qt.numpy(), qo.numpy()))


@pytest.mark.parametrize("budget", [0, 2000])
@pytest.mark.parametrize("n", [1023, 1024, 1025, 2600])
def test_several_parts(K, budget, n):
    prompts = some_prompts(n)
    pt, po = W.to_csr(prompts)
    tree = K.rt_create(max_nodes=2 * n + 16, max_pool_tokens=pt.numel() + 8 * n + 16, budget_tokens=budget, max_clock=n + 16)
    new = torch.full((n,), -7, dtype=torch.int32, device="cuda")
    K.rt_insert(tree, pt.cuda(), po.cuda(), new)
    assert K.rt_sync_status(tree) == 0
    ot = oracle.OracleTree(budget)
    assert np.array_equal(new.cpu().numpy(), ot.insert(pt.numpy(), po.numpy()))
    same_tree(K, tree, ot, prompts)


@pytest.mark.parametrize("budget", [0, 300])
def test_first_call_inside_a_capture(K, budget):
    """The call only enqueues work: a program may capture it, on a tree nothing was stored in before."""
    prompts = some_prompts(40)
    pt, po = W.to_csr(prompts)
    tok, off = pt.cuda(), po.cuda()
    tree = K.rt_create(max_nodes=400, max_pool_tokens=2 * pt.numel() + 800, budget_tokens=budget, max_clock=200)
    new = torch.full((40,), -7, dtype=torch.int32, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        K.rt_insert(tree, tok, off, new)
    ot = oracle.OracleTree(budget)
    for _ in range(2):                                       # (the second time on the tree the first left)
        graph.replay()
        torch.cuda.synchronize()
        assert np.array_equal(new.cpu().numpy(), ot.insert(pt.numpy(), po.numpy()))
    assert K.rt_sync_status(tree) == 0
    same_tree(K, tree, ot, prompts)


@pytest.mark.parametrize("room", [700, 1024, 1500])
def test_no_room_left_in_one_of_the_parts(K, room):
    """The prompts before the one there is no room for stay, nothing behind it is stored or reported."""
    n = 2600
    prompts = some_prompts(n)
    pt, po = W.to_csr(prompts)
    tree = K.rt_create(max_nodes=2 * n + 16, max_pool_tokens=pt.numel() + 8 * n + 16, max_clock=room)
    new = torch.full((n,), -7, dtype=torch.int32, device="cuda")
    K.rt_insert(tree, pt.cuda(), po.cuda(), new)
    assert K.rt_sync_status(tree) == -2
    stored = K.rt_stats(tree)["clock"]
    assert room - 2 <= stored <= room + 2
    ot = oracle.OracleTree(0)
    want = ot.insert(*[x.numpy() for x in W.to_csr(prompts[:stored])])
    got = new.cpu().numpy()
    assert np.array_equal(got[:stored], want) and (got[stored:] == -7).all()
    same_tree(K, tree, ot, prompts)


@pytest.mark.parametrize("budget", [0, 2000])
@pytest.mark.parametrize("n,at", [(5, 0), (40, 17), (1500, 1023), (2600, 1030)])
def test_offsets_that_are_not_prompts(K, budget, n, at):
    """A prompt of negative length ends the call there: what is before it is stored, nothing behind it is looked at (its offsets may be
    anything), and the status says which check it was."""
    prompts = some_prompts(n)
    pt, po = W.to_csr(prompts)
    bad = po.clone()
    bad[at + 1] = bad[at] - 1
    bad[at + 2:] = torch.tensor([-5, 1 << 40, 7, -(1 << 40)], dtype=torch.int64).repeat(n)[:n - at - 1]
    tree = K.rt_create(max_nodes=2 * n + 16, max_pool_tokens=pt.numel() + 8 * n + 16, budget_tokens=budget, max_clock=n + 16)
    new = torch.full((n,), -7, dtype=torch.int32, device="cuda")
    K.rt_insert(tree, pt.cuda(), bad.cuda(), new)
    assert K.rt_sync_status(tree) == -1
    assert K.rt_status_detail(tree) == 108
    ot = oracle.OracleTree(budget)
    want = ot.insert(*[x.numpy() for x in W.to_csr(prompts[:at])]) if at else np.zeros(0, dtype=np.int32)
    got = new.cpu().numpy()
    assert np.array_equal(got[:at], want) and (got[at:] == -7).all()
    same_tree(K, tree, ot, prompts)
