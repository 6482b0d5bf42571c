"""Queues whose two pick orders -- longest match and arrival -- run side by side, so that nearly every pick of one is met by the
other: CTA-wide batches that are played through decision by decision, against the oracle."""
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


@pytest.mark.parametrize("n", [33, 1000, 1025, 3100])
@pytest.mark.parametrize("jitter", [0, 3, 60])
def test_orders_side_by_side(K, n, jitter):
    """Match lengths fall with the arrival order up to a jitter (0: all equal, ties go by arrival), and a few prompts share their
    continuation (groups), so that batches also stop at decisions which need the one-at-a-time path."""
    rng = np.random.RandomState(n + jitter)
    trunk = rng.randint(0, 50_000, size=4000).tolist()
    prompts = []
    for i in range(n):
        depth = 50 if jitter == 0 else max(1, 3500 - i + int(rng.randint(-jitter, jitter + 1)))
        own = 50_000 + i if rng.randint(0, 40) else 50_000 + max(0, i - int(rng.randint(1, 30)))
        prompts.append(trunk[:depth] + [own] + [int(x) for x in rng.randint(0, 3, size=rng.randint(0, 4))])
    ct, co = W.to_csr([trunk])
    qt, qo = W.to_csr(prompts)
    arr = np.arange(n, dtype=np.int64)
    for k in (2, 3, 5, 40, 1500):
        tree = K.rt_build(ct.cuda(), co.cuda(), max_nodes=2 * n + 64, max_pool_tokens=ct.numel() + qt.numel() + 8 * n + 64, max_clock=n + 64)
        out = [torch.full((n,), -1, dtype=d, device="cuda") for d in (torch.int32, torch.int32, torch.int64, torch.int64)]
        K.klpm_run(tree, qt.cuda(), qo.cuda(), torch.from_numpy(arr).cuda(), K.make_params(K.POLICY_KLPM, k, 1, 3, n), *out)
        assert K.rt_sync_status(tree) == 0
        ot = oracle.OracleTree(0)
        ot.insert(ct.numpy(), co.numpy())
        want = oracle.schedule(qt.numpy(), qo.numpy(), arr, oracle.POLICY_KLPM, k, 1, 3, n, oracle.CACHE_TREE, oracle.TIER_UPDATE, ot)
        for g, w in zip(out, want):
            assert np.array_equal(g.cpu().numpy(), w), k
