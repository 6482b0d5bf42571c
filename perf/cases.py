"""What the performance of this library is measured on: calls that a user's program makes, over the sizes it makes them at.

Every case is one pass through the public entry points (paper_2502_04677_b200.binding).  The inputs are the seeded
streams of paper_2502_04677_b200.workloads -- the configurations that the tests and the benchmark use -- at their full
sizes and at smaller and odd ones.  Five kinds of work:

  tick        one step of an online scheduler: match the waiting queue against the cache and decide who goes next
  store       the prompts that were just served enter a cache that is full, least recently used leaves leave it
  drain       a queue is matched and scheduled to its end on a cache without a budget, then some prompts are asked again
  stream      queries arrive over time and are scheduled under a cache budget with LRU eviction
  replay      a known order is charged again under another attention cost, and in batches
  montecarlo  many small queues under the last-prompt cache (random arrival orders)

A pass that changes the tree begins with rt_rollback: that is how a program tries one queue several times (another k,
another policy) on one cache.  All results are whole numbers and the library promises them bit for bit, whatever the
order in which its threads run, so the tolerance is "exact".
"""
import math

import torch

from paper_2502_04677_b200 import workloads as W

POLICIES = {"fcfs": 0, "lpm": 1, "klpm": 2}
FILL = 12_000            # prompts that went through the cache before a tick, a store: five times what its budget holds
QUEUE = 32               # prompts per queue of the Monte-Carlo, four per user context of 96 tokens, 32 tokens of their own
USER, DOC, REPLICAS = 96, 32, 4


def listed():
    return [
        # a lightly loaded server decides who goes next: 32 waiting queries, a cache in steady state
        dict(name="tick_32", kind="tick", queries=32, top=0),
        # the same under load, with the candidates for the following turns
        dict(name="tick_4001", kind="tick", queries=4001, top=3),
        # a served batch of 16 prompts enters the full cache
        dict(name="store_16", kind="store", queries=16),
        # the smallest configuration: 1,000 waiting queries on 8 short shared prefixes
        dict(name="drain_tiny", kind="drain", recipe="tiny", queries=1000, policy="klpm", k=2, ties=False, rate=False, attn=0),
        # the prefix-to-prompt ratio experiment: Poisson arrivals on an empty cache, random tie-breaking, longest match first
        dict(name="drain_arrivals", kind="drain", recipe="ratio", queries=2000, policy="lpm", k=1, ties=True, rate=False, attn=0),
        # a backlog over 64 long shared prefixes
        dict(name="drain_medium", kind="drain", recipe="medium", queries=32_768, policy="klpm", k=4, ties=False, rate=False, attn=0),
        # three levels of sharing, a tree of a million prompts, the hit-rate reading of the score, attention cost
        dict(name="drain_hierarchical", kind="drain", recipe="hierarchical", queries=65_536, policy="klpm", k=4, ties=False, rate=True,
             attn=1),
        # the largest configuration: 8.7 GB of query tokens against 4 M nodes, mismatches deep inside long edges
        dict(name="drain_adversarial", kind="drain", recipe="adversarial", queries=262_144, policy="klpm", k=4, ties=False, rate=False,
             attn=0),
        # ten minutes of arrivals on a cold cache with a budget of 50 M tokens
        dict(name="stream_cold", kind="stream", queries=120_000, policy="klpm", k=4, warm=False, attn=0),
        # one minute on a cache in steady state, longest match first, an odd number of queries
        dict(name="stream_warm", kind="stream", queries=12_007, policy="lpm", k=1, warm=True, attn=0),
        # a schedule that is known is charged again with attention cost, and in batches of 8
        dict(name="replay_8191", kind="replay", recipe="medium", queries=8191, k=4, batch=8),
        # random arrival orders of 32 prompts each, as the analysis of k-LPM averages over
        dict(name="montecarlo_65536", kind="montecarlo", queues=65_536, policy="klpm", k=4, ties=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["tick", "store", "drain", "drain", "drain", "stream", "replay", "montecarlo"])
    policy = rng.choice(["klpm", "klpm", "lpm", "fcfs"])
    k = rng.choice([1, 2, 3, 4, 8]) if policy == "klpm" else 1
    if kind == "tick":
        return dict(kind=kind, queries=_log(rng, 1, 8192), top=rng.choice([0, 0, 1, 3, 7]))
    if kind == "store":
        return dict(kind=kind, queries=_log(rng, 1, 64))
    if kind == "drain":
        recipe = rng.choice(["tiny", "ratio", "medium", "hierarchical", "adversarial"])
        lo, hi = {"tiny": (16, 2000), "ratio": (16, 2000), "medium": (64, 32_768), "hierarchical": (256, 65_536),
                  "adversarial": (256, 131_072)}[recipe]
        return dict(kind=kind, recipe=recipe, queries=_log(rng, lo, hi), policy=policy, k=k, ties=rng.random() < 0.25,
                    rate=rng.random() < 0.25, attn=rng.choice([0, 0, 1]))
    if kind == "stream":
        return dict(kind=kind, queries=_log(rng, 200, 50_000), policy=policy, k=k, warm=rng.random() < 0.5, attn=rng.choice([0, 0, 1]))
    if kind == "replay":
        recipe = rng.choice(["tiny", "medium", "hierarchical"])
        return dict(kind=kind, recipe=recipe, queries=_log(rng, 64, 2000 if recipe == "tiny" else 32_768), k=rng.choice([1, 2, 4, 8]),
                    batch=rng.choice([1, 8, 32]))
    return dict(kind=kind, queues=_log(rng, 64, 65_536), policy=policy, k=k, ties=rng.random() < 0.5)


def _workload(recipe, queries, seed):
    """The named configuration with that many queries (its other counts in proportion, its lengths as they are)."""
    if recipe == "tiny":
        return W.tiny(seed=seed, n_queries=queries, n_prefill=2 * queries)
    if recipe == "ratio":
        return W.prefix_ratio(3000, 3000, seed=seed, n=queries)
    maker, full = {"medium": (W.medium, 32_768), "hierarchical": (W.hierarchical, 65_536), "streaming": (W.streaming, 120_000),
                   "adversarial": (W.adversarial, 262_144)}[recipe]
    return maker(seed=seed, scale=(queries + 0.5) / full)


def _distinct(prompts):
    """At most this many different tokens: every stream window once, at its longest."""
    total, before = 0, None
    for key, end in zip(prompts.seg_key, prompts.seg_end):
        length = end if before is None else end - before
        uniq, inv = torch.unique(key, return_inverse=True)
        total += int(torch.zeros(uniq.numel(), dtype=torch.int64).scatter_reduce_(0, inv, length, "amax").sum())
        before = end
    return total


def _csr(prompts, device):
    tok, off = prompts.materialize(device)
    return tok, off.to(device)


def _filled_tree(w, device):
    """A cache without a budget that holds the configuration's prompts, with room for its queries, and a checkpoint."""
    from paper_2502_04677_b200 import binding as K
    n = w.prefill.n + w.queries.n
    tree = K.rt_create(max_nodes=2 * n + 64, max_pool_tokens=_distinct(w.prefill) + _distinct(w.queries) + 8 * n + 1024, vocab=w.vocab,
                       max_clock=n + 64)
    ends = torch.cumsum(w.prefill.lengths, 0)
    a = 0
    while a < w.prefill.n:                              # about a billion tokens at a time
        limit = (int(ends[a - 1]) if a else 0) + (1 << 30)
        b = max(a + 1, int(torch.searchsorted(ends, torch.tensor(limit), right=True)))
        tok, off = w.prefill.materialize(device, a, b)
        K.rt_insert(tree, tok, off.to(device))
        a = b
    K.rt_checkpoint(tree)
    if K.rt_sync_status(tree) != 0:
        raise RuntimeError("the cache could not be filled")
    return tree


def _budget_tree(w, before, device):
    """A cache with the configuration's budget through which its first `before` prompts have gone in arrival order, and a checkpoint."""
    from paper_2502_04677_b200 import binding as K
    n = w.queries.n
    tree = K.rt_create(max_nodes=2 * (n + before) + 64, max_pool_tokens=2 * w.queries.total_tokens() + 8 * (n + before) + 1024,
                       budget_tokens=w.budget_tokens, vocab=w.vocab, max_clock=n + before + 64)
    if before:
        first = w.queries.select(torch.arange(before))
        tok, off = _csr(first, device)
        out = [torch.zeros(before, dtype=t, device=device) for t in (torch.int32, torch.int32, torch.int64)]
        K.klpm_run(tree, tok, off, w.arrivals[:before].to(device), K.make_params(K.POLICY_FCFS), *out)
    K.rt_checkpoint(tree)
    if K.rt_sync_status(tree) != 0:
        raise RuntimeError("the cache could not be filled")
    return tree


def _asked_again(w, device):
    """Every sixteenth prompt of the queue, as it comes back after the queue has been served."""
    idx = torch.arange(0, w.queries.n, 16)
    tok, off = _csr(w.queries.select(idx), device)
    return dict(tok=tok, off=off, m=torch.zeros(idx.numel(), dtype=torch.int32, device=device),
                at=torch.zeros(idx.numel(), dtype=torch.int32, device=device))


def _outputs(n, device):
    return dict(order=torch.zeros(n, dtype=torch.int32, device=device), uncached=torch.zeros(n, dtype=torch.int32, device=device),
                ttft=torch.zeros(n, dtype=torch.int64, device=device), done=torch.zeros(n, dtype=torch.int64, device=device))


def _params(K, case, start):
    # attention cost of one tick per 4,096 tokens of the prompt, in units of 1/4096 tick
    c_num, c_den = (1, 4096) if case.get("attn") else (0, 1)
    return K.make_params(POLICIES[case.get("policy", "klpm")], case.get("k", 1), c_num, c_den, start)


def prepare(case, seed):
    from paper_2502_04677_b200 import binding as K
    device = torch.device("cuda", torch.cuda.current_device())
    kind = case["kind"]
    s = dict(case=case, K=K)
    if kind in ("tick", "store"):
        n = case["queries"]
        w = _workload("streaming", FILL + n, seed)
        s["tree"] = _budget_tree(w, FILL, device)
        s["tok"], s["off"] = _csr(w.queries.select(torch.arange(FILL, FILL + n)), device)
        s["m"] = torch.zeros(n, dtype=torch.int32, device=device)
        if kind == "store":
            s["new"] = torch.zeros(n, dtype=torch.int32, device=device)
            return s
        s["arrival"] = w.arrivals[FILL:].to(device)
        s["waiting"] = torch.ones(n, dtype=torch.uint8, device=device)
        s["pick"] = torch.zeros(1, dtype=torch.int32, device=device)
        s["next"] = torch.zeros(max(1, case["top"]), dtype=torch.int32, device=device)
        s["params"] = K.make_params(K.POLICY_KLPM, 4)
        return s
    if kind == "montecarlo":
        q = case["queues"]
        g = torch.Generator().manual_seed(seed)
        i = torch.arange(QUEUE, device=device)
        one = torch.zeros(QUEUE, USER + DOC, dtype=torch.int32, device=device)
        one[:, 0] = (1 + i % (QUEUE // REPLICAS)).to(torch.int32)
        one[:, USER] = (1 + QUEUE // REPLICAS + i).to(torch.int32)
        s["tok"] = one.reshape(-1).repeat(q)
        s["off"] = torch.arange(q * QUEUE + 1, dtype=torch.int64, device=device) * (USER + DOC)
        sigma = torch.argsort(torch.rand(q, QUEUE, generator=g), dim=1).to(device) + 1
        s["arrival"] = (sigma * 2).reshape(-1).to(torch.int64)
        s["prio"] = torch.randint(0, 1 << 30, (q * QUEUE,), generator=g, dtype=torch.int64).to(device) if case["ties"] else None
        s["queues"] = (torch.arange(q + 1, dtype=torch.int64, device=device) * QUEUE).to(torch.int32)
        s["out"] = _outputs(q * QUEUE, device)
        s["params"] = _params(K, case, 2 * QUEUE)
        return s
    n = case["queries"]
    if kind == "stream":
        w = _workload("streaming", n, seed)
        s["tree"] = _budget_tree(w, n if case["warm"] else 0, device)
    else:
        w = _workload(case["recipe"], n, seed)
        n = w.queries.n
        s["tree"] = _filled_tree(w, device)
    s["tok"], s["off"] = _csr(w.queries, device)
    s["arrival"] = w.arrivals.to(device)
    s["params"] = _params(K, case, w.start_tick)
    s["out"] = _outputs(n, device)
    s["again"] = _asked_again(w, device)
    if kind == "drain":
        s["m"] = torch.zeros(n, dtype=torch.int32, device=device)
        s["state"] = K.match_state_buffer(n, device)
        g = torch.Generator().manual_seed(seed)
        s["prio"] = torch.randint(0, 1 << 30, (n,), generator=g, dtype=torch.int64).to(device) if case["ties"] else None
    if kind == "replay":
        o = s["out"]
        K.klpm_run(s["tree"], s["tok"], s["off"], s["arrival"], s["params"], o["order"], o["uncached"], o["ttft"], o["done"])
        s["params"] = _params(K, dict(case, attn=1), w.start_tick)
        s["ttft_b"], s["done_b"] = torch.zeros_like(o["ttft"]), torch.zeros_like(o["done"])
    return s


def run(s):
    K, case, kind = s["K"], s["case"], s["case"]["kind"]
    if kind == "tick":
        K.rt_match_batch(s["tree"], s["tok"], s["off"], s["m"])
        K.klpm_select(s["m"], s["arrival"], s["waiting"], 1, s["params"], s["pick"])
        if not case["top"]:
            return [s["m"], s["pick"]]
        K.klpm_select_topk(s["m"], s["arrival"], s["waiting"], s["next"])
        return [s["m"], s["pick"], s["next"]]
    if kind == "store":
        K.rt_rollback(s["tree"])
        K.rt_insert(s["tree"], s["tok"], s["off"], s["new"])
        K.rt_match_batch(s["tree"], s["tok"], s["off"], s["m"])
        return [s["new"], s["m"]]
    o = s["out"]
    if kind == "montecarlo":
        K.klpm_run_last_only_batch(s["tok"], s["off"], s["arrival"], s["prio"], s["queues"], s["params"], o["order"], o["uncached"],
                                   o["ttft"], o["done"])
        return o
    K.rt_rollback(s["tree"])
    again = s["again"]
    out = dict(o, again=again["m"], at=again["at"])
    if kind == "drain":
        K.rt_match_batch_ex(s["tree"], s["tok"], s["off"], s["m"], None, None, s["state"])
        K.klpm_run_ex(s["tree"], s["tok"], s["off"], s["arrival"], s["params"], s["prio"], 1 if case["rate"] else 0, o["order"],
                      o["uncached"], o["ttft"], o["done"], s["state"])
        out["m"] = s["m"]
    elif kind == "stream":
        K.klpm_run(s["tree"], s["tok"], s["off"], s["arrival"], s["params"], o["order"], o["uncached"], o["ttft"], o["done"])
    else:
        K.klpm_replay(s["tree"], o["order"], s["tok"], s["off"], s["arrival"], s["params"], o["uncached"], o["ttft"], o["done"])
        K.klpm_batch_times(o["order"], s["arrival"], o["done"], case["batch"], s["ttft_b"], s["done_b"])
        out.update(ttft_b=s["ttft_b"], done_b=s["done_b"])
    # what the cache holds now, as the next queries find it: matched tokens, and how far into the node the match ends
    K.rt_match_batch(s["tree"], again["tok"], again["off"], again["m"], None, again["at"])
    return out


def work(case):
    """Bytes a pass cannot do without.  A prompt that is matched: its tokens up to the first one that is not cached.  One that
    is stored: all its tokens read once, those that were not cached written once.  What it is compared with: every shared
    stretch once.  Per query: offset, arrival (16) and the results.  There is no arithmetic worth counting."""
    kind = case["kind"]
    if kind == "montecarlo":
        n = case["queues"] * QUEUE
        return {"bytes": float(n * (4 * (USER + DOC) + 16 + (8 if case["ties"] else 0) + 24) + 4 * case["queues"]), "flops": 0.0}
    if kind in ("tick", "store"):
        w = _workload("streaming", FILL + case["queries"], 0)
        q = w.queries.select(torch.arange(FILL, FILL + case["queries"]))
    else:
        w = _workload("streaming" if kind == "stream" else case["recipe"], case["queries"], 0)
        q = w.queries
    n, total = q.n, q.total_tokens()
    shared = int(q.seg_end[-2].sum())
    once = _distinct(W.SegmentedPrompts(q.vocab, q.seg_key[:-1], q.seg_end[:-1]))
    if kind == "tick":
        return {"bytes": float(4 * (shared + n + once) + n * (8 + 8 + 1 + 4) + 4 * (1 + case["top"])), "flops": 0.0}
    if kind == "store":
        return {"bytes": float(4 * (total + (total - shared) + once) + n * (8 + 8)), "flops": 0.0}
    stored = total - shared if case.get("recipe") != "ratio" and kind != "stream" else _distinct(q)
    asked = n // 16 + 1
    more = 8 if case.get("ties") else 0
    more += {"drain": 4, "stream": 0, "replay": 16}[kind]
    again = 4 * total * asked // max(1, n)                 # the prompts that are asked again are compared in full
    return {"bytes": float(4 * (total + stored + once) + n * (16 + 24 + more) + again + 16 * asked), "flops": 0.0}


def tolerance(case):
    return "exact"
