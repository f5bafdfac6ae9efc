"""The library's lookup paths at the sizes they are used at.

Every case is one pass through a public entry point over data resident as a
user's program would have it: built trees (and models, forests, servers),
queries and outputs on the GPU, or in page-locked host memory where the entry
point takes host buffers.  The listed cases are the configured workloads (the
4096-key uint32 tree, the 2^24-key uint64 tree, the paper's 32-byte-key tree,
the 10,000-batch work list, the learned search over lognormal keys, the served
request stream) and sizes between them; `draw` gives others of the same
ranges.  Keys, values and queries are drawn on the GPU from the seed, by the
recipes of the package's workloads module (uniform and lognormal-mixture keys,
uniform and Zipf queries, log-uniform batch sizes, geometric request sizes);
values are random words.  All outputs are stored integers and found flags, so
they have no floating-point reference.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2604_21117_gb300 import btree as bt
from paper_2604_21117_gb300 import workloads as W


def listed():
    return [
        # The smallest configured search: a 4096-key uint32 tree at fanout 16,
        # 256 lookups, half of them misses.
        dict(name="lookup_256_u32", kind="lookup", n=4096, key_bits=32, val_bits=32, fanout=16, batch=256, hits=0.5,
             zipf=0.0),
        # A latency-sized batch on the large tree: 1024 lookups over 2^24
        # uint64 keys at fanout 32.
        dict(name="lookup_1024", kind="lookup", n=1 << 24, key_bits=64, val_bits=64, fanout=32, batch=1024, hits=0.9,
             zipf=0.0),
        # An ordinary batch of ragged size on a tree that the L2 holds.
        dict(name="lookup_50021", kind="lookup", n=1_000_000, key_bits=64, val_bits=64, fanout=32, batch=50_021,
             hits=0.9, zipf=0.0),
        # 32-bit keys and values at the widest fanout, the largest key count,
        # a skewed ragged batch.
        dict(name="lookup_300007_u32_zipf", kind="lookup", n=20_000_000, key_bits=32, val_bits=32, fanout=64,
             batch=300_007, hits=0.9, zipf=1.1),
        # The benchmark's headline: 2^20 lookups over 2^24 uint64 keys.
        dict(name="lookup_2p20", kind="lookup", n=1 << 24, key_bits=64, val_bits=64, fanout=32, batch=1 << 20,
             hits=0.9, zipf=0.0),
        # The paper's own tree (2^20 32-byte keys, fanout 16) at its batch of
        # 1000, and at 2^20.
        dict(name="bytes_1000", kind="bytes", n=1 << 20, prefix=0, fanout=16, batch=1000, hits=0.9),
        dict(name="bytes_2p20", kind="bytes", n=1 << 20, prefix=0, fanout=16, batch=1 << 20, hits=0.9),
        # One launch over a work list of 10,000 batches on four trees.
        dict(name="forest_10000", kind="forest", batches=10_000, fanout=32, hits=0.8, zipf=0.9, lane_queries=2,
             n0=1000, n1=100_000, n2=1_000_000, n3=20_000_000),
        # The learned search: piecewise-linear at 2^20 lookups, the MLP at a
        # latency-sized batch, over 2^24 lognormal keys.
        dict(name="learned_pl_2p20", kind="learned", model="pl", n=1 << 24, fanout=32, batch=1 << 20, hits=0.9),
        dict(name="learned_mlp_1024", kind="learned", model="mlp", n=1 << 24, fanout=32, batch=1024, hits=0.9),
        # Lookups from page-locked host buffers and back, one call.
        dict(name="host_2p20", kind="host", n=1 << 24, key_bits=64, val_bits=64, fanout=32, batch=1 << 20, hits=0.9,
             zipf=0.0),
        # A burst of requests through the serving loop over two trees.
        dict(name="serve_20000", kind="serve", requests=20_000, fanout=32, n0=1_000_000, n1=20_000_000, hits=0.9),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lookup"] * 6 + ["bytes", "forest", "learned", "host", "serve", "bytes"])
    fanout = rng.choice([8, 16, 32, 64])
    hits = round(rng.uniform(0.5, 0.95), 2)
    zipf = rng.choice([0.0, 0.0, 0.9, 1.1])
    if kind in ("lookup", "host"):
        key_bits = rng.choice([32, 64, 64])
        return dict(kind=kind, n=_log_int(rng, 10, 20_000_000), key_bits=key_bits, val_bits=rng.choice([32, 64]),
                    fanout=fanout, batch=_log_int(rng, 1, 1 << 20), hits=hits, zipf=zipf)
    if kind == "bytes":
        return dict(kind=kind, n=_log_int(rng, 10, 1 << 20), prefix=rng.choice([0, 0, 3, 12]), fanout=fanout,
                    batch=_log_int(rng, 1, 1 << 20), hits=hits)
    if kind == "forest":
        return dict(kind=kind, batches=_log_int(rng, 1, 10_000), fanout=fanout, hits=hits, zipf=zipf,
                    lane_queries=rng.choice([1, 2]), n0=_log_int(rng, 10, 10_000), n1=_log_int(rng, 1000, 200_000),
                    n2=_log_int(rng, 100_000, 2_000_000), n3=_log_int(rng, 1_000_000, 20_000_000))
    if kind == "learned":
        return dict(kind=kind, model=rng.choice(["pl", "mlp"]), n=_log_int(rng, 1000, 1 << 24), fanout=fanout,
                    batch=_log_int(rng, 1, 1 << 20), hits=hits)
    return dict(kind=kind, requests=_log_int(rng, 100, 20_000), fanout=fanout, n0=_log_int(rng, 1000, 1_000_000),
                n1=_log_int(rng, 1_000_000, 20_000_000), hits=hits)


# ------------------------------------------------------------------ inputs

_TOP = -(1 << 63)


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _words(g, size):
    """Uniform random 64-bit words (as int64)."""
    a = torch.randint(0, 1 << 32, (size,), generator=g, device="cuda", dtype=torch.int64)
    return (a << 32) | torch.randint(0, 1 << 32, (size,), generator=g, device="cuda", dtype=torch.int64)


def _distinct(g, n, some):
    """n distinct values of some(size), ascending as signed integers."""
    pool = torch.empty(0, dtype=torch.int64, device="cuda")
    while pool.numel() < n:
        need = n - pool.numel()
        pool = torch.unique_consecutive(torch.sort(torch.cat([pool, some(need + need // 16 + 16)])).values)
    if pool.numel() > n:
        keep = torch.randperm(pool.numel(), generator=g, device="cuda")[:n]
        pool = pool[torch.sort(keep).values]
    return pool


def _uniform_keys(g, n, bits):
    """n distinct uniform keys in unsigned order, as int64 bit patterns."""
    if bits == 32:
        return _distinct(g, n, lambda s: torch.randint(0, 1 << 32, (s,), generator=g, device="cuda",
                                                       dtype=torch.int64))
    return _distinct(g, n, lambda s: _words(g, s)) ^ _TOP


def _lognormal_keys(g, n):
    mu = torch.tensor([0.0, 1.0, 2.0], device="cuda", dtype=torch.float64)
    sigma = torch.tensor([1.0, 2.0, 0.5], device="cuda", dtype=torch.float64)

    def some(s):
        c = torch.randint(0, 3, (s,), generator=g, device="cuda")
        z = torch.randn(s, generator=g, device="cuda", dtype=torch.float64)
        return torch.exp(mu[c] + sigma[c] * z).mul(2.0**40).clamp(max=2.0**62).to(torch.int64)

    return _distinct(g, n, some)


def _picks(g, n, size, zipf):
    """Key ranks of `size` hits: uniform, or Zipf over a random key order."""
    if not zipf:
        return torch.randint(0, n, (size,), generator=g, device="cuda")
    cdf = torch.cumsum(torch.arange(1, n + 1, device="cuda", dtype=torch.float64).pow_(-zipf), 0)
    u = torch.rand(size, generator=g, device="cuda", dtype=torch.float64) * cdf[-1]
    return torch.randperm(n, generator=g, device="cuda")[torch.searchsorted(cdf, u).clamp(max=n - 1)]


def _queries(g, keys, size, hits, zipf, bits):
    miss = _words(g, size) if bits == 64 else torch.randint(0, 1 << 32, (size,), generator=g, device="cuda",
                                                            dtype=torch.int64)
    hit = torch.rand(size, generator=g, device="cuda") < hits
    return torch.where(hit, keys[_picks(g, keys.numel(), size, zipf)], miss)


def _narrow(a, bits):
    """int64 bit patterns as a device array of `bits`-bit words."""
    return a if bits == 64 else a.to(torch.int32)


def _host(a, bits):
    return _narrow(a, bits).cpu().numpy().view(np.uint64 if bits == 64 else np.uint32)


def _tree(g, keys, key_bits, val_bits, fanout):
    return bt.BTree(_host(keys, key_bits), _host(_words(g, keys.numel()), val_bits), fanout)


def _outputs(size, val_bits, **where):
    return (torch.empty(size, dtype=torch.int64 if val_bits == 64 else torch.int32, **where),
            torch.empty(size, dtype=torch.uint8, **where))


def _byte_rows(words):
    """(n, 32) bytes of (n, 4) words, each word's most significant byte first."""
    return words.contiguous().view(torch.uint8).view(-1, 4, 8).flip(2).reshape(-1, 32)


class _Server:
    """A server handle that ends with the state that holds it."""

    def __init__(self, trees):
        self.trees = trees
        self.handle = bt.bt_server_create([t.handle for t in trees], None, slots=8, max_batch=8192, deadline_us=50.0)

    def __del__(self):
        bt.bt_server_destroy(self.handle)


class _Forest:
    def __init__(self, trees, lane_queries):
        self.trees = trees
        self.handle = bt.bt_forest_create([t.handle for t in trees])
        # what the forest's autotuner chooses for such work lists: four warps
        # per block, nothing pinned, every level read through L1
        bt.bt_forest_set_launch(self.handle, 4, 0, lane_queries, 1)

    def __del__(self):
        bt.bt_forest_free(self.handle)


class _Model:
    def __init__(self, tree, model, n):
        self.tree = tree
        if model == "pl":
            self.handle = bt.bt_model_train(tree.handle, bt.BT_MODEL_PL, segments=256)
        else:
            self.handle = bt.bt_model_train(tree.handle, bt.BT_MODEL_MLP, h_init=W.mlp_init_params(5), steps=400,
                                            batch=16384, lr=2e-3, seed=6)

    def __del__(self):
        bt.bt_model_free(self.handle)


def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    s = dict(kind=kind)
    if kind in ("lookup", "host"):
        kb, vb, nq = case["key_bits"], case["val_bits"], case["batch"]
        keys = _uniform_keys(g, case["n"], kb)
        s["tree"] = tree = _tree(g, keys, kb, vb, case["fanout"])
        q = _narrow(_queries(g, keys, nq, case["hits"], case["zipf"], kb), kb)
        if kind == "lookup":
            s["q"] = q
            s["v"], s["f"] = _outputs(nq, vb, device="cuda")
            s["ws"], s["nb"] = tree.alloc_workspace(nq)
        else:
            s["q"] = q.cpu().pin_memory()
            s["v"], s["f"] = _outputs(nq, vb, pin_memory=True)
            s["ws"], s["nb"] = tree.alloc_workspace(nq, host=True)
    elif kind == "bytes":
        n, nq, p = case["n"], case["batch"], case["prefix"]
        words = _words(g, 4 * n).view(n, 4)
        words[:, 0] = _uniform_keys(g, n, 64)
        # `prefix` bytes that every key shares, before the distinct ones
        rows = _byte_rows(words)
        rows = torch.cat([rows[:1, 32 - p:].expand(n, p), rows[:, :32 - p]], 1).contiguous()
        vals = _host(_words(g, n), 64)
        s["tree"] = tree = bt.BTree(rows.cpu().numpy(), vals, case["fanout"])
        hit = torch.rand(nq, generator=g, device="cuda") < case["hits"]
        # misses share a random number of leading bytes with a stored key
        lead = torch.where(hit, 32, torch.randint(0, 17, (nq,), generator=g, device="cuda"))
        own = _byte_rows(_words(g, 4 * nq).view(nq, 4))
        s["q"] = torch.where(torch.arange(32, device="cuda") < lead[:, None], rows[_picks(g, n, nq, 0.0)],
                             own).contiguous()
        s["v"], s["f"] = _outputs(nq, 64, device="cuda")
        s["ws"], s["nb"] = tree.alloc_workspace(nq)
    elif kind == "learned":
        nq = case["batch"]
        keys = _lognormal_keys(g, case["n"])
        s["tree"] = tree = _tree(g, keys, 64, 64, case["fanout"])
        s["model"] = _Model(tree, case["model"], case["n"])
        s["q"] = _queries(g, keys, nq, case["hits"], 0.0, 64)
        s["v"], s["f"] = _outputs(nq, 64, device="cuda")
        s["ws"], s["nb"] = tree.alloc_workspace(nq)
    elif kind == "forest":
        nb = case["batches"]
        h = W.rng(seed)
        counts = h.permutation(W.log_uniform_batch_sizes(nb, seed=nb))  # the same total for every seed
        tids = h.integers(0, 4, size=nb)
        desc = np.zeros(nb, bt.BATCH_DESC_DTYPE)
        desc["tree"], desc["count"], desc["offset"] = tids, counts, np.cumsum(counts) - counts
        total = int(counts.sum())
        owner = torch.from_numpy(np.repeat(tids, counts)).cuda()
        q = torch.empty(total, dtype=torch.int64, device="cuda")
        trees = []
        for i in range(4):
            keys = _uniform_keys(g, case["n%d" % i], 64)
            trees.append(_tree(g, keys, 64, 64, case["fanout"]))
            mine = owner == i
            q[mine] = _queries(g, keys, int(mine.sum()), case["hits"], case["zipf"], 64)
        s["forest"] = _Forest(trees, case["lane_queries"])
        s["desc"], s["n"], s["q"] = torch.from_numpy(desc.view(np.uint8)).cuda(), nb, q
        s["v"], s["f"] = _outputs(total, 64, device="cuda")
        s["nb"] = bt.bt_forest_workspace_bytes(nb)
        s["ws"] = torch.empty(s["nb"], dtype=torch.uint8, device="cuda")
    else:
        nr = case["requests"]
        h = W.rng(seed)
        sizes = h.permutation(W.geometric_request_sizes(nr, seed=nr))  # the same total for every seed
        tids = h.integers(0, 2, size=nr).astype(np.uint32)
        total = int(sizes.sum())
        owner = torch.from_numpy(np.repeat(tids.astype(np.int64), sizes)).cuda()
        q = torch.empty(total, dtype=torch.int64, device="cuda")
        trees = []
        for i in range(2):
            keys = _uniform_keys(g, case["n%d" % i], 64)
            trees.append(_tree(g, keys, 64, 64, case["fanout"]))
            mine = owner == i
            q[mine] = _queries(g, keys, int(mine.sum()), case["hits"], 0.0, 64)
        s["server"] = _Server(trees)
        s["at"] = np.zeros(nr)  # all at once: the server sets the pace
        s["tree_of"], s["count"] = tids, sizes.astype(np.uint32)
        s["offset"] = (np.cumsum(sizes) - sizes).astype(np.uint64)
        s["q"] = q.cpu().numpy().view(np.uint64)
        s["v"], s["f"] = np.empty(total, np.uint64), np.empty(total, np.uint8)
    return s


def run(s):
    kind = s["kind"]
    if kind in ("lookup", "bytes"):
        t = s["tree"]
        bt.bt_search_batch(t.handle, s["q"], t.count(s["q"]), s["v"], s["f"], s["ws"], s["nb"])
    elif kind == "learned":
        bt.bt_learned_search_batch(s["tree"].handle, s["model"].handle, s["q"], s["q"].numel(), s["v"], s["f"],
                                   s["ws"], s["nb"])
    elif kind == "forest":
        bt.bt_forest_search(s["forest"].handle, s["desc"], s["n"], s["q"], s["v"], s["f"], s["ws"], s["nb"])
    elif kind == "host":
        bt.bt_search_batch_host(s["tree"].handle, s["q"], s["q"].numel(), s["v"], s["f"], s["ws"], s["nb"])
    else:
        bt.bt_server_run_trace(s["server"].handle, s["at"], s["tree_of"], s["count"], s["offset"], s["q"], s["v"],
                               s["f"])
        return s["v"].view(np.int64), s["f"]
    return s["v"], s["f"]


# -------------------------------------------------------------------- work

def _distinct_picks(n, draws, zipf):
    """Expected number of distinct keys among `draws` picks of n."""
    if n < 1 or draws <= 0:
        return 0.0
    if not zipf:
        return n * -math.expm1(draws * math.log1p(-1.0 / n)) if n > 1 else 1.0
    r = np.arange(1, n + 1, dtype=np.float64) ** -zipf
    return float(-np.expm1(draws * np.log1p(-np.minimum(r / r.sum(), 1 - 1e-12))).sum())


def _touched(n, nq, key_bytes, val_bytes, hits, zipf):
    """Bytes of the stored keys and values that a batch has to look at, in
    32-byte sectors: the sector of every distinct queried key (a miss has to
    see its neighbours) and of every hit's value."""
    keys = min(_distinct_picks(n, nq * hits, zipf) + nq * (1 - hits), float(n))
    sk, sv = math.ceil(n * key_bytes / 32), math.ceil(n * val_bytes / 32)
    vals = _distinct_picks(n, nq * hits, zipf)
    return 32.0 * (_distinct_picks(sk, keys, 0.0) + _distinct_picks(sv, vals, 0.0))


def work(case):
    kind = case["kind"]
    if kind in ("lookup", "host"):
        kb, vb = case["key_bits"] // 8, case["val_bits"] // 8
        nq = case["batch"]
        b = nq * (kb + vb + 1) + _touched(case["n"], nq, kb, vb, case["hits"], case["zipf"])
    elif kind == "bytes":
        nq = case["batch"]
        b = nq * (32 + 8 + 1) + _touched(case["n"], nq, 32, 8, case["hits"], 0.0)
    elif kind == "learned":
        nq = case["batch"]
        b = nq * (8 + 8 + 1) + _touched(case["n"], nq, 8, 8, case["hits"], 0.0)
    elif kind == "forest":
        mean = 1023.0 / math.log(1024.0)  # of the log-uniform batch sizes
        nq = case["batches"] * mean
        b = nq * (8 + 8 + 1) + sum(_touched(case["n%d" % i], nq / 4, 8, 8, case["hits"], case["zipf"])
                                   for i in range(4))
    else:
        nq = case["requests"] * 8.0  # the request sizes' mean
        b = nq * (8 + 8 + 1) + sum(_touched(case["n%d" % i], nq / 2, 8, 8, case["hits"], 0.0) for i in range(2))
    flops = 0.0
    if case.get("model") == "mlp":
        flops = nq * 2.0 * (32 + 32 * 32 + 32)
    return {"bytes": float(b), "flops": flops}
