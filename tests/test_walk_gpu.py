"""Batches searched as given through the walk index, against the CPU oracle
and against the partitioned descent, at the sizes where the index changes
shape: one entry, a full and an overfull top, one node more per level, ragged
last entries; for 32-byte keys also words that tie."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2604_21117_gb300 import workloads as W
from oracle import OracleTree
from oracle.bytes_keys import OracleBytesTree
import pins

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bt():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_21117_gb300 import build_lib
    build_lib.build()
    from paper_2604_21117_gb300 import btree
    return btree


def _same(tree, o, q):
    import torch
    ov, of, _, _ = o.search(q)
    for sb in (-1, 0, 12):  # the walk index twice, the partition and descent once
        v, f = tree.search(torch.from_numpy(np.ascontiguousarray(q)).cuda(), sort_bits=sb)
        assert np.array_equal(v.cpu().numpy().astype(np.uint64), ov)
        assert np.array_equal(f.cpu().numpy(), of)


# entries hold 32 / max(widths) keys; up to 2^12 entries the top alone, then
# one coded level of 17 children up to 2^12 segments, then two
@pytest.mark.parametrize("kw,vw,n", [
    (64, 64, 1), (64, 64, 4), (64, 64, 5), (64, 64, 4 * 4096), (64, 64, 4 * 4096 + 1), (64, 64, 4 * 17 * 4096),
    (64, 64, 4 * 17 * 4096 + 1), (64, 64, 4 * 289 * 700 + 3), (64, 32, 4 * 4096 + 2), (32, 64, 4 * 4096 + 1),
    (32, 32, 7), (32, 32, 8 * 4096), (32, 32, 8 * 4096 + 1), (32, 32, 8 * 17 * 4096), (32, 32, 8 * 17 * 4096 + 5)])
@pytest.mark.parametrize("nq", [1, 33, 152 * 1024 + 33])
def test_index_shape_boundaries(bt, kw, vw, n, nq):
    keys = W.uniform_keys(n, kw, seed=900 + n)
    vals = W.rng(901).integers(0, 2**vw, size=n, dtype=np.uint64).astype(W.key_dtype(vw))
    tree = bt.BTree(keys, vals, 16)
    o = OracleTree(keys, vals, 16, val_bits=vw)
    g = W.rng(902 + nq)
    probes = pins.probe_queries(keys, kw, g) if nq > 1000 else W.make_queries(keys, nq, 0.7, seed=nq, width_bits=kw)
    _same(tree, o, np.resize(probes, nq).astype(W.key_dtype(kw)))


def test_all_ones_key_stored_and_not(bt):
    top = 2**64 - 1
    for keys in ([1, 2, 3, top], [1, 2, 3, top - 1, top], [5], [top], [0, top]):
        keys = np.array(keys, np.uint64)
        tree = bt.BTree(keys, np.arange(10, 10 + keys.size, dtype=np.uint64), 8)
        o = OracleTree(keys, np.arange(10, 10 + keys.size, dtype=np.uint64), 8)
        _same(tree, o, np.array([top, top - 1, 0, 1, 4, 5], np.uint64))


def _crowded(kind, kw, n):
    """Keys whose distances inside a few hundred entries differ too much for
    16-bit codes: everywhere ("runs": nodes of full words, several levels of
    them), in one key of 300 ("some": codes that tie here and there), at both
    ends, and all keys consecutive (codes are exact)."""
    g = W.rng(915)
    i = np.arange(n, dtype=np.uint64)
    if kind == "runs":
        return (i // 100 << np.uint64(kw // 2)) | i % 100 if kw == 64 else (i // 20 << np.uint64(11)) | i % 20
    if kind == "dense":
        return i + np.uint64(12345)
    far = W.uniform_keys(n - n // 300, kw, seed=916).astype(np.uint64)
    if kind == "some":
        starts = g.choice(far, size=n // 300 // 40 + 1)
        near = (starts[:, None] + np.arange(1, 41, dtype=np.uint64)).ravel()
    else:
        near = np.concatenate([i[: n // 100], np.uint64(2**kw - 1) - i[: n // 100]])
    return np.unique(np.concatenate([far, near]))


@pytest.mark.parametrize("kind", ["runs", "some", "ends", "dense"])
@pytest.mark.parametrize("kw,n", [(64, 100_000), (64, 1_500_000), (32, 1_500_000)])
def test_keys_that_crowd(bt, kind, kw, n):
    keys = _crowded(kind, kw, n).astype(W.key_dtype(kw))
    vals = W.rank_values(keys.size, 64)
    tree = bt.BTree(keys, vals, 32)
    o = OracleTree(keys, vals, 32)
    g = W.rng(917)
    near = keys[g.integers(0, keys.size, size=30_000)] + g.integers(0, 3, size=30_000).astype(keys.dtype)
    _same(tree, o, np.concatenate([W.make_queries(keys, 30_001, 0.8, seed=918, width_bits=kw), near, keys[:3],
                                   keys[-3:]]))


@pytest.mark.parametrize("n", [1, 2, 4096, 4097, 17 * 4096 + 1])
@pytest.mark.parametrize("tie", [0, 7, 100, 5000])
def test_byte_keys_with_tied_words(bt, n, tie):
    """Runs of `tie` keys that share the 8 bytes the index walks and differ
    only later, so that the search has to go on from the first of a run (at
    5000 keys to a run the tree has no index and descends);
    queries inside runs, at their ends, between them and outside all keys."""
    g = W.rng(910 + n + tie)
    keys = g.integers(0, 256, size=(n, 32), dtype=np.uint8)
    if tie:
        keys[:, :8] = g.integers(0, 256, size=(n // tie + 1, 8), dtype=np.uint8)[np.arange(n) // tie]
    keys = W._sort_rows(keys)
    vals = W.rank_values(keys.shape[0], 64)
    tree = bt.BTree(keys, vals, 16)
    o = OracleBytesTree(keys, vals, 16)
    q = W.make_byte_queries(keys, 3001, 0.7, seed=911)
    near = keys[g.integers(0, keys.shape[0], size=500)].copy()
    near[:, 31] ^= 1
    ends = np.stack([keys[0], keys[-1], np.zeros(32, np.uint8), np.full(32, 255, np.uint8)])
    _same(tree, o, np.concatenate([q, near, ends]))
    o.close()


@pytest.mark.parametrize("ntrees,nb", [(1, 1), (3, 31), (3, 33), (40, 700), (4, 65_536), (4, 65_537)])
def test_work_lists_through_the_walk_kernel(bt, ntrees, nb):
    """Lists shorter and longer than a row, longer than the kernel plans
    itself (then the descent's), more trees than its table and its tops have
    room for, empty trees and batches, and bad entries."""
    import torch
    g = W.rng(920 + nb)
    sizes = [0 if i % 7 == 6 else int(3 * 8 ** (1 + i % 5)) for i in range(ntrees)]
    keysets = [W.uniform_keys(n, 64, seed=921 + i) for i, n in enumerate(sizes)]
    trees = [bt.BTree(k, W.rank_values(k.size, 64), 16) for k in keysets]
    forest = bt.bt_forest_create([t.handle for t in trees])
    desc = np.zeros(nb, bt.BATCH_DESC_DTYPE)
    desc["tree"] = g.integers(0, ntrees, size=nb)
    counts = g.choice([0, 1, 5, 31, 32, 33, 70], size=nb)
    desc["count"], desc["offset"] = counts, np.cumsum(counts) - counts
    total = max(1, int(counts.sum()))
    q = g.integers(0, 2**64, size=total, dtype=np.uint64)
    want_v, want_f = np.full(total, 5, np.uint64), np.full(total, 9, np.uint8)
    for i, k in enumerate(keysets):
        rows = np.flatnonzero(desc["tree"] == i)
        at = np.concatenate([np.arange(o, o + c) for o, c in zip(desc["offset"][rows], counts[rows])] or
                            [np.empty(0)]).astype(np.int64)
        if k.size:
            hit = g.random(at.size) < 0.7
            q[at[hit]] = k[g.integers(0, k.size, size=int(hit.sum()))]
        pos = np.searchsorted(k, q[at]) if k.size else np.zeros(at.size, np.int64)
        found = (pos < k.size) & (k[np.minimum(pos, max(k.size - 1, 0))] == q[at]) if k.size else np.zeros(at.size, bool)
        want_v[at], want_f[at] = np.where(found, pos.astype(np.uint64), np.uint64(2**64 - 1)), found
    bad = np.flatnonzero(counts > 0)[: 2 if nb > 30 else 0]  # rejected: nothing is written for them
    for b, (field, value) in zip(bad, [("tree", ntrees), ("offset", total + 1)]):
        o, c = int(desc["offset"][b]), int(counts[b])
        want_v[o:o + c], want_f[o:o + c] = 5, 9
        desc[field][b] = value
    dq = torch.from_numpy(q).cuda()
    v = torch.full((total,), 5, dtype=torch.int64, device="cuda")
    f = torch.full((total,), 9, dtype=torch.uint8, device="cuda")
    wsb = bt.bt_forest_workspace_bytes(nb)
    ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
    bt.bt_forest_bad_batches()
    bt.bt_forest_search(forest, torch.from_numpy(desc.view(np.uint8)).cuda(), nb, dq, v, f, ws, wsb)
    torch.cuda.synchronize()
    assert bt.bt_forest_bad_batches() == len(bad)
    assert np.array_equal(v.cpu().numpy().view(np.uint64), want_v) and np.array_equal(f.cpu().numpy(), want_f)
    bt.bt_forest_free(forest)


@pytest.mark.parametrize("kind", ["pl1", "pl", "pl_many", "mlp"])
@pytest.mark.parametrize("kw,n", [(64, 3), (64, 200), (64, 4 * 8192 + 5), (64, 400_000), (32, 8 * 16384 + 9)])
def test_learned_search_through_the_walk(bt, kind, kw, n):
    """Models whose windows span one leaf, many segments and the whole tree
    (one line over lognormal keys), parameters in shared and in global memory."""
    import torch
    keys = W.lognormal_mixture_keys(n, seed=930) if kw == 64 else W.uniform_keys(n, kw, seed=930)
    vals = W.rank_values(n, 64)
    tree = bt.BTree(keys, vals, 32)
    o = OracleTree(keys, vals, 32)
    if kind == "mlp":
        m = bt.bt_model_train(tree.handle, bt.BT_MODEL_MLP, h_init=W.mlp_init_params(931), steps=20, batch=1024,
                              lr=2e-3, seed=932)
    else:
        m = bt.bt_model_train(tree.handle, bt.BT_MODEL_PL, segments={"pl1": 1, "pl": 64, "pl_many": 2000}[kind])
    for nq in (1, 4099, 152 * 512 + 7):
        q = W.make_queries(keys, nq, 0.7, seed=933 + nq, width_bits=kw)
        q[:1] = keys[-1]
        ov, of, _, _ = o.search(q)
        v, f = tree.alloc_outputs(nq)
        ws, nb = tree.alloc_workspace(nq)
        bt.bt_learned_search_batch(tree.handle, m, torch.from_numpy(q).cuda(), nq, v, f, ws, nb)
        assert np.array_equal(v.cpu().numpy(), ov) and np.array_equal(f.cpu().numpy(), of)
    bt.bt_model_free(m)


@pytest.mark.parametrize("kw,vw", [(64, 64), (32, 64), (64, 32), (256, 64)])
@pytest.mark.parametrize("where", ["pinned", "pageable", "queries", "results", "misaligned", "shared"])
def test_host_buffers_in_place_and_copied(bt, kw, vw, where):
    """Host buffers used in place (page-locked), copied (pageable, off their
    alignment, results over the queries' memory), and some of each."""
    import torch
    n, nq = 30_000, 5003
    if kw == 256:
        keys = W.byte_keys(n, 32, seed=940)
        q = W.make_byte_queries(keys, nq, 0.7, seed=941)
        o = OracleBytesTree(keys, W.rank_values(n, vw), 16)
    else:
        keys = W.uniform_keys(n, kw, seed=940)
        q = W.make_queries(keys, nq, 0.7, seed=941, width_bits=kw)
        o = OracleTree(keys, W.rank_values(n, vw), 16, val_bits=vw)
    tree = bt.BTree(keys, W.rank_values(n, vw), 16)
    off = 1 if where == "misaligned" else 0

    def buf(nbytes, pin):
        return torch.full((nbytes + off,), 9, dtype=torch.uint8, pin_memory=pin)[off:]

    raw = torch.from_numpy(q.view(np.uint8).reshape(-1).copy())
    hq = buf(max(raw.numel(), nq * vw // 8), where not in ("pageable", "results"))
    hq[: raw.numel()] = raw
    hv = hq if where == "shared" else buf(nq * vw // 8, where not in ("pageable", "queries"))
    hf = buf(nq, where not in ("pageable", "queries"))
    ws, nb = tree.alloc_workspace(nq, host=True)
    bt.bt_search_batch_host(tree.handle, hq, nq, hv, hf, ws, nb)
    torch.cuda.synchronize()
    ov, of = o.search(q)[:2]
    got = hv[: nq * vw // 8].numpy().copy().view(np.uint64 if vw == 64 else np.uint32)
    assert np.array_equal(got.astype(np.uint64), ov) and np.array_equal(hf.numpy(), of)


def test_walk_and_host_buffers_under_capture(bt):
    """A search and one from page-locked host buffers captured in one graph;
    the replay reads what the buffers hold then."""
    import torch
    keys = W.uniform_keys(300_000, 64, seed=950)
    vals = W.rank_values(keys.size, 64)
    tree = bt.BTree(keys, vals, 32)
    o = OracleTree(keys, vals, 32)
    nq = 40_013
    dq = torch.zeros(nq, dtype=torch.int64, device="cuda")
    hq = torch.zeros(nq, dtype=torch.int64, pin_memory=True)
    v, f = tree.alloc_outputs(nq)
    hv, hf = torch.zeros(nq, dtype=torch.int64, pin_memory=True), torch.zeros(nq, dtype=torch.uint8, pin_memory=True)
    ws, nb = tree.alloc_workspace(nq, host=True)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        bt.bt_search_batch(tree.handle, dq, nq, v, f, ws, nb)
        bt.bt_search_batch_host(tree.handle, hq, nq, hv, hf, ws, nb)
    for seed in (951, 952):
        q = [W.make_queries(keys, nq, 0.8, seed=seed + k, width_bits=64) for k in (0, 10)]
        dq.copy_(torch.from_numpy(q[0].view(np.int64)))
        hq.copy_(torch.from_numpy(q[1].view(np.int64)))
        graph.replay()
        torch.cuda.synchronize()
        for gv, gf, qq in ((v.cpu().numpy(), f.cpu().numpy(), q[0]), (hv.numpy().view(np.uint64), hf.numpy(), q[1])):
            ov, of = o.search(qq)[:2]
            assert np.array_equal(gv, ov) and np.array_equal(gf, of)
