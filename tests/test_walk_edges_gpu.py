"""Edges of the searches through the walk index: waits that run out, buffers
that overlap or are page-locked in part, and trees at the sizes where the
index changes shape."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import OracleTree
from paper_2604_21117_gb300 import workloads as W

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


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.fixture
def no_polls(bt):
    """Every bounded wait gives up at once while the test runs."""
    import torch
    torch.cuda.synchronize()
    bt.bt_check_timeouts()  # clear anything earlier
    bt.bt_debug_set_wait_polls(0)
    yield
    torch.cuda.synchronize()
    bt.bt_debug_set_wait_polls(bt.BT_DEFAULT_WAIT_POLLS)


def _two_trees(bt):
    out = []
    for i, n in enumerate((20_000, 300_000)):
        keys = W.uniform_keys(n, 64, seed=960 + i)
        vals = W.rank_values(n, 64)
        out.append((keys, bt.BTree(keys, vals, 32), OracleTree(keys, vals, 32)))
    return out


def test_work_list_whose_wait_gives_up_is_searched_all_the_same(bt, no_polls):
    """The wait for the tops gives up in every warp: reported, and every
    result is there (a completion flag says that the list has been searched)."""
    import torch
    trees = _two_trees(bt)
    forest = bt.bt_forest_create([t[1].handle for t in trees])
    nb, per = 300, 77
    desc = np.zeros(nb, bt.BATCH_DESC_DTYPE)
    desc["tree"], desc["count"], desc["offset"] = np.arange(nb) % 2, per, np.arange(nb) * per
    q = np.concatenate([W.make_queries(trees[i % 2][0], per, 0.8, seed=970 + i, width_bits=64) for i in range(nb)])
    v = torch.full((nb * per,), 5, dtype=torch.int64, device="cuda")
    f = torch.full((nb * per,), 9, dtype=torch.uint8, device="cuda")
    wsb = bt.bt_forest_workspace_bytes(nb)
    ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
    bt.bt_forest_search(forest, _dev(desc.view(np.uint8)), nb, _dev(q), v, f, ws, wsb)
    with pytest.raises(bt.BTreeError) as e:
        bt.bt_check_timeouts()
    assert e.value.code == "BT_ERR_TIMEOUT"
    gv, gf = v.cpu().numpy().view(np.uint64).reshape(nb, per), f.cpu().numpy().reshape(nb, per)
    for i in range(2):
        ov, of = trees[i][2].search(q.reshape(nb, per)[i::2].ravel())[:2]
        assert np.array_equal(gv[i::2].ravel(), ov) and np.array_equal(gf[i::2].ravel(), of)
    bt.bt_forest_free(forest)


def test_served_requests_have_their_results_when_waits_give_up(bt, no_polls):
    trees = _two_trees(bt)
    srv = bt.bt_server_create([t[1] for t in trees], None, slots=2, max_batch=512, deadline_us=20.0)
    for r in range(40):
        q = W.make_queries(trees[r % 2][0], 1 + 9 * r, 0.8, seed=980 + r, width_bits=64)
        v, f = np.full(q.size, 5, np.uint64), np.full(q.size, 9, np.uint8)
        ticket = bt.bt_server_submit(srv, r % 2, q, v, f)
        bt.bt_server_drain(srv, 10.0)
        assert bt.bt_server_poll(srv, 16) == [ticket]
        ov, of = trees[r % 2][2].search(q)[:2]
        assert np.array_equal(v, ov) and np.array_equal(f, of)
    bt.bt_server_destroy(srv)
    with pytest.raises(bt.BTreeError) as e:
        bt.bt_check_timeouts()
    assert e.value.code == "BT_ERR_TIMEOUT"


@pytest.mark.parametrize("learned", [False, True])
@pytest.mark.parametrize("vw,over", [(32, "values"), (64, "values, 8 bytes on"), (64, "found"), (64, "values, same place")])
def test_results_over_the_queries_of_a_large_batch(bt, learned, vw, over):
    """A batch that the automatic choice partitions is copied before results
    are written: they may lie over the queries, narrower and shifted too."""
    import torch
    n, nq = 4_300_000, 800_003
    keys = W.uniform_keys(n, 64, seed=990)
    tree = bt.BTree(keys, W.rank_values(n, vw), 32)
    assert bt.bt_sort_bits(tree.handle, nq) > 0
    q = W.make_queries(keys, nq, 0.8, seed=991, width_bits=64)
    pos = np.searchsorted(keys, q)
    hit = keys[np.minimum(pos, n - 1)] == q
    want = np.where(hit, pos.astype(np.uint64), np.uint64(2**vw - 1))
    buf = torch.zeros(8 * nq + 8, dtype=torch.uint8, device="cuda")
    buf[: 8 * nq] = _dev(q.view(np.uint8))
    v = torch.zeros(nq * vw // 8, dtype=torch.uint8, device="cuda") if over == "found" else \
        buf[8 if over.endswith("on") else 0:][: nq * vw // 8]
    f = buf[5 * nq: 6 * nq] if over == "found" else torch.zeros(nq, dtype=torch.uint8, device="cuda")
    ws, nb = tree.alloc_workspace(nq)
    if learned:
        m = bt.bt_model_train(tree.handle, bt.BT_MODEL_PL, segments=256)
        bt.bt_learned_search_batch(tree.handle, m, buf.data_ptr(), nq, v, f, ws, nb)
    else:
        bt.bt_search_batch(tree.handle, buf.data_ptr(), nq, v, f, ws, nb)
    got = v.cpu().numpy().view(np.uint64 if vw == 64 else np.uint32).astype(np.uint64)
    assert np.array_equal(got, want) and np.array_equal(f.cpu().numpy().astype(bool), hit)
    if learned:
        bt.bt_model_free(m)
    tree.close()


def test_a_reported_error_does_not_fail_the_next_build(bt):
    """A call refused by the runtime (an allocation while a stream captures)
    reports its error; the next call starts without it."""
    import ctypes
    import torch
    keys = W.uniform_keys(3000, 64, seed=997)
    tree = bt.BTree(keys, W.rank_values(3000, 64), 16)
    cu = ctypes.CDLL("libcuda.so.1")
    s, graph = torch.cuda.Stream(), ctypes.c_void_p()
    torch.cuda.synchronize()
    assert cu.cuStreamBeginCapture_v2(ctypes.c_void_p(s.cuda_stream), 0) == 0  # global: no allocations meanwhile
    with pytest.raises(bt.BTreeError) as e:
        bt.bt_forest_create([tree.handle])
    assert e.value.code == "BT_ERR_CUDA"
    cu.cuStreamEndCapture(ctypes.c_void_p(s.cuda_stream), ctypes.byref(graph))
    if graph.value:
        cu.cuGraphDestroy(graph)
    again = bt.BTree(keys, W.rank_values(3000, 64), 16)
    v, f = again.search(_dev(keys))
    assert np.array_equal(v.cpu().numpy(), np.arange(3000, dtype=np.uint64)) and f.cpu().numpy().all()



def _captured_nodes(call, stream):
    """Nodes of the graph that `call` on the raw stream captures (nothing
    runs); None when the call fails."""
    import ctypes
    cu = ctypes.CDLL("libcuda.so.1")
    graph, count, s = ctypes.c_void_p(), ctypes.c_size_t(), ctypes.c_void_p(stream)
    assert cu.cuStreamBeginCapture_v2(s, 2) == 0  # relaxed
    try:
        call()
        failed = False
    except Exception:
        failed = True
    ended = cu.cuStreamEndCapture(s, ctypes.byref(graph))
    if failed or ended != 0:
        return None
    assert cu.cuGraphGetNodes(graph, None, ctypes.byref(count)) == 0
    assert cu.cuGraphDestroy(graph) == 0
    return count.value


@pytest.mark.parametrize("locked", ["one range", "two ranges", "a gap between two ranges"])
def test_only_wholly_page_locked_queries_are_read_in_place(bt, locked):
    """A batch searched in place is one kernel node of a captured graph, one
    that is copied several (with a gap, only captured: it never runs)."""
    import mmap
    import torch
    part = 1 << 16
    nq = 3 * part // 8
    keys = W.uniform_keys(50_000, 64, seed=995)
    tree = bt.BTree(keys, W.rank_values(keys.size, 64), 32)
    region = mmap.mmap(-1, 3 * part)
    q = np.frombuffer(region, np.uint64)
    q[:] = W.make_queries(keys, nq, 0.8, seed=996, width_bits=64)
    ranges = {"one range": [(0, 3)], "two ranges": [(0, 1), (1, 2)], "a gap between two ranges": [(0, 1), (2, 1)]}
    v, f = torch.zeros(nq, dtype=torch.int64, pin_memory=True), torch.zeros(nq, dtype=torch.uint8, pin_memory=True)
    ws, nb = tree.alloc_workspace(nq, host=True)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    rt = torch.cuda.cudart()
    for at, count in ranges[locked]:
        assert int(rt.cudaHostRegister(q.ctypes.data + at * part, count * part, 0)) == 0
    try:
        def call():
            bt.bt_search_batch_host(tree.handle, q, nq, v, f, ws, nb, stream=stream.cuda_stream)
        nodes = _captured_nodes(call, stream.cuda_stream)
        if locked == "a gap between two ranges":
            assert nodes != 1
        else:
            assert nodes == 1
            call()
            stream.synchronize()
            ov, of = OracleTree(keys, W.rank_values(keys.size, 64), 32).search(q.copy())[:2]
            assert np.array_equal(v.numpy().view(np.uint64), ov) and np.array_equal(f.numpy(), of)
    finally:
        torch.cuda.synchronize()
        for at, _ in ranges[locked]:
            rt.cudaHostUnregister(q.ctypes.data + at * part)


@pytest.mark.parametrize("staged", [False, True])
def test_forest_autotune_times_the_walk_once(bt, staged):
    """The settings that lead to the walk are one: the choice among them is
    fixed and not the luckiest of many timings of the same launch."""
    import torch
    trees = _two_trees(bt)
    if staged:  # the trees' own design no longer walks, reading through L1 does
        bt.bt_tree_set_staging(trees[0][1].handle, bt.BT_STAGE_CP_ASYNC)
    forest = bt.bt_forest_create([t[1].handle for t in trees])
    nb, per = 200, 64
    desc = np.zeros(nb, bt.BATCH_DESC_DTYPE)
    desc["tree"], desc["count"], desc["offset"] = np.arange(nb) % 2, per, np.arange(nb) * per
    q = _dev(W.make_queries(trees[1][0], nb * per, 0.8, seed=998, width_bits=64))
    v, f = trees[0][1].alloc_outputs(nb * per)
    wsb = bt.bt_forest_workspace_bytes(nb)
    ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
    best = bt.bt_forest_autotune(forest, _dev(desc.view(np.uint8)), nb, q, v, f, ws, wsb)
    walk = (8, 16384, 0, 1 if staged else 0)
    got = (best.warps_per_block, best.pin_budget, best.lane_queries, best.staging)
    assert got == walk or best.staging == 2 or (staged and best.staging == 0)
    bt.bt_forest_free(forest)


# Keys per entry: 32 / (key + value bytes).  Up to 2^12 entries the top alone,
# then one coded level of 17 children up to 2^12 segments, then two, then from
# 15360 segments (25600 for 32-bit keys) a level of full words above those.
def _per_entry(kw, vw):
    return 32 // ((kw + vw) // 8)


def _expect(keys, vw, q):
    pos = np.searchsorted(keys, q)
    hit = keys[np.minimum(pos, keys.size - 1)] == q
    return np.where(hit, pos.astype(np.uint64), np.uint64(2**vw - 1)), hit


def _edge_queries(keys, kw, vw, seed):
    """Keys at the ends of entries, nodes and segments and the values beside
    them, random keys, random values."""
    G, n, g = _per_entry(kw, vw), keys.size, W.rng(seed)
    ranks = [g.integers(0, n, size=40_000)]
    for span in (1, 17, 289, 289 * 5, 289 * 9):
        ends = np.arange(1, n // (span * G) + 1) * (span * G)
        ends = ends if ends.size < 20_000 else np.concatenate([ends[:5000], ends[-5000:], g.choice(ends, 10_000)])
        ranks += [ends - 1, np.minimum(ends, n - 1), np.minimum(ends + 1, n - 1)]
    k = keys[np.concatenate(ranks + [np.array([0, n - 1])])]
    return np.concatenate([k, k + keys.dtype.type(1), k - keys.dtype.type(1),
                           g.integers(0, 2**kw, size=2000, dtype=np.uint64).astype(keys.dtype)])


@pytest.mark.parametrize("kw,vw", [(64, 64), (64, 32), (32, 64), (32, 32)])
@pytest.mark.parametrize("entries,more", [(1, 0), (1, 1), (4096, 0), (4096, 1), (17 * 4096, 0), (17 * 4096, 1)])
def test_where_the_index_changes_shape(bt, kw, vw, entries, more):
    n = _per_entry(kw, vw) * entries + more
    keys = W.uniform_keys(n, kw, seed=1020 + n)
    tree = bt.BTree(keys, W.rank_values(n, vw), 16)
    q = _edge_queries(keys, kw, vw, 1021)
    want, hit = _expect(keys, vw, q)
    for nq in (1, 33, q.size):
        v, f = tree.search(_dev(q[-nq:]))
        assert np.array_equal(v.cpu().numpy().astype(np.uint64), want[-nq:])
        assert np.array_equal(f.cpu().numpy().astype(bool), hit[-nq:])


@pytest.mark.parametrize("kw,vw,segs", [(64, 64, 15360), (32, 64, 25600), (32, 32, 25600)])
@pytest.mark.parametrize("more", [0, 3])
def test_full_words_above_coded_levels(bt, kw, vw, segs, more):
    """The largest top over two coded levels, and the smallest trees with a
    level of full words between them."""
    n = _per_entry(kw, vw) * 289 * segs + more
    keys = W.uniform_keys(n, kw, seed=1022)
    tree = bt.BTree(keys, W.rank_values(n, vw), 64)
    q = _edge_queries(keys, kw, vw, 1023)
    want, hit = _expect(keys, vw, q)
    v, f = tree.search(_dev(q))
    assert np.array_equal(v.cpu().numpy().astype(np.uint64), want)
    assert np.array_equal(f.cpu().numpy().astype(bool), hit)
    tree.close()


@pytest.mark.parametrize("ties", ["few", "many"])
def test_full_words_of_byte_keys_that_tie(bt, ties):
    """Words that tie across the ends of nodes and segments, in so few keys
    that the lower levels stay coded and in so many that none is."""
    n = 289 * 15360 + 3
    words = W.uniform_keys(n, 64, seed=1024).astype(np.uint64)
    second = np.arange(1445, n, 1445) if ties == "few" else np.arange(3, n, 3)
    words[second] = words[second - 1]
    keys = np.zeros((n, 32), np.uint8)
    keys[:, :8] = words.astype(">u8").view(np.uint8).reshape(n, 8)
    keys[:, 31] = 1
    keys[second, 31] = 3
    tree = bt.BTree(keys, W.rank_values(n, 64), 64)
    assert bt.bt_tree_walk_bytes(tree.handle) > 0
    g = W.rng(1025)
    at = np.concatenate([second[:30_000] - 1, second[:30_000], second[-30_000:], g.integers(0, n, size=60_000),
                         np.array([0, n - 1])])
    q = np.concatenate([keys[at]] * 3)
    q[at.size: 2 * at.size, 31] += 1   # between the two of a pair, or above it: stored nowhere
    q[2 * at.size:, 31] = 0            # below both
    v, f = tree.search(_dev(q))
    v, f = v.cpu().numpy(), f.cpu().numpy()
    assert np.array_equal(v[: at.size], at.astype(np.uint64)) and f[: at.size].all()
    assert (v[at.size:] == np.uint64(2**64 - 1)).all() and not f[at.size:].any()
    tree.close()


@pytest.mark.parametrize("ntrees", [128, 129])
def test_as_many_trees_as_the_walks_table_holds_and_one_more(bt, ntrees):
    import torch
    keysets = [W.uniform_keys(20 + 37 * i, 64, seed=1026 + i) for i in range(ntrees)]
    trees = [bt.BTree(k, W.rank_values(k.size, 64), 16) for k in keysets]
    forest = bt.bt_forest_create([t.handle for t in trees])
    per = 45
    desc = np.zeros(ntrees, bt.BATCH_DESC_DTYPE)
    desc["tree"], desc["count"], desc["offset"] = np.arange(ntrees), per, np.arange(ntrees) * per
    q = np.concatenate([W.make_queries(k, per, 0.7, seed=1027, width_bits=64) for k in keysets])
    v, f = trees[0].alloc_outputs(q.size)
    wsb = bt.bt_forest_workspace_bytes(ntrees)
    bt.bt_forest_search(forest, _dev(desc.view(np.uint8)), ntrees, _dev(q), v, f,
                        torch.empty(wsb, dtype=torch.uint8, device="cuda"), wsb)
    want = [_expect(k, 64, q[i * per:(i + 1) * per]) for i, k in enumerate(keysets)]
    assert np.array_equal(v.cpu().numpy(), np.concatenate([w[0] for w in want]))
    assert np.array_equal(f.cpu().numpy().astype(bool), np.concatenate([w[1] for w in want]))
    bt.bt_forest_free(forest)


@pytest.mark.parametrize("kind", ["pl", "pl_many", "mlp"])
@pytest.mark.parametrize("kw,entries", [(64, 4096), (64, 17 * 4096), (32, 4096), (32, 17 * 4096)])
def test_learned_search_where_the_index_changes_shape(bt, kind, kw, entries):
    n = _per_entry(kw, 64) * entries + 1
    keys = W.lognormal_mixture_keys(n, seed=1028) if kw == 64 else W.uniform_keys(n, kw, seed=1028)
    tree = bt.BTree(keys, W.rank_values(n, 64), 32)
    if kind == "mlp":
        m = bt.bt_model_train(tree.handle, bt.BT_MODEL_MLP, h_init=W.mlp_init_params(1029), steps=20, batch=1024,
                              lr=2e-3, seed=1030)
    else:
        m = bt.bt_model_train(tree.handle, bt.BT_MODEL_PL, segments={"pl": 64, "pl_many": 2000}[kind])
    q = _edge_queries(keys, kw, 64, 1031)
    want, hit = _expect(keys, 64, q)
    v, f = tree.alloc_outputs(q.size)
    ws, nb = tree.alloc_workspace(q.size)
    bt.bt_learned_search_batch(tree.handle, m, _dev(q), q.size, v, f, ws, nb)
    assert np.array_equal(v.cpu().numpy(), want) and np.array_equal(f.cpu().numpy().astype(bool), hit)
    bt.bt_model_free(m)
