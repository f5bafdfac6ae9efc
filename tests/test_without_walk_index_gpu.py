"""Trees built without the walk index: what searches them then -- the level-wise
descent of batches as given, the automatic partition before it, the learned
descent, the work lists' descent -- gives the oracle's results, and the memory
such a tree does not hold is told."""
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


def _tree(bt, n, m=32, kw=64, vw=64, seed=1000):
    keys = W.uniform_keys(n, kw, seed=seed)
    vals = W.rank_values(n, vw)
    tree = bt.BTree(keys, vals, m, walk_index=False)
    assert bt.bt_tree_walk_bytes(tree.handle) == 0
    return keys, tree, OracleTree(keys, vals, m, val_bits=vw)


def _same(tree, o, q, sort_bits=-1):
    v, f = tree.search(_dev(q), sort_bits=sort_bits)
    ov, of, _, _ = o.search(q)
    assert np.array_equal(v.cpu().numpy().astype(np.uint64), ov) and np.array_equal(f.cpu().numpy(), of)


@pytest.mark.parametrize("n,kw,vw", [(5, 64, 64), (3000, 32, 64), (1 << 20, 64, 64), (1 << 20, 32, 32),
                                     (3_000_000, 64, 64), (50_000, 256, 64)])
def test_memory_of_the_index_is_told_and_can_be_declined(bt, n, kw, vw):
    """Behind the image (up to 8 MB of entries) and in its own allocation:
    one more copy of keys and values and not much else."""
    keys = W.byte_keys(n, 32, seed=1001) if kw == 256 else W.uniform_keys(n, kw, seed=1001)
    vals = W.rank_values(n, vw)
    with_index, without = bt.BTree(keys, vals, 32), bt.BTree(keys, vals, 32, walk_index=False)
    assert with_index.device_bytes == without.device_bytes
    assert bt.bt_tree_walk_bytes(without.handle) == 0
    entry = 64 * n if kw == 256 else n * (kw + vw) // 8
    assert entry <= bt.bt_tree_walk_bytes(with_index.handle) <= 1.5 * entry + (1 << 18)
    q = W.make_byte_queries(keys, 2001, 0.8, seed=1002) if kw == 256 else \
        W.make_queries(keys, 2001, 0.8, seed=1002, width_bits=kw)
    (v0, f0), (v1, f1) = with_index.search(_dev(q)), without.search(_dev(q))
    assert np.array_equal(v0.cpu().numpy(), v1.cpu().numpy()) and np.array_equal(f0.cpu().numpy(), f1.cpu().numpy())


def test_build_options_are_checked(bt):
    import ctypes
    keys = np.arange(4, dtype=np.uint64)
    out = ctypes.c_void_p()
    bad = bt.bt_build_opts(2)
    assert bt._lib.bt_build_ex(keys.ctypes.data, keys.ctypes.data, 4, 8, 8, 16, ctypes.byref(bad), None,
                               ctypes.byref(out)) == 1
    assert bt._lib.bt_build_ex(keys.ctypes.data, keys.ctypes.data, 4, 8, 8, 16, None, None, ctypes.byref(out)) == 0
    assert bt.bt_tree_walk_bytes(out.value) > 0
    bt.bt_free(out.value)
    assert bt.bt_tree_walk_bytes(None) == 0


@pytest.mark.parametrize("inner,ballot", [(0, 0), (1, 0), (2, 0), (0, 1), (1, 1)])
@pytest.mark.parametrize("m", [8, 64])
@pytest.mark.parametrize("kw,vw", [(32, 32), (64, 64), (64, 32)])
def test_pipelined_options(bt, inner, ballot, m, kw, vw):
    keys, tree, o = _tree(bt, 90_000 + m, m, kw, vw)
    bt.bt_tree_set_descent(tree.handle, inner, ballot)
    q = W.make_queries(keys, 40_011, 0.8, seed=1003 + m, width_bits=kw, zipf_s=1.1)
    for sb in (-1, 0, 12):
        _same(tree, o, q, sb)
    bt.bt_check_timeouts()


@pytest.mark.parametrize("nq", [1, 31, 33, 1000, 16_384, 100_003])
def test_batch_sizes_of_the_pipelined_descent(bt, nq):
    keys, tree, o = _tree(bt, 400_000)
    _same(tree, o, W.make_queries(keys, nq, 0.9, seed=1004 + nq, width_bits=64))
    bt.bt_check_timeouts()


@pytest.mark.parametrize("warps,pin,window", [(4, 0, 0), (8, 16384, 64 << 20), (16, 49152, 0)])
def test_launch_settings_and_l2_window(bt, warps, pin, window):
    keys, tree, o = _tree(bt, 700_000, 16)
    bt.bt_tree_set_launch(tree.handle, warps, pin)
    bt.bt_tree_set_l2_window(tree.handle, window)
    _same(tree, o, W.make_queries(keys, 70_001, 0.9, seed=1005, width_bits=64))
    bt.bt_tree_set_l2_window(tree.handle, 0)


@pytest.mark.parametrize("sort_bits", [0, 12])
def test_the_pipelined_descents_wait_gives_up_and_is_reported(bt, sort_bits):
    import torch
    keys, tree, o = _tree(bt, 300_000)
    q = W.make_queries(keys, 50_000, 0.9, seed=1006, width_bits=64)
    bt.bt_check_timeouts()
    try:
        bt.bt_debug_set_wait_polls(0)
        tree.search(_dev(q), sort_bits=sort_bits)
        torch.cuda.synchronize()
    finally:
        bt.bt_debug_set_wait_polls(bt.BT_DEFAULT_WAIT_POLLS)
    with pytest.raises(bt.BTreeError) as e:
        bt.bt_check_timeouts()
    assert e.value.code == "BT_ERR_TIMEOUT"
    _same(tree, o, q, sort_bits)
    bt.bt_check_timeouts()


@pytest.mark.parametrize("caps", [(3, 1), (0, 1)])
def test_two_streams_with_corun_caps(bt, caps):
    """Partition and descent of batches on two streams side by side."""
    import torch
    B = 70_001
    keys, tree, o = _tree(bt, 300_000)
    bt.bt_tree_set_corun(tree.handle, *caps)
    qs = [W.make_queries(keys, B, 0.9, seed=1007 + i, width_bits=64) for i in range(2)]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    bufs = [(_dev(q), *tree.alloc_outputs(B), *tree.alloc_workspace(B)) for q in qs]
    torch.cuda.synchronize()
    for _ in range(3):
        for s, (dq, v, f, ws, nb) in zip(streams, bufs):
            tree.search_into(dq, v, f, ws, nb, sort_bits=14, stream=s)
    torch.cuda.synchronize()
    bt.bt_check_timeouts()
    for q, (_, v, f, _, _) in zip(qs, bufs):
        ov, of = o.search(q)[:2]
        assert np.array_equal(v.cpu().numpy(), ov) and np.array_equal(f.cpu().numpy(), of)


@pytest.mark.parametrize("how", ["plain", "host", "learned"])
def test_large_batches_are_partitioned_by_themselves(bt, how):
    """The automatic partition inside the search, from host buffers too, and
    before the learned descent."""
    import torch
    n, nq = 4_300_000, 800_003
    keys = W.uniform_keys(n, 64, seed=1010)
    tree = bt.BTree(keys, W.rank_values(n, 64), 32, walk_index=False)
    assert bt.bt_sort_bits(tree.handle, nq) > 0
    q = W.make_queries(keys, nq, 0.8, seed=1011, width_bits=64)
    if how == "host":
        v, f = tree.search_host(q)
    else:
        v, f = tree.alloc_outputs(nq)
        ws, nb = tree.alloc_workspace(nq)
        if how == "learned":
            m = bt.bt_model_train(tree.handle, bt.BT_MODEL_PL, segments=256)
            bt.bt_learned_search_batch(tree.handle, m, _dev(q), nq, v, f, ws, nb)
        else:
            bt.bt_search_batch(tree.handle, _dev(q), nq, v, f, ws, nb)
        torch.cuda.synchronize()
        v, f = v.cpu().numpy(), f.cpu().numpy()
    pos = np.searchsorted(keys, q)
    hit = keys[np.minimum(pos, n - 1)] == q
    assert np.array_equal(v, np.where(hit, pos.astype(np.uint64), np.uint64(2**64 - 1)))
    assert np.array_equal(f.astype(bool), hit)
    tree.close()


@pytest.mark.parametrize("kind", ["pl", "pl_many", "mlp"])
def test_learned_descent_of_batches_as_given(bt, kind):
    keys = W.lognormal_mixture_keys(400_000, seed=1012)
    vals = W.rank_values(keys.size, 64)
    tree = bt.BTree(keys, vals, 32, walk_index=False)
    o = OracleTree(keys, vals, 32)
    if kind == "mlp":
        m = bt.bt_model_train(tree.handle, bt.BT_MODEL_MLP, h_init=W.mlp_init_params(1013), steps=20, batch=1024,
                              lr=2e-3, seed=1014)
    else:
        m = bt.bt_model_train(tree.handle, bt.BT_MODEL_PL, segments={"pl": 64, "pl_many": 2000}[kind])
    for nq in (1, 33, 1000, 40_003):
        q = W.make_queries(keys, nq, 0.7, seed=1015 + nq, width_bits=64)
        v, f = tree.alloc_outputs(nq)
        ws, nb = tree.alloc_workspace(nq)
        bt.bt_learned_search_batch(tree.handle, m, _dev(q), nq, v, f, ws, nb)
        ov, of, _, _ = o.search(q)
        assert np.array_equal(v.cpu().numpy(), ov) and np.array_equal(f.cpu().numpy(), of)
    bt.bt_model_free(m)


@pytest.mark.parametrize("lanes", [0, 2])
def test_one_tree_without_an_index_among_a_forests(bt, lanes):
    """Such a forest's lists are descended, the other trees' index or not."""
    import torch
    k0, t0, o0 = _tree(bt, 50_000)
    k1 = W.uniform_keys(300_000, 64, seed=1016)
    t1, o1 = bt.BTree(k1, W.rank_values(k1.size, 64), 16), OracleTree(k1, W.rank_values(k1.size, 64), 16)
    forest = bt.bt_forest_create([t0.handle, t1.handle])
    bt.bt_forest_set_launch(forest, 8, 32768, lanes, 0)
    nb, per = 120, 83
    desc = np.zeros(nb, bt.BATCH_DESC_DTYPE)
    desc["tree"], desc["count"], desc["offset"] = np.arange(nb) % 2, per, np.arange(nb) * per
    q = np.concatenate([W.make_queries((k0, k1)[i % 2], per, 0.8, seed=1017 + i, width_bits=64) for i in range(nb)])
    v, f = t1.alloc_outputs(q.size)
    wsb = bt.bt_forest_workspace_bytes(nb)
    bt.bt_forest_search(forest, _dev(desc.view(np.uint8)), nb, _dev(q), v, f,
                        torch.empty(wsb, dtype=torch.uint8, device="cuda"), wsb)
    gv, gf = v.cpu().numpy().reshape(nb, per), f.cpu().numpy().reshape(nb, per)
    for i, o in enumerate((o0, o1)):
        ov, of = o.search(q.reshape(nb, per)[i::2].ravel())[:2]
        assert np.array_equal(gv[i::2].ravel(), ov) and np.array_equal(gf[i::2].ravel(), of)
    bt.bt_forest_free(forest)
