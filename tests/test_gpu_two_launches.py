"""The two-launch path (score_fused, then select_cluster or select_stream) behind the entry points whose short calls take one
launch: prefixes past what that launch has room for, so that the strides, the window rows and the way back into the cache
run here.  Against the fp64 oracle under the end-to-end rule of gpu_util."""
import numpy as np
import pytest
import torch

import oracle
import jq_workloads as W
import paper_2509_10798_b200 as jq
from gpu_util import assert_kept_sets_agree, dev_bf16, host_bits, shape_of

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as entry
    entry.build()


def wl_of(Hkv, g, w, L, budget, pool=7):
    return W.Workload("t", 2, Hkv=Hkv, Hq=Hkv * g, L=L, w=w, budget=budget, pool=pool)


def filled(*rows):
    """Rows of a value that no input holds: what a call does not write shows."""
    return torch.full((*rows, 128), 7.0e30, dtype=torch.bfloat16, device="cuda")


def indices(*rows):
    return torch.full(rows, -1, dtype=torch.int32, device="cuda")


# few heads (a cluster each) and many (a CTA each up to pool 9, clusters again beyond); budgets below and above the prefix
@pytest.mark.parametrize("Hkv,g,w,L,budget,pool", [(2, 4, 32, 13001, 700, 7), (3, 2, 5, 12290, 13000, 7), (1, 4, 64, 30011, 2000, 13),
                                                   (129, 1, 3, 12291, 130, 9), (130, 1, 4, 12289, 20000, 7), (129, 1, 2, 12293, 99, 11)])
def test_window_kept_in_two_launches(Hkv, g, w, L, budget, pool):
    wl = wl_of(Hkv, g, w, L, budget, pool)
    K, V, Q, _ = W.make_layer(wl)
    Kw = W.make_window_keys(wl, Q)
    Vw = W.make_v(wl_of(Hkv, g, w, w, 1), 77)
    s = shape_of(wl)
    np_ = min(budget - w, L)
    Ko, Vo, idx = filled(Hkv, np_ + w), filled(Hkv, np_ + w), indices(Hkv, np_)
    ws = jq.new_workspace(s)
    n0 = jq.launch_count()
    jq.evict_layer_window_kept(dev_bf16(K), dev_bf16(V), dev_bf16(Q), dev_bf16(Kw), dev_bf16(Vw), s, Ko, Vo, idx, ws)
    assert jq.launch_count() - n0 == 2 and jq.last_device_status(ws) == jq.JQ_OK
    gi, gK, gV = idx.cpu().numpy(), host_bits(Ko), host_bits(Vo)
    pooled = oracle.pool(oracle.score_windowed(K, Q, Kw), pool)
    assert_kept_sets_agree(gi, oracle.select(pooled, np_), pooled, np_)
    for kv in range(Hkv):
        assert np.array_equal(gK[kv, :np_], K[kv][gi[kv]]) and np.array_equal(gV[kv, :np_], V[kv][gi[kv]])
        assert np.array_equal(gK[kv, np_:], Kw[kv]) and np.array_equal(gV[kv, np_:], Vw[kv])


@pytest.mark.parametrize("Hkv,g,w,L,budget,pool", [(2, 4, 32, 13001, 700, 7), (1, 4, 64, 20011, 25000, 5)])
def test_windowed_in_two_launches(Hkv, g, w, L, budget, pool):
    wl = wl_of(Hkv, g, w, L, budget, pool)
    K, V, Q, _ = W.make_layer(wl)
    Kw = W.make_window_keys(wl, Q)
    s = shape_of(wl)
    Ko, Vo, idx = filled(Hkv, wl.nkeep), filled(Hkv, wl.nkeep), indices(Hkv, wl.nkeep)
    ws = jq.new_workspace(s)
    n0 = jq.launch_count()
    jq.evict_layer_windowed(dev_bf16(K), dev_bf16(V), dev_bf16(Q), dev_bf16(Kw), s, Ko, Vo, idx, ws)
    assert jq.launch_count() - n0 == 2 and jq.last_device_status(ws) == jq.JQ_OK
    gi, gK, gV = idx.cpu().numpy(), host_bits(Ko), host_bits(Vo)
    pooled = oracle.pool(oracle.score_windowed(K, Q, Kw), pool)
    assert_kept_sets_agree(gi, oracle.select(pooled, budget), pooled, wl.nkeep)
    for kv in range(Hkv):
        assert np.array_equal(gK[kv], K[kv][gi[kv]]) and np.array_equal(gV[kv], V[kv][gi[kv]])


# n_old no multiple of anything, a cache with room behind the rows and one without, no new rows, everything kept, many heads
@pytest.mark.parametrize("Hkv,g,w,n_old,n_new,budget,cap", [(2, 4, 32, 12000, 1001, 12000, 13500), (1, 4, 64, 9001, 5000, 700, 14001), (3, 2, 5, 12300, 0, 4000, 12400),
                                                             (2, 4, 16, 12288, 1, 13000, 12289), (130, 1, 2, 12200, 100, 50, 12303)])
def test_append_in_two_launches(Hkv, g, w, n_old, n_new, budget, cap):
    wl = wl_of(Hkv, g, w, n_old + n_new, budget)
    K, V, Q, _ = W.make_layer(wl, layer=2)
    s = shape_of(wl)
    Kc, Vc, idx = filled(Hkv, cap), filled(Hkv, cap), indices(Hkv, wl.nkeep)
    Kc[:, :n_old] = dev_bf16(K[:, :n_old]); Vc[:, :n_old] = dev_bf16(V[:, :n_old])
    Kn, Vn = (dev_bf16(K[:, n_old:]), dev_bf16(V[:, n_old:])) if n_new else (None, None)
    ws = jq.new_append_workspace(s)
    n0 = jq.launch_count()
    jq.evict_append(Kc, Vc, n_old, Kn, Vn, dev_bf16(Q), s, idx, ws)
    assert jq.launch_count() - n0 == 2 and jq.last_device_status(ws) == jq.JQ_OK
    gi = idx.cpu().numpy()
    pooled = oracle.pool(oracle.score(K, Q), wl.pool)
    assert_kept_sets_agree(gi, oracle.select(pooled, budget), pooled, wl.nkeep)
    gK, gV = host_bits(Kc), host_bits(Vc)
    for kv in range(Hkv):
        assert np.array_equal(gK[kv, :wl.nkeep], K[kv][gi[kv]]) and np.array_equal(gV[kv, :wl.nkeep], V[kv][gi[kv]])
