"""The eviction in one pass over the keys (row_stats, block_bounds, score_candidates, a selection): the scores of the keys that can be
kept, found through bounds per block of 16 keys.  The kept sets are the oracle's under the end-to-end rule of gpu_util, and those of
jq_score -> jq_select_topk except among positions whose scores agree to fp32 rounding."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

import oracle
import jq_workloads as W
import paper_2509_10798_b200 as jq
from gpu_util import assert_kept_sets_agree, dev_bf16, gpu_select, host_bits, shape_of

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
LAUNCHES = 4


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as entry
    entry.build()


def wl_of(Hkv, g, w, L, budget, pool=7):
    return W.Workload("t", 2, Hkv=Hkv, Hq=Hkv * g, L=L, w=w, budget=budget, pool=pool)


def device_layer(Hkv, g, w, L, seed):
    """Keys with four outlier channels per head, queries that lean towards 64 keys of their head (too many keys for the host's generator)."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    K = torch.randn((Hkv, L, 128), generator=gen, device="cuda", dtype=torch.float32)
    for h in range(Hkv):
        K[h, :, torch.randperm(128, generator=gen, device="cuda")[:4]] *= 8.0
    K = K.to(torch.bfloat16)
    at = torch.randint(0, L, (Hkv, 64), generator=gen, device="cuda")
    near = torch.stack([K[h, at[h, torch.arange(g * w, device="cuda") % 64]] for h in range(Hkv)]).float()
    Q = (0.7 * torch.randn(near.shape, generator=gen, device="cuda") + 0.3 * near).to(torch.bfloat16).reshape(Hkv * g, w, 128)
    V = torch.randn((Hkv, L, 128), generator=gen, device="cuda", dtype=torch.float32).to(torch.bfloat16)
    return K, V, Q.contiguous()


def two_pass(K, Q, s):
    """Scores of the two-pass kernel, and the positions that a selection on them keeps."""
    sc = torch.empty((s.Hkv, s.L), dtype=torch.float32, device="cuda")
    ws = jq.new_workspace(s)
    jq.score(K, Q, s, sc, ws)
    assert jq.last_device_status(ws) == jq.JQ_OK
    sc = sc.cpu().numpy()
    return sc, gpu_select(sc, s, want_pooled=False)[0]


def check(K, V, Q, s, Ko, Vo, idx, oracle_heads):
    sc, want = two_pass(K, Q, s)
    pooled = oracle.pool(sc.astype(np.float64), s.pool)
    gi = idx.cpu().numpy()
    assert_kept_sets_agree(gi, want, pooled, gi.shape[1])
    at = idx.long()[:, :, None].expand(-1, -1, 128)
    assert torch.equal(Ko, torch.gather(K, 1, at)) and torch.equal(Vo, torch.gather(V, 1, at))
    g = s.group
    for kv in oracle_heads:
        po = oracle.pool(oracle.score(host_bits(K[kv:kv + 1]), host_bits(Q[kv * g:(kv + 1) * g])), s.pool)
        assert_kept_sets_agree(gi[kv:kv + 1], oracle.select(po, s.budget), po, gi.shape[1])


# a cluster per head and a CTA per head; up to 128 query rows and more; lengths around a multiple of 16 and of 128; windows of 1 to 63
@pytest.mark.parametrize("Hkv,g,w,L,budget,pool", [
    (8, 4, 64, 65537, 500, 7), (8, 4, 32, 100001, 300, 7), (2, 4, 64, 300015, 900, 9), (70, 1, 8, 11279, 64, 7), (40, 7, 20, 20033, 300, 13),
    (66, 2, 64, 12160, 100, 63), (129, 1, 33, 10001, 40, 1), (130, 3, 11, 10240, 100, 3), (150, 4, 33, 10017, 90, 5)])
def test_layer(Hkv, g, w, L, budget, pool):
    K, V, Q = device_layer(Hkv, g, w, L, 7)
    s = shape_of(wl_of(Hkv, g, w, L, budget, pool))
    Ko, Vo = (torch.zeros((Hkv, budget, 128), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    idx = torch.full((Hkv, budget), -1, dtype=torch.int32, device="cuda")
    ws = jq.new_workspace(s)
    n0 = jq.launch_count()
    jq.evict_layer(K, V, Q, s, Ko, Vo, idx, ws)
    assert jq.launch_count() - n0 == LAUNCHES and jq.last_device_status(ws) == jq.JQ_OK
    check(K, V, Q, s, Ko, Vo, idx, (0, Hkv - 1))


@pytest.mark.parametrize("scale", [0.0, 1e-3, 3e4])   # no bound separates; hardly any does; logits that a half cannot hold
@pytest.mark.parametrize("Hkv,g,w,L,budget", [(66, 4, 32, 11000, 100), (8, 4, 64, 66000, 300)])
def test_layer_whose_bounds_say_nothing(scale, Hkv, g, w, L, budget):
    K, V, Q = device_layer(Hkv, g, w, L, 3)
    Q = (Q.float() * scale).to(torch.bfloat16)
    s = shape_of(wl_of(Hkv, g, w, L, budget))
    Ko, Vo = (torch.zeros((Hkv, budget, 128), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    idx = torch.full((Hkv, budget), -1, dtype=torch.int32, device="cuda")
    ws = jq.new_workspace(s)
    n0 = jq.launch_count()
    jq.evict_layer(K, V, Q, s, Ko, Vo, idx, ws)
    assert jq.launch_count() - n0 == LAUNCHES and jq.last_device_status(ws) == jq.JQ_OK
    if scale == 0.0:
        # equal scores but for rounding, which follows the order of the additions: any kept set of the right size in the rule of gpu_util
        sc, _ = two_pass(K, Q, s)
        assert np.ptp(sc) <= 1e-5 * sc.max()
        gi = idx.cpu().numpy()
        assert np.all(np.diff(gi, axis=1) > 0) and gi.min() >= 0 and gi.max() < L
        return
    check(K, V, Q, s, Ko, Vo, idx, ())


def test_ragged_units():
    """Units of different lengths and budgets: long ones, one of a single key, budgets at and above the length, a last block of one key."""
    Hkv, g, w = 8, 4, 32
    Ls, Bs = [20000, 17, 30017, 1, 40961, 128, 25000, 30001], [200, 17, 300, 5, 64, 1000, 1, 400]
    units = [device_layer(Hkv, g, w, L, 11 + i) for i, L in enumerate(Ls)]
    s = shape_of(wl_of(Hkv, g, w, max(Ls), max(Bs)))
    rows = jq.ragged_output_rows(s, len(Ls), Ls, Bs)
    Ko, Vo = (torch.zeros((rows, 128), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    idx = torch.full((rows,), -1, dtype=torch.int32, device="cuda")
    ws = jq.new_ragged_workspace(s, len(Ls), Ls)
    n0 = jq.launch_count()
    jq.evict_ragged([u[0] for u in units], [u[1] for u in units], [u[2] for u in units], s, Ls, Bs, Ko, Vo, idx, ws)
    assert jq.launch_count() - n0 == LAUNCHES and jq.last_device_status(ws) == jq.JQ_OK
    r0 = 0
    for (K, V, Q), L, B in zip(units, Ls, Bs):
        n = min(B, L)
        r1 = r0 + Hkv * n
        check(K, V, Q, shape_of(wl_of(Hkv, g, w, L, B)), Ko[r0:r1].view(Hkv, n, 128), Vo[r0:r1].view(Hkv, n, 128), idx[r0:r1].view(Hkv, n), (0,))
        r0 = r1


@pytest.mark.parametrize("Hkv,g,w,L,budget", [(8, 4, 64, 66001, 400), (130, 2, 16, 10100, 100)])
def test_window_kept(Hkv, g, w, L, budget):
    K, V, Q = device_layer(Hkv, g, w, L, 5)
    Kw, Vw = (torch.randn((Hkv, w, 128), device="cuda").to(torch.bfloat16) for _ in range(2))
    s = shape_of(wl_of(Hkv, g, w, L, budget + w))
    Ko, Vo = (torch.zeros((Hkv, budget + w, 128), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    idx = torch.full((Hkv, budget), -1, dtype=torch.int32, device="cuda")
    ws = jq.new_workspace(s)
    n0 = jq.launch_count()
    jq.evict_layer_window_kept(K, V, Q, Kw, Vw, s, Ko, Vo, idx, ws)
    assert jq.launch_count() - n0 == LAUNCHES and jq.last_device_status(ws) == jq.JQ_OK
    gi = idx.cpu().numpy()
    for kv in (0, Hkv - 1):
        po = oracle.pool(oracle.score_windowed(host_bits(K[kv:kv + 1]), host_bits(Q[kv * g:(kv + 1) * g]), host_bits(Kw[kv:kv + 1])), s.pool)
        assert_kept_sets_agree(gi[kv:kv + 1], oracle.select(po, budget), po, budget)
    at = idx.long()[:, :, None].expand(-1, -1, 128)
    assert torch.equal(Ko[:, :budget], torch.gather(K, 1, at)) and torch.equal(Vo[:, :budget], torch.gather(V, 1, at))
    assert torch.equal(Ko[:, budget:], Kw) and torch.equal(Vo[:, budget:], Vw)


def test_append_to_a_long_cache():
    Hkv, g, w, n_old, n_new, budget, cap = 8, 4, 64, 65000, 1001, 300, 66100
    K, V, Q = device_layer(Hkv, g, w, n_old + n_new, 9)
    s = shape_of(wl_of(Hkv, g, w, n_old + n_new, budget))
    Kc, Vc = (torch.zeros((Hkv, cap, 128), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    Kc[:, :n_old] = K[:, :n_old]; Vc[:, :n_old] = V[:, :n_old]
    idx = torch.full((Hkv, budget), -1, dtype=torch.int32, device="cuda")
    ws = jq.new_append_workspace(s)
    n0 = jq.launch_count()
    jq.evict_append(Kc, Vc, n_old, K[:, n_old:].contiguous(), V[:, n_old:].contiguous(), Q, s, idx, ws)
    assert jq.launch_count() - n0 == LAUNCHES and jq.last_device_status(ws) == jq.JQ_OK
    check(K, V, Q, s, Kc[:, :budget], Vc[:, :budget], idx, (3,))


def test_a_workspace_without_room_for_it_goes_the_other_way():
    """What the two-pass kernels need is enough for every call, as it was: status, normalisers, partial statistics, scores, keys."""
    Hkv, g, w, L, budget = 8, 4, 64, 65537, 500
    K, V, Q = device_layer(Hkv, g, w, L, 4)
    s = shape_of(wl_of(Hkv, g, w, L, budget))
    up = lambda x: (x + 255) // 256 * 256
    least = 256 + up(Hkv * g * w * 4) + up(Hkv * 640 * g * w * 8) + 2 * up(Hkv * L * 4)
    assert least < jq.workspace_bytes(s)
    kept = []
    for size, launches in ((least, 2), (jq.workspace_bytes(s), LAUNCHES)):
        ws = torch.empty(size, dtype=torch.uint8, device="cuda")
        jq._raise("jq_workspace_init", jq.lib().jq_workspace_init(jq._ptr(ws), ws.numel(), jq._stream(None)))
        Ko, Vo = (torch.zeros((Hkv, budget, 128), dtype=torch.bfloat16, device="cuda") for _ in range(2))
        idx = torch.full((Hkv, budget), -1, dtype=torch.int32, device="cuda")
        n0 = jq.launch_count()
        jq.evict_layer(K, V, Q, s, Ko, Vo, idx, ws)
        assert jq.launch_count() - n0 == launches and jq.last_device_status(ws) == jq.JQ_OK
        check(K, V, Q, s, Ko, Vo, idx, ())
        kept.append(idx)
    with pytest.raises(jq.JqError):
        jq.evict_layer(K, V, Q, s, Ko, Vo, idx, torch.empty(least - 256, dtype=torch.uint8, device="cuda"))


@pytest.mark.parametrize("Ls,budget,launches", [([80000, 17, 60017], 300, LAUNCHES), ([3000, 130, 5000], 64, 2)])
def test_units_in_a_workspace_without_room_for_it(Ls, budget, launches):
    """The same for calls over several units: the tables of the two-pass kernels are all that has to fit behind the scratch."""
    Hkv, g, w, n = 8, 4, 32, len(Ls)
    units = [device_layer(Hkv, g, w, L, 21 + i) for i, L in enumerate(Ls)]
    s = shape_of(wl_of(Hkv, g, w, max(Ls), budget))
    up = lambda x: (x + 255) // 256 * 256
    heads, R = n * Hkv, g * w
    least = 256 + up(heads * R * 4) + up(heads * 640 * R * 8) + 2 * up(Hkv * sum(Ls) * 4)
    least += up(n * 2 * 128) + 2 * up(n * 8) + up(heads * 40) + up(heads * 32)
    rows = jq.ragged_output_rows(s, n, Ls, [budget] * n)
    for size, count in ((least, 2), (jq.ragged_workspace_bytes(s, n, Ls), launches)):
        ws = torch.empty(size, dtype=torch.uint8, device="cuda")
        jq._raise("jq_workspace_init", jq.lib().jq_workspace_init(jq._ptr(ws), ws.numel(), jq._stream(None)))
        Ko, Vo = (torch.zeros((rows, 128), dtype=torch.bfloat16, device="cuda") for _ in range(2))
        idx = torch.full((rows,), -1, dtype=torch.int32, device="cuda")
        n0 = jq.launch_count()
        jq.evict_ragged([u[0] for u in units], [u[1] for u in units], [u[2] for u in units], s, Ls, [budget] * n, Ko, Vo, idx, ws)
        assert jq.launch_count() - n0 == count and jq.last_device_status(ws) == jq.JQ_OK
        r0 = 0
        for (K, V, Q), L in zip(units, Ls):
            k = min(budget, L)
            r1 = r0 + Hkv * k
            check(K, V, Q, shape_of(wl_of(Hkv, g, w, L, budget)), Ko[r0:r1].view(Hkv, k, 128), Vo[r0:r1].view(Hkv, k, 128), idx[r0:r1].view(Hkv, k), ())
            r0 = r1


def test_a_host_call_with_a_buffer_without_room_for_it():
    """The device buffer of a call on host tensors: K, V, queries, the kept rows, the indices, and what the two-pass kernels need."""
    Hkv, g, w, L, budget = 8, 4, 64, 65537, 500
    K, V, Q = device_layer(Hkv, g, w, L, 4)
    s = shape_of(wl_of(Hkv, g, w, L, budget))
    up = lambda x: (x + 255) // 256 * 256
    least = 2 * up(Hkv * L * 256) + up(Hkv * g * w * 256) + 2 * up(Hkv * budget * 256) + up(Hkv * budget * 4) + 256
    least += 256 + up(Hkv * g * w * 4) + up(Hkv * 640 * g * w * 8) + 2 * up(Hkv * L * 4)
    assert least < jq.host_call_bytes(s)
    host = [x.cpu().pin_memory() for x in (K, V, Q)]
    for size in (least, jq.host_call_bytes(s)):
        out = [torch.zeros((Hkv, budget, 128), dtype=torch.bfloat16).pin_memory() for _ in range(2)] + [torch.full((Hkv, budget), -1, dtype=torch.int32).pin_memory()]
        jq.evict_layer_host(*host, s, *out, torch.empty(size, dtype=torch.uint8, device="cuda"))
        torch.cuda.synchronize()
        check(K, V, Q, s, *(x.cuda() for x in out), ())
    with pytest.raises(jq.JqError):
        jq.evict_layer_host(*host, s, *out, torch.empty(least - 256, dtype=torch.uint8, device="cuda"))


def test_in_a_graph_and_on_two_streams():
    """Captured once and replayed on other inputs in the same buffers, while another stream evicts with a workspace of its own."""
    Hkv, g, w, L, budget = 70, 1, 32, 11264, 64
    s = shape_of(wl_of(Hkv, g, w, L, budget))
    A, B, C = (device_layer(Hkv, g, w, L, i) for i in (1, 2, 3))
    out = [[torch.zeros((Hkv, budget, 128), dtype=torch.bfloat16, device="cuda") for _ in range(2)] + [torch.zeros((Hkv, budget), dtype=torch.int32, device="cuda")] for _ in range(2)]
    ws = [jq.new_workspace(s) for _ in range(2)]
    buf = [x.clone() for x in A]
    jq.evict_layer(*buf, s, *out[0], ws[0])
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        jq.evict_layer(*buf, s, *out[0], ws[0])
    for x, y in zip(buf, B):
        x.copy_(y)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    for _ in range(20):
        graph.replay()
        with torch.cuda.stream(side):
            jq.evict_layer(*C, s, *out[1], ws[1])
    torch.cuda.synchronize()
    for (K, V, Q), o, x in zip((B, C), out, ws):
        assert jq.last_device_status(x) == jq.JQ_OK
        check(K, V, Q, s, o[0], o[1], o[2], ())


@pytest.mark.parametrize("Hkv,g,w,L,budget,pool", [(66, 4, 32, 11000, 100, 7), (8, 4, 64, 66000, 300, 7), (130, 2, 16, 10100, 77, 5), (9, 1, 32, 90001, 500, 13)])
def test_equal_scores_keep_the_lowest_positions(Hkv, g, w, L, budget, pool):
    """Q = 0: every score is the same number, every block a candidate, and the first `budget` positions stay."""
    K, V, Q = device_layer(Hkv, g, w, L, 3)
    s = shape_of(wl_of(Hkv, g, w, L, budget, pool))
    Ko, Vo = (torch.zeros((Hkv, budget, 128), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    idx = torch.full((Hkv, budget), -1, dtype=torch.int32, device="cuda")
    ws = jq.new_workspace(s)
    n0 = jq.launch_count()
    jq.evict_layer(K, V, torch.zeros_like(Q), s, Ko, Vo, idx, ws)
    assert jq.launch_count() - n0 == LAUNCHES and jq.last_device_status(ws) == jq.JQ_OK
    assert torch.equal(idx, torch.arange(budget, dtype=torch.int32, device="cuda").expand(Hkv, -1))
    assert torch.equal(Ko, K[:, :budget]) and torch.equal(Vo, V[:, :budget])


# logits that are what is left of products that cancel, in the first and the last of eight steps of the product: the sum of |q k| is 2 a b,
# and what is lost of it in 32 bits is far more than the margin of the bounds (c 2^-24 2 a b against 1 / 512 in the exponent).  The same query
# in every row, so that a block's bound is the score of its best key and nothing more.
@pytest.mark.parametrize("a,b", [(256.0, 256.0), (2048.0, 1024.0), (8192.0, 8192.0)])
def test_logits_that_cancel(a, b):
    Hkv, g, w, L, budget = 70, 1, 8, 11279, 64
    K, V, Q = device_layer(Hkv, g, w, L, 6)
    gen = torch.Generator(device="cuda").manual_seed(1)
    big = (a * (1 + torch.rand((Hkv, L), generator=gen, device="cuda"))).to(torch.bfloat16)
    Q = Q[:, :1].expand(-1, w, -1).contiguous()
    K[:, :, 3] = big; K[:, :, 120] = big
    Q[:, :, 3] = b; Q[:, :, 120] = -b
    s = shape_of(wl_of(Hkv, g, w, L, budget))
    Ko, Vo = (torch.zeros((Hkv, budget, 128), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    idx = torch.full((Hkv, budget), -1, dtype=torch.int32, device="cuda")
    ws = jq.new_workspace(s)
    n0 = jq.launch_count()
    jq.evict_layer(K, V, Q, s, Ko, Vo, idx, ws)
    assert jq.launch_count() - n0 == LAUNCHES and jq.last_device_status(ws) == jq.JQ_OK
    check(K, V, Q, s, Ko, Vo, idx, ())


@pytest.mark.parametrize("Hkv,g,w,L,budget", [(8, 4, 64, 66001, 400), (130, 2, 16, 10100, 100)])
def test_windowed(Hkv, g, w, L, budget):
    K, V, Q = device_layer(Hkv, g, w, L, 5)
    Kw = torch.randn((Hkv, w, 128), device="cuda").to(torch.bfloat16)
    s = shape_of(wl_of(Hkv, g, w, L, budget))
    Ko, Vo = (torch.zeros((Hkv, budget, 128), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    idx = torch.full((Hkv, budget), -1, dtype=torch.int32, device="cuda")
    ws = jq.new_workspace(s)
    n0 = jq.launch_count()
    jq.evict_layer_windowed(K, V, Q, Kw, s, Ko, Vo, idx, ws)
    assert jq.launch_count() - n0 == LAUNCHES and jq.last_device_status(ws) == jq.JQ_OK
    gi = idx.cpu().numpy()
    for kv in (0, Hkv - 1):
        po = oracle.pool(oracle.score_windowed(host_bits(K[kv:kv + 1]), host_bits(Q[kv * g:(kv + 1) * g]), host_bits(Kw[kv:kv + 1])), s.pool)
        assert_kept_sets_agree(gi[kv:kv + 1], oracle.select(po, budget), po, budget)
    at = idx.long()[:, :, None].expand(-1, -1, 128)
    assert torch.equal(Ko, torch.gather(K, 1, at)) and torch.equal(Vo, torch.gather(V, 1, at))


# 136 heads in 17 units: the selection reads the scored blocks by their bits, of units of one length and of units whose tiles are
# numbered in another order than the call's (lengths that are no multiple of 16 or 128, a unit of one key, budgets at and above the length)
MANY_UNITS = {
    "one length": ([10100] * 17, [90] * 17),
    "two budgets": ([10100] * 17, [90, 130] * 8 + [1]),
    "lengths": ([10017, 20000, 17, 11279, 9001, 1, 30001, 12345, 128, 10100, 16384, 10017, 7777, 25001, 129, 10240, 20033], [90, 200, 17, 100, 64, 5, 300, 1, 1000, 90, 50, 91, 77, 250, 128, 100, 10]),
}


@pytest.mark.parametrize("units", sorted(MANY_UNITS))
def test_many_units_of_many_heads(units):
    Hkv, g, w = 8, 4, 32
    Ls, Bs = MANY_UNITS[units]
    U = [device_layer(Hkv, g, w, L, 31 + i) for i, L in enumerate(Ls)]
    s = shape_of(wl_of(Hkv, g, w, Ls[0], Bs[0]))
    rows = jq.ragged_output_rows(s, len(Ls), Ls, Bs)
    Ko, Vo = (torch.zeros((rows, 128), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    idx = torch.full((rows,), -1, dtype=torch.int32, device="cuda")
    ws = jq.new_ragged_workspace(s, len(Ls), Ls)
    n0 = jq.launch_count()
    if units == "one length":
        jq.evict_layers([u[0] for u in U], [u[1] for u in U], [u[2] for u in U], s, Ko, Vo, idx, ws)
    else:
        jq.evict_ragged([u[0] for u in U], [u[1] for u in U], [u[2] for u in U], s, Ls, Bs, Ko, Vo, idx, ws)
    assert jq.launch_count() - n0 == LAUNCHES and jq.last_device_status(ws) == jq.JQ_OK
    r0 = 0
    for i, ((K, V, Q), L, B) in enumerate(zip(U, Ls, Bs)):
        n = min(B, L)
        r1 = r0 + Hkv * n
        check(K, V, Q, shape_of(wl_of(Hkv, g, w, L, B)), Ko[r0:r1].view(Hkv, n, 128), Vo[r0:r1].view(Hkv, n, 128), idx[r0:r1].view(Hkv, n), (i % Hkv,))
        r0 = r1


SWEEP = r'''
import ctypes, os, sys
import torch
sys.path.insert(0, %(root)r)
sys.path.insert(0, os.path.join(%(root)r, "tests"))
import paper_2509_10798_b200 as jq
from paper_2509_10798_b200 import build
jq.LIB_PATH = build.build(debug=True)
from test_gpu_candidates import device_layer, wl_of
from gpu_util import shape_of
lib = jq.lib()
rec = (ctypes.c_longlong * 5)()
assert lib.jq_debug_reset() == 0
for Hkv, g, w, L, B, p, scale in [(8, 4, 64, 65537, 500, 7, 1.0), (8, 4, 64, 65537, 500, 7, 0.0), (70, 1, 8, 11279, 64, 7, 1.0), (40, 7, 20, 20033, 300, 13, 1.0),
                                  (129, 1, 33, 10001, 40, 1, 1.0), (130, 4, 33, 10017, 90, 5, 0.0)]:
    K, V, Q = device_layer(Hkv, g, w, L, 7)
    Q = (Q.float() * scale).to(torch.bfloat16)
    s = shape_of(wl_of(Hkv, g, w, L, B, p))
    Ko, Vo = (torch.zeros((Hkv, B, 128), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    idx = torch.zeros((Hkv, B), dtype=torch.int32, device="cuda")
    ws = jq.new_workspace(s)
    n0 = jq.launch_count()
    jq.evict_layer(K, V, Q, s, Ko, Vo, idx, ws)
    assert jq.launch_count() - n0 == 4 and jq.last_device_status(ws) == jq.JQ_OK
Ls, Bs = [20000, 17, 30017, 1, 40961, 128, 25000, 30001], [200, 17, 300, 5, 64, 1000, 1, 400]
u = [device_layer(8, 4, 32, L, 11) for L in Ls]
s = shape_of(wl_of(8, 4, 32, max(Ls), max(Bs)))
rows = jq.ragged_output_rows(s, len(Ls), Ls, Bs)
Ko, Vo = (torch.zeros((rows, 128), dtype=torch.bfloat16, device="cuda") for _ in range(2))
ws = jq.new_ragged_workspace(s, len(Ls), Ls)
jq.evict_ragged([x[0] for x in u], [x[1] for x in u], [x[2] for x in u], s, Ls, Bs, Ko, Vo, torch.zeros((rows,), dtype=torch.int32, device="cuda"), ws)
assert jq.last_device_status(ws) == jq.JQ_OK
assert lib.jq_debug_read(rec) == 0
print("DEBUG-SWEEP violations=%%d kernel=%%d site=%%d index=%%d extent=%%d" %% tuple(rec))
'''


def test_no_index_leaves_its_array_in_the_bounds_checked_build():
    out = subprocess.run([sys.executable, "-c", SWEEP % {"root": ROOT}], capture_output=True, text=True, timeout=900)
    assert out.returncode == 0, out.stdout[-2000:] + out.stderr[-4000:]
    line = [ln for ln in out.stdout.splitlines() if ln.startswith("DEBUG-SWEEP")]
    assert line and line[0].startswith("DEBUG-SWEEP violations=0 "), out.stdout[-2000:]


MANY_SWEEP = SWEEP[:SWEEP.index("for Hkv, g, w, L, B, p, scale in")] + r'''
from test_gpu_candidates import MANY_UNITS
for Ls, Bs in MANY_UNITS.values():
    for scale in (1.0, 0.0):
        u = [device_layer(8, 4, 32, L, 11) for L in Ls]
        s = shape_of(wl_of(8, 4, 32, Ls[0], Bs[0]))
        rows = jq.ragged_output_rows(s, len(Ls), Ls, Bs)
        Ko, Vo = (torch.zeros((rows, 128), dtype=torch.bfloat16, device="cuda") for _ in range(2))
        ws = jq.new_ragged_workspace(s, len(Ls), Ls)
        n0 = jq.launch_count()
        jq.evict_ragged([x[0] for x in u], [x[1] for x in u], [(x[2].float() * scale).to(torch.bfloat16) for x in u], s, Ls, Bs, Ko, Vo, torch.zeros((rows,), dtype=torch.int32, device="cuda"), ws)
        assert jq.launch_count() - n0 == 4 and jq.last_device_status(ws) == jq.JQ_OK
K, V, Q = device_layer(130, 2, 16, 10100, 5)
Kw = torch.randn((130, 16, 128), device="cuda").to(torch.bfloat16)
s = shape_of(wl_of(130, 2, 16, 10100, 100))
Ko, Vo = (torch.zeros((130, 100, 128), dtype=torch.bfloat16, device="cuda") for _ in range(2))
ws = jq.new_workspace(s)
jq.evict_layer_windowed(K, V, Q, Kw, s, Ko, Vo, torch.zeros((130, 100), dtype=torch.int32, device="cuda"), ws)
assert jq.last_device_status(ws) == jq.JQ_OK
''' + SWEEP[SWEEP.index("assert lib.jq_debug_read(rec) == 0"):]


def test_no_index_leaves_its_array_with_many_units():
    out = subprocess.run([sys.executable, "-c", MANY_SWEEP % {"root": ROOT}], capture_output=True, text=True, timeout=900)
    assert out.returncode == 0, out.stdout[-2000:] + out.stderr[-4000:]
    line = [ln for ln in out.stdout.splitlines() if ln.startswith("DEBUG-SWEEP")]
    assert line and line[0].startswith("DEBUG-SWEEP violations=0 "), out.stdout[-2000:]
