"""The one-launch layer pass (a cluster per KV head, csrc/jq_fused.cu) and the clustered decoding step at the sizes where they
can go wrong: tile and quad edges, parts whose lengths are no multiple of anything, every cluster size, budgets that make
the in-place move take several steps, tied scores.  Against the fp64 oracle under the end-to-end rule of gpu_util."""
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


def outputs(Hkv, rows, nidx):
    return (torch.zeros((Hkv, rows, 128), dtype=torch.bfloat16, device="cuda"), torch.zeros((Hkv, rows, 128), dtype=torch.bfloat16, device="cuda"),
            torch.full((Hkv, nidx), -1, dtype=torch.int32, device="cuda"))


# Hkv, g, w, L, budget, pool: L around a tile, around 2 and 4 tiles per CTA, up to the longest the kernel takes; one head and more
# heads than clusters fit at a time; one and two blocks of query rows, rows that are no multiple of 32; pools on both code paths
CASES = [(1, 1, 1, 1, 1, 1), (1, 1, 3, 5, 2, 3), (2, 4, 16, 127, 40, 7), (2, 4, 16, 128, 128, 7), (2, 4, 32, 129, 128, 7),
         (3, 4, 33, 257, 100, 9), (2, 4, 16, 2048, 256, 7), (1, 8, 32, 2049, 64, 7), (8, 4, 32, 1025, 1000, 5), (5, 7, 36, 1500, 333, 11),
         (2, 4, 8, 4096, 4095, 63), (8, 4, 32, 4097, 512, 7), (8, 4, 64, 3001, 700, 7), (4, 4, 32, 12288, 2048, 7), (40, 2, 32, 513, 50, 7),
         (2, 1, 5, 6001, 1, 7)]


@pytest.mark.parametrize("Hkv,g,w,L,budget,pool", CASES)
def test_layer_in_one_launch(Hkv, g, w, L, budget, pool):
    wl = wl_of(Hkv, g, w, L, budget, pool)
    K, V, Q, _ = W.make_layer(wl)
    s = shape_of(wl)
    Ko, Vo, idx = outputs(Hkv, wl.nkeep, wl.nkeep)
    ws = jq.new_workspace(s)
    n0 = jq.launch_count()
    jq.evict_layer(dev_bf16(K), dev_bf16(V), dev_bf16(Q), s, Ko, Vo, idx, ws)
    assert jq.last_device_status(ws) == jq.JQ_OK
    assert jq.launch_count() - n0 == 1
    pooled = oracle.pool(oracle.score(K, Q), pool)
    gi = idx.cpu().numpy()
    assert_kept_sets_agree(gi, oracle.select(pooled, budget), pooled, wl.nkeep)
    gK, gV = host_bits(Ko), host_bits(Vo)
    for kv in range(Hkv):
        assert np.array_equal(gK[kv], K[kv][gi[kv]]) and np.array_equal(gV[kv], V[kv][gi[kv]])


# windows wider than nine: every remainder of the radius modulo the quad, windows wider than the prefix, prefixes that end
# anywhere in a quad
@pytest.mark.parametrize("pool", [11, 13, 15, 17, 19, 31, 61, 63])
@pytest.mark.parametrize("L,budget", [(3, 2), (30, 7), (1027, 200), (4098, 999)])
def test_wide_pools_in_one_launch(pool, L, budget):
    wl = wl_of(2, 4, 8, L, budget, pool)
    K, V, Q, _ = W.make_layer(wl)
    s = shape_of(wl)
    Ko, Vo, idx = outputs(2, budget, budget)
    n0 = jq.launch_count()
    jq.evict_layer(dev_bf16(K), dev_bf16(V), dev_bf16(Q), s, Ko, Vo, idx, jq.new_workspace(s))
    assert jq.launch_count() - n0 == 1
    pooled = oracle.pool(oracle.score(K, Q), pool)
    assert_kept_sets_agree(idx.cpu().numpy(), oracle.select(pooled, budget), pooled, budget)


@pytest.mark.parametrize("L,budget", [(700, 100), (4096, 513), (9000, 2048)])
def test_tied_scores_keep_the_lowest_positions(L, budget):
    """Equal keys give equal scores: with Q = 0 every pooled score is the same number, and the first `budget` positions stay."""
    wl = wl_of(2, 4, 16, L, budget)
    K, V, Q, _ = W.make_layer(wl)
    s = shape_of(wl)
    Ko, Vo, idx = outputs(2, budget, budget)
    jq.evict_layer(dev_bf16(K), dev_bf16(V), dev_bf16(np.zeros_like(Q)), s, Ko, Vo, idx, jq.new_workspace(s))
    assert np.array_equal(idx.cpu().numpy(), np.tile(np.arange(budget), (2, 1)))


def in_the_first_bin(pooled, budget):
    """Keys in the threshold's bin when the range of a head's pooled scores (as 32-bit patterns) is cut into 2048."""
    k = np.sort(pooled.astype(np.float32).view(np.uint32).astype(np.int64))[::-1]
    width = int(k[0] - k[-1])
    sh = max(width.bit_length() - 11, 0)
    return int(np.sum((k - k[-1]) >> sh == (k[budget - 1] - k[-1]) >> sh))


# a flat head with a dominant key: most scores fall into one of 2048 bins, which has to be cut again.  With equal keys around
# the threshold (a run of copies of one row, or copies all over) the third cut ends at a single value, kept by position.
@pytest.mark.parametrize("L,budget,pool", [(4096, 1000, 1), (10000, 3000, 1), (9001, 4500, 3)])
@pytest.mark.parametrize("copies", ["none", "run", "spread"])
def test_a_threshold_among_nearly_equal_scores(L, budget, pool, copies):
    wl = wl_of(1, 2, 8, L, budget, pool)
    rng = np.random.default_rng(L)
    Kf = rng.standard_normal((1, L, 128)).astype(np.float32)
    Qf = 2e-3 * rng.standard_normal((2, 8, 128)).astype(np.float32)         # logits of about 2e-3: scores within a per mille or two
    Kf[0, 5] = 10 * 11.3 * Qf[0, 0] / np.sum(Qf[0, 0] ** 2)                 # and a key with a logit of 10 for one query row
    at = np.arange(0)
    if copies != "none":
        at = np.arange(100, 1600) if copies == "run" else np.sort(rng.choice(np.arange(6, L - 1), 1500, replace=False))
        Kf[0, at] = 0.1 * Kf[0, L - 1]
    K, Q, V = W.bf16_bits(Kf), W.bf16_bits(Qf), W.make_v(wl, 3)
    pooled = oracle.pool(oracle.score(K, Q), pool)
    if len(at):                                                             # the threshold in the middle of the copies
        budget = int(np.sum(pooled[0] > pooled[0, at].min())) + int(np.sum(pooled[0] == pooled[0, at].min())) // 2
    assert in_the_first_bin(pooled[0], budget) > 512
    s = shape_of(wl.with_budget(budget))
    Ko, Vo, idx = outputs(1, budget, budget)
    n0 = jq.launch_count()
    jq.evict_layer(dev_bf16(K), dev_bf16(V), dev_bf16(Q), s, Ko, Vo, idx, jq.new_workspace(s))
    assert jq.launch_count() - n0 == 1
    gi = idx.cpu().numpy()
    # sums of 16 terms of equal size in 32 bits, against an exact normaliser: 16 x 2^-24 and the 2^-22 of an exponential
    kth = np.sort(pooled[0])[L - budget]
    diff = np.setxor1d(gi[0], oracle.select(pooled, budget)[0])
    assert np.all(np.diff(gi[0]) > 0) and np.all(np.abs(pooled[0, diff] - kth) <= 2e-6 * kth)
    assert np.array_equal(host_bits(Ko)[0], K[0][gi[0]]) and np.array_equal(host_bits(Vo)[0], V[0][gi[0]])
    if len(at) and pool == 1:                                               # of equal rows the lowest positions stay
        kept = np.isin(at, gi[0])
        assert 0 < np.sum(kept) < len(at) and np.all(kept[:-1] >= kept[1:])


@pytest.mark.parametrize("Hkv,g,w,L,budget", [(2, 4, 32, 128, 64), (8, 4, 32, 1000, 300), (2, 2, 128, 2500, 700), (3, 4, 64, 5001, 900)])
def test_window_kept_in_one_launch(Hkv, g, w, L, budget):
    wl = wl_of(Hkv, g, w, L, budget)
    if budget <= w:
        wl = wl.with_budget(w + 5)
    K, V, Q, _ = W.make_layer(wl)
    Kw = W.make_window_keys(wl, Q)
    Vw = W.make_v(wl_of(Hkv, g, w, w, 1), 77)
    s = shape_of(wl)
    np_ = min(wl.budget - w, L)
    Ko, Vo, _ = outputs(Hkv, np_ + w, 1)
    idx = torch.full((Hkv, np_), -1, dtype=torch.int32, device="cuda")
    ws = jq.new_workspace(s)
    jq.evict_layer_window_kept(dev_bf16(K), dev_bf16(V), dev_bf16(Q), dev_bf16(Kw), dev_bf16(Vw), s, Ko, Vo, idx, ws)
    assert jq.last_device_status(ws) == jq.JQ_OK
    gi, gK, gV = idx.cpu().numpy(), host_bits(Ko), host_bits(Vo)
    pooled = oracle.pool(oracle.score_windowed(K, Q, Kw), wl.pool)
    assert_kept_sets_agree(gi, oracle.select(pooled, np_), pooled, np_)
    for kv in range(Hkv):
        assert np.array_equal(gK[kv, :np_], K[kv][gi[kv]]) and np.array_equal(gV[kv, :np_], V[kv][gi[kv]])
        assert np.array_equal(gK[kv, np_:], Kw[kv]) and np.array_equal(gV[kv, np_:], Vw[kv])


# n_old, n_new: parts that end inside a tile and inside a quad; everything kept; a move of several steps (many rows)
@pytest.mark.parametrize("Hkv,g,w,n_old,n_new,budget,cap", [(2, 4, 32, 129, 127, 200, 256), (2, 4, 32, 130, 3, 133, 200), (8, 4, 32, 1021, 257, 1021, 1300),
                                                             (1, 4, 64, 4096, 1000, 4096, 5200), (2, 2, 16, 3, 2000, 1500, 2003), (2, 4, 16, 0, 300, 100, 300),
                                                             (1, 4, 32, 9000, 3000, 11000, 12000)])
def test_append_in_one_launch(Hkv, g, w, n_old, n_new, budget, cap):
    wl = wl_of(Hkv, g, w, n_old + n_new, budget)
    K, V, Q, _ = W.make_layer(wl, layer=2)
    s = shape_of(wl)
    Kc = torch.zeros((Hkv, cap, 128), dtype=torch.bfloat16, device="cuda")
    Vc = torch.zeros_like(Kc)
    Kc[:, :n_old] = dev_bf16(K[:, :n_old]); Vc[:, :n_old] = dev_bf16(V[:, :n_old])
    idx = torch.full((Hkv, wl.nkeep), -1, dtype=torch.int32, device="cuda")
    ws = jq.new_append_workspace(s)
    n0 = jq.launch_count()
    jq.evict_append(Kc, Vc, n_old, dev_bf16(K[:, n_old:]), dev_bf16(V[:, n_old:]), dev_bf16(Q), s, idx, ws)
    assert jq.last_device_status(ws) == jq.JQ_OK
    assert jq.launch_count() - n0 == 1
    gi = idx.cpu().numpy()
    pooled = oracle.pool(oracle.score(K, Q), wl.pool)
    assert_kept_sets_agree(gi, oracle.select(pooled, budget), pooled, wl.nkeep)
    gK, gV = host_bits(Kc), host_bits(Vc)
    for kv in range(Hkv):
        assert np.array_equal(gK[kv, :wl.nkeep], K[kv][gi[kv]]) and np.array_equal(gV[kv, :wl.nkeep], V[kv][gi[kv]])


# keys around a unit of 16 and around what one, two and sixteen CTAs of eight warps take at a time; groups on both sides of 4
@pytest.mark.parametrize("Hkv,group,n", [(1, 1, 1), (2, 4, 15), (2, 5, 16), (2, 8, 17), (3, 3, 129), (1, 4, 2049), (2, 7, 4100), (150, 2, 40), (40, 4, 700)])
def test_decode_step_edges(Hkv, group, n):
    rng = np.random.default_rng(n)
    Kc, Vc = W.bf16_bits(rng.standard_normal((Hkv, n, 128))), W.bf16_bits(rng.standard_normal((Hkv, n, 128)))
    q = W.bf16_bits(2.0 * rng.standard_normal((Hkv * group, 128)))
    out = torch.full((Hkv * group, 128), -1.0, dtype=torch.float32, device="cuda")
    ws = torch.empty(jq.decode_workspace_bytes(Hkv, Hkv * group, n), dtype=torch.uint8, device="cuda")
    jq.decode_attention(dev_bf16(Kc), dev_bf16(Vc), dev_bf16(q), out, ws)
    # fp32 sums of n <= 4100 terms whose weights add up to 1 (bounded by sqrt(n) 2^-24 of values of size 1) and ex2 (2 ulp)
    np.testing.assert_allclose(out.cpu().numpy(), oracle.decode_attention(Kc, Vc, q), rtol=2e-5, atol=5e-6)


# heads that go over the link in several chunks: odd kept counts (every chunk's indices start at an alignment of their own),
# a last chunk that is shorter, pageable values
@pytest.mark.parametrize("Hkv,g,w,L,budget,pageable", [(3, 2, 4, 44001, 333, False), (8, 1, 8, 16411, 1001, False), (5, 1, 4, 26301, 77, True)])
def test_host_call_in_chunks(Hkv, g, w, L, budget, pageable):
    wl = wl_of(Hkv, g, w, L, budget)
    K, V, Q, _ = W.make_layer(wl)
    s = shape_of(wl)
    pin = lambda a: torch.from_numpy(a.view(np.int16)).pin_memory()
    hKo = torch.zeros((Hkv, wl.nkeep, 128), dtype=torch.int16).pin_memory()
    hVo, hidx = torch.zeros_like(hKo).pin_memory(), torch.zeros((Hkv, wl.nkeep), dtype=torch.int32).pin_memory()
    buf = torch.empty(jq.host_call_bytes(s), dtype=torch.uint8, device="cuda")
    hK, hQ, hV = pin(K), pin(Q), torch.from_numpy(V.view(np.int16).copy()) if pageable else pin(V)
    # a second layer right behind, through the same device buffer into outputs of its own; and what the stream does next
    # finds the first call's results
    K2, V2, Q2, _ = W.make_layer(wl, layer=1)
    hK2, hQ2, hV2 = pin(K2), pin(Q2), torch.from_numpy(V2.view(np.int16).copy()) if pageable else pin(V2)
    hKo2, hVo2, hidx2 = torch.zeros_like(hKo).pin_memory(), torch.zeros_like(hKo).pin_memory(), torch.zeros_like(hidx).pin_memory()
    seen = [torch.empty(x.shape, dtype=x.dtype, device="cuda") for x in (hKo, hVo, hidx)]
    jq.evict_layer_host(hK, hV, hQ, s, hKo, hVo, hidx, buf)
    for d, h in zip(seen, (hKo, hVo, hidx)):
        d.copy_(h, non_blocking=True)
    jq.evict_layer_host(hK2, hV2, hQ2, s, hKo2, hVo2, hidx2, buf)
    torch.cuda.current_stream().synchronize()
    for (Ki, Vi, Qi), outs in (((K, V, Q), (hKo, hVo, hidx)), ((K, V, Q), [d.cpu() for d in seen]), ((K2, V2, Q2), (hKo2, hVo2, hidx2))):
        pooled = oracle.pool(oracle.score(Ki, Qi), wl.pool)
        gKo, gVo, gi = outs[0].numpy().view(np.uint16), outs[1].numpy().view(np.uint16), outs[2].numpy()
        assert_kept_sets_agree(gi, oracle.select(pooled, budget), pooled, wl.nkeep)
        for kv in range(Hkv):
            assert np.array_equal(gKo[kv], Ki[kv][gi[kv]]) and np.array_equal(gVo[kv], Vi[kv][gi[kv]])


def test_host_calls_of_one_thread_on_two_streams():
    """They share the stream that the library works on beside a caller's, and nothing else."""
    wl = wl_of(4, 2, 8, 33001, 500)
    s = shape_of(wl)
    pin = lambda a: torch.from_numpy(a.view(np.int16)).pin_memory()
    work = []
    for i in range(4):
        K, V, Q, _ = W.make_layer(wl, layer=i)
        outs = (torch.zeros((4, 500, 128), dtype=torch.int16).pin_memory(), torch.zeros((4, 500, 128), dtype=torch.int16).pin_memory(),
                torch.zeros((4, 500), dtype=torch.int32).pin_memory())
        work.append(((K, V, Q), (pin(K), pin(V), pin(Q)), outs))
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    bufs = [torch.empty(jq.host_call_bytes(s), dtype=torch.uint8, device="cuda") for _ in streams]
    torch.cuda.synchronize()
    for i, (_, (hK, hV, hQ), outs) in enumerate(work):
        jq.evict_layer_host(hK, hV, hQ, s, *outs, bufs[i & 1], stream=streams[i & 1])
    for st in streams:
        st.synchronize()
    for (K, V, Q), _, (gKo, gVo, gi) in work:
        pooled = oracle.pool(oracle.score(K, Q), wl.pool)
        gi = gi.numpy()
        assert_kept_sets_agree(gi, oracle.select(pooled, 500), pooled, 500)
        for kv in range(4):
            assert np.array_equal(gKo.numpy().view(np.uint16)[kv], K[kv][gi[kv]]) and np.array_equal(gVo.numpy().view(np.uint16)[kv], V[kv][gi[kv]])



def test_each_kernel_sees_what_the_one_before_it_wrote():
    """Re-eviction in place, decoding over the cache, selection, and a copy by the positions it kept, queued back to back
    round after round: every result is what the same calls give one at a time."""
    Hkv, g, w, n, new = 8, 4, 16, 512, 96
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    rnd = lambda *sh: torch.randn(sh, generator=gen, device="cuda", dtype=torch.bfloat16)
    s = jq.shape(Hkv, Hkv * g, n + new, w, n)
    s2 = jq.shape(Hkv, Hkv * g, n, w, 100)
    rounds = [(rnd(Hkv, new, 128), rnd(Hkv, new, 128), rnd(Hkv * g, w, 128), rnd(Hkv * g, 128), torch.rand((Hkv, n), generator=gen, device="cuda")) for _ in range(40)]
    K0, V0 = rnd(Hkv, n + new, 128), rnd(Hkv, n + new, 128)
    ws, ws2 = jq.new_append_workspace(s), jq.new_workspace(s2)
    wsd = torch.empty(jq.decode_workspace_bytes(Hkv, Hkv * g, n), dtype=torch.uint8, device="cuda")

    def run(step_by_step):
        Kc, Vc = K0.clone(), V0.clone()
        outs = [tuple(torch.zeros(sh, dtype=t, device="cuda") for sh, t in (((Hkv, n), torch.int32), ((Hkv * g, 128), torch.float32),
                ((Hkv, 100), torch.int32), ((Hkv, 100, 128), torch.bfloat16), ((Hkv, 100, 128), torch.bfloat16))) for _ in rounds]
        packed = torch.empty((2, Hkv, n, 128), dtype=torch.bfloat16, device="cuda")
        torch.cuda.synchronize()
        for (Kn, Vn, Q, q, sc), (idx, out, idx2, Ko, Vo) in zip(rounds, outs):
            for call in (lambda: jq.evict_append(Kc, Vc, n, Kn, Vn, Q, s, idx, ws), lambda: jq.compact_kv(Kc, Vc, first, s, packed[0], packed[1]),
                         lambda: jq.decode_attention(packed[0], packed[1], q, out, wsd), lambda: jq.select_topk(sc, s2, idx2, ws2),
                         lambda: jq.compact_kv(packed[0], packed[1], idx2, s2, Ko, Vo)):
                call()
                if step_by_step:
                    torch.cuda.synchronize()
        torch.cuda.synchronize()
        assert jq.last_device_status(ws) == jq.JQ_OK
        return [t for o in outs for t in o]

    first = torch.arange(n, dtype=torch.int32, device="cuda")[None].expand(Hkv, n).contiguous()
    want = run(True)
    for _ in range(3):
        for a, b in zip(run(False), want):
            assert torch.equal(a, b)


# one launch where it is the faster way: few heads or short prefixes; two where the rows are many or the heads leave most of
# the GPU's last round idle
@pytest.mark.parametrize("Hkv,g,w,L,launches", [(8, 4, 32, 8192, 1), (128, 4, 32, 8192, 1), (512, 4, 32, 1000, 1), (128, 4, 64, 8192, 2), (160, 4, 32, 3000, 2),
                                                (300, 4, 64, 5000, 2), (8, 4, 32, 12289, 2)])
def test_calls_over_many_heads_take_the_faster_way(Hkv, g, w, L, launches):
    """... and both give what the stages give one by one (here their scores stand in for the oracle's)."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(L)
    K, V = (torch.randn((Hkv, L, 128), generator=gen, device="cuda", dtype=torch.bfloat16) for _ in range(2))
    Q = torch.randn((Hkv * g, w, 128), generator=gen, device="cuda", dtype=torch.bfloat16)
    s = jq.shape(Hkv, Hkv * g, L, w, 300)
    Ko, Vo, idx = outputs(Hkv, 300, 300)
    ws = jq.new_workspace(s)
    n0 = jq.launch_count()
    jq.evict_layer(K, V, Q, s, Ko, Vo, idx, ws)
    assert jq.last_device_status(ws) == jq.JQ_OK and jq.launch_count() - n0 == launches
    scores, pooled, want = torch.empty((Hkv, L), device="cuda"), torch.empty((Hkv, L), device="cuda"), torch.empty_like(idx)
    jq.score(K, Q, s, scores, ws)
    jq.select_topk(scores, s, want, ws, pooled=pooled)
    assert_kept_sets_agree(idx.cpu().numpy(), want.cpu().numpy(), pooled.cpu().numpy().astype(np.float64), 300)
    at = idx.long()[:, :, None].expand(-1, -1, 128)
    assert torch.equal(Ko.view(torch.int16), K.gather(1, at).view(torch.int16)) and torch.equal(Vo.view(torch.int16), V.gather(1, at).view(torch.int16))


# CTAs of six tiles and more send their scores to the others as one copy each: lengths that end anywhere in a quad, with the window and
# without
@pytest.mark.parametrize("L", [11995, 11997, 11998, 11999])
@pytest.mark.parametrize("window", [False, True])
def test_scores_of_many_tiles_between_ctas(L, window):
    Hkv, g, w, budget = 8, 4, 32, 300
    wl = wl_of(Hkv, g, w, L, budget)
    K, V, Q, _ = W.make_layer(wl)
    s = shape_of(wl)
    Kw = W.make_window_keys(wl, Q)
    np_ = budget - w if window else budget
    Ko, Vo, idx = outputs(Hkv, budget, np_)
    ws = jq.new_workspace(s)
    n0 = jq.launch_count()
    if window:
        jq.evict_layer_window_kept(dev_bf16(K), dev_bf16(V), dev_bf16(Q), dev_bf16(Kw), dev_bf16(Kw), s, Ko, Vo, idx, ws)
    else:
        jq.evict_layer(dev_bf16(K), dev_bf16(V), dev_bf16(Q), s, Ko, Vo, idx, ws)
    assert jq.launch_count() - n0 == 1 and jq.last_device_status(ws) == jq.JQ_OK
    pooled = oracle.pool(oracle.score_windowed(K, Q, Kw) if window else oracle.score(K, Q), s.pool)
    gi = idx.cpu().numpy()
    assert_kept_sets_agree(gi, oracle.select(pooled, np_), pooled, np_)
    gK, gV = host_bits(Ko), host_bits(Vo)
    for kv in range(Hkv):
        assert np.array_equal(gK[kv][:np_], K[kv][gi[kv]]) and np.array_equal(gV[kv][:np_], V[kv][gi[kv]])


# the same in two parts: copies where the first part is a multiple of four, four scores at a time where it is not
@pytest.mark.parametrize("n_old,n_new", [(11000, 997), (11004, 1), (128, 11002), (11001, 996), (11003, 998)])
def test_scores_of_many_tiles_in_two_parts(n_old, n_new):
    Hkv, g, w, budget, L = 8, 4, 32, 100, n_old + n_new
    wl = wl_of(Hkv, g, w, L, budget)
    K, V, Q, _ = W.make_layer(wl)
    s = shape_of(wl)
    Kc, Vc = (torch.zeros((Hkv, L + 3, 128), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    dK, dV = dev_bf16(K), dev_bf16(V)
    Kc[:, :n_old] = dK[:, :n_old]; Vc[:, :n_old] = dV[:, :n_old]
    idx = torch.full((Hkv, budget), -1, dtype=torch.int32, device="cuda")
    ws = jq.new_append_workspace(s)
    n0 = jq.launch_count()
    jq.evict_append(Kc, Vc, n_old, dK[:, n_old:].contiguous(), dV[:, n_old:].contiguous(), dev_bf16(Q), s, idx, ws)
    assert jq.launch_count() - n0 == 1 and jq.last_device_status(ws) == jq.JQ_OK
    pooled = oracle.pool(oracle.score(K, Q), s.pool)
    gi = idx.cpu().numpy()
    assert_kept_sets_agree(gi, oracle.select(pooled, budget), pooled, budget)
    gK, gV = host_bits(Kc), host_bits(Vc)
    for kv in range(Hkv):
        assert np.array_equal(gK[kv][:budget], K[kv][gi[kv]]) and np.array_equal(gV[kv][:budget], V[kv][gi[kv]])
