"""The work this library is used for, as cases that can be timed.

A serving program prefills a prompt, appends the soft tokens, and evicts each layer's KV cache down to a budget; it
then decodes over the pruned cache and, when that has grown, evicts it again.  The cases call the public entry points
the way such a program does: with tensors, outputs and an initialised workspace of its own that it keeps from call to
call.  `listed` holds the sizes of the library's own workloads (caches of 2K to 128K keys, 32 or 64 soft tokens,
budgets of 256 to 4096, one layer or the 32 layers of a model, a ragged batch), `draw` the ranges around them.
"""
import torch

import paper_2509_10798_b200 as jq

D = 128


def listed():
    return [
        # the smallest call: a short prompt on a small model (2 KV heads); launches and latency are all there is
        dict(name="layer_2k", kind="layer", Hkv=2, group=4, L=2048, w=16, budget=256, pool=7),
        # one layer right after its prefill, the ordinary prompt
        dict(name="layer_8k", kind="layer", Hkv=8, group=4, L=8192, w=32, budget=1024, pool=7),
        # one layer of the longest prompt, 256 query rows per KV head
        dict(name="layer_128k", kind="layer", Hkv=8, group=4, L=131072, w=64, budget=4096, pool=7),
        # the whole cache of a 32-layer model after the prefill, every layer in a buffer of its own
        dict(name="layers_32k", kind="layers", layers=32, Hkv=8, group=4, L=32768, w=32, budget=512, pool=7),
        # the same with the longest prompt: the largest call
        dict(name="layers_128k", kind="layers", layers=32, Hkv=8, group=4, L=131072, w=64, budget=1024, pool=7),
        # a batch of four prompts of different lengths, all layers in one call
        dict(name="ragged_batch", kind="ragged", seqs=4, layers=32, Hkv=8, group=4, L=32768, w=32, budget=1024, pool=7),
        # the last-window form with the window itself retained, a prompt whose length is no multiple of anything
        dict(name="window_kept", kind="window", Hkv=8, group=4, L=11999, w=32, budget=1024, pool=7),
        # the three stages as calls of their own, with scores and pooled scores handed back (analysis, other policies)
        dict(name="stages", kind="stages", Hkv=8, group=4, L=30011, w=32, budget=2048, pool=7),
        # decoding: the cache has grown by 256 pairs behind the 1024 retained ones and is evicted again, in place
        dict(name="reevict", kind="reevict", Hkv=8, group=4, n_old=1024, n_new=256, w=32, pool=7),
        # decoding: attention of one new position over one layer's pruned cache
        dict(name="decode_step", kind="decode", Hkv=8, group=4, n=1024),
        # the same for a batch of 16 sequences of equal budget, stacked along the KV-head axis
        dict(name="decode_batch", kind="decode", Hkv=128, group=4, n=2048),
        # a layer whose cache was offloaded: page-locked host buffers in and out
        dict(name="host_layer", kind="host", Hkv=8, group=4, L=32768, w=32, budget=1024, pool=7),
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(("layer", "layer", "layer", "layers", "layers", "ragged", "window", "stages", "reevict", "decode",
                       "decode", "host"))
    group = rng.choice((1, 2, 4, 4, 4, 7, 8))
    c = dict(kind=kind, group=group)
    if kind == "decode":
        c["Hkv"] = _log_int(rng, 2, 160)
        c["n"] = _log_int(rng, 128, 4096)
        return c
    c["w"] = min(rng.choice((8, 16, 24, 32, 32, 32, 48, 64)), 256 // group)
    c["pool"] = rng.choice((1, 3, 5, 7, 7, 7, 9, 13))
    c["Hkv"] = rng.choice((2, 4, 8, 8, 8))
    if kind == "reevict":
        c["n_old"] = _log_int(rng, 256, 4096)
        c["n_new"] = _log_int(rng, 32, 1024)
        return c
    # prefixes from a short prompt to the longest; the calls over many layers keep their keys below 4 GiB
    most = {"layers": 65536, "ragged": 40000, "host": 65536}.get(kind, 131072)
    c["L"] = _log_int(rng, 1024, most)
    c["budget"] = min(_log_int(rng, 64, 4096), max(64, c["L"] // 2))
    if kind == "window":
        c["budget"] += c["w"]
    if kind == "layers":
        c["layers"] = min(rng.choice((8, 16, 28, 32, 48)), (1 << 24) // (c["Hkv"] * c["L"]))
    if kind == "ragged":
        c["seqs"] = rng.randint(2, 6)
        c["layers"] = min(rng.choice((8, 16, 32)), (1 << 24) // (c["Hkv"] * c["L"] * c["seqs"]) or 1)
    return c


# ------------------------------------------------------------------ inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _normal(g, *shape):
    return torch.empty(shape, dtype=torch.bfloat16, device="cuda").normal_(generator=g)


def _keys(g, Hkv, L, topics):
    """Post-RoPE keys: noise with a few outlier channels per head, or (topics) segments that share a direction."""
    K = _normal(g, Hkv, L, D)
    if topics:
        K *= 0.5
        centre = _normal(g, Hkv, 16, D)
        label = torch.randint(0, 16, (Hkv, L // 512 + 1), generator=g, device="cuda")
        seg = torch.arange(L, device="cuda") // 512
        for h in range(Hkv):
            K[h] += centre[h, label[h]][seg]
    else:
        for h in range(Hkv):
            K[h, :, torch.randperm(D, generator=g, device="cuda")[:4]] *= 8.0
    return K


def _queries(g, K, group, w):
    """Soft-token queries: noise plus a pull towards 80 keys of their KV head, 16 of them among the last 256."""
    Hkv, L = K.shape[0], K.shape[1]
    at = torch.cat([torch.randint(0, L, (Hkv, 64), generator=g, device="cuda"),
                    torch.randint(max(0, L - 256), L, (Hkv, 16), generator=g, device="cuda")], 1)
    row = torch.arange(group * w, device="cuda") % 80
    near = torch.stack([K[h, at[h, row]] for h in range(Hkv)]).float()
    Q = 0.7 * torch.empty(near.shape, device="cuda").normal_(generator=g) + 0.3 * near
    return Q.to(torch.bfloat16).reshape(Hkv * group, w, D).contiguous()


def _lengths(case):
    """Prefix lengths of a ragged batch: from an eighth of the longest up, odd ones among them."""
    n = case["seqs"]
    return [case["L"] - (case["L"] * 7 // 8 - i) * i // (n - 1) for i in range(n)]


def _outputs(rows):
    return (torch.empty((*rows, D), dtype=torch.bfloat16, device="cuda"), torch.empty((*rows, D), dtype=torch.bfloat16, device="cuda"),
            torch.empty(rows, dtype=torch.int32, device="cuda"))


def _kept(idx, Kout, Vout):
    # the compacted rows are copies, bit for bit: they are compared as 16-bit patterns
    return {"idx": idx, "K": Kout.view(torch.int16), "V": Vout.view(torch.int16)}


def prepare(case, seed):
    g = _gen(seed)
    kind, Hkv, group = case["kind"], case["Hkv"], case["group"]
    Hq = Hkv * group
    st = dict(kind=kind)
    if kind == "decode":
        n = case["n"]
        st["Kc"], st["Vc"], st["q"] = _normal(g, Hkv, n, D), _normal(g, Hkv, n, D), _normal(g, Hq, D)
        st["out"] = torch.empty((Hq, D), dtype=torch.float32, device="cuda")
        st["ws"] = torch.empty(jq.decode_workspace_bytes(Hkv, Hq, n), dtype=torch.uint8, device="cuda")
        return st
    w, pool = case["w"], case["pool"]
    if kind == "reevict":
        n_old, n_new = case["n_old"], case["n_new"]
        L = n_old + n_new
        st["s"] = s = jq.shape(Hkv, Hq, L, w, n_old, pool)
        st["Kc"], st["Vc"] = _keys(g, Hkv, L, False), _normal(g, Hkv, L, D)
        # the pairs decoded between two evictions and the queries of the last positions: several rounds of them, since
        # the cache goes on from call to call
        st["new"] = []
        for _ in range(16):
            Kn = _keys(g, Hkv, n_new, False)
            st["new"].append((Kn, _normal(g, Hkv, n_new, D), _queries(g, torch.cat([st["Kc"][:, :n_old], Kn], 1), group, w)))
        st["turn"], st["n_old"] = 0, n_old
        st["idx"] = torch.empty((Hkv, n_old), dtype=torch.int32, device="cuda")
        st["ws"] = jq.new_append_workspace(s)
        return st
    L, budget = case["L"], case["budget"]
    if kind in ("layers", "ragged"):
        lengths = [L] * case["layers"] if kind == "layers" else [n for n in _lengths(case) for _ in range(case["layers"])]
        st["K"] = [_keys(g, Hkv, n, kind == "ragged") for n in lengths]
        st["V"] = [_normal(g, Hkv, n, D) for n in lengths]
        st["Q"] = [_queries(g, K, group, w) for K in st["K"]]
        st["s"] = s = jq.shape(Hkv, Hq, L, w, budget, pool)
        if kind == "layers":
            st["out"] = _outputs((len(lengths) * Hkv, jq.num_kept(s)))
            st["ws"] = jq.new_layers_workspace(s, len(lengths))
        else:
            st["L"], st["budget"] = lengths, [budget] * len(lengths)
            st["out"] = _outputs((jq.ragged_output_rows(s, len(lengths), st["L"], st["budget"]),))
            st["ws"] = jq.new_ragged_workspace(s, len(lengths), st["L"])
        return st
    st["s"] = s = jq.shape(Hkv, Hq, L, w, budget, pool)
    nkeep = jq.num_kept(s)
    K = _keys(g, Hkv, L, False)
    Q = _queries(g, K, group, w)
    V = _normal(g, Hkv, L, D)
    if kind == "host":
        st["K"], st["V"], st["Q"] = K.cpu().pin_memory(), V.cpu().pin_memory(), Q.cpu().pin_memory()
        st["out"] = tuple(torch.empty(sh, dtype=t, pin_memory=True) for sh, t in (
            ((Hkv, nkeep, D), torch.bfloat16), ((Hkv, nkeep, D), torch.bfloat16), ((Hkv, nkeep), torch.int32)))
        st["ws"] = torch.empty(jq.host_call_bytes(s), dtype=torch.uint8, device="cuda")
        return st
    st["K"], st["V"], st["Q"] = K, V, Q
    st["out"] = _outputs((Hkv, nkeep))
    st["ws"] = jq.new_workspace(s)
    if kind == "window":
        # keys of the query positions themselves; they resemble the positions' queries a little
        mean = Q.view(Hkv, group, w, D).float().mean(1)
        st["Kwin"] = (torch.empty(mean.shape, device="cuda").normal_(generator=g) + 0.3 * mean).to(torch.bfloat16)
        st["Vwin"] = _normal(g, Hkv, w, D)
        np_ = min(budget - w, L)
        st["out"] = (*_outputs((Hkv, np_ + w))[:2], torch.empty((Hkv, np_), dtype=torch.int32, device="cuda"))
    if kind == "stages":
        st["scores"] = torch.empty((Hkv, L), dtype=torch.float32, device="cuda")
        st["pooled"] = torch.empty((Hkv, L), dtype=torch.float32, device="cuda")
    return st


# ------------------------------------------------------------------ one pass

def run(st):
    kind = st["kind"]
    if kind == "decode":
        jq.decode_attention(st["Kc"], st["Vc"], st["q"], st["out"], st["ws"])
        return st["out"]
    s = st["s"]
    if kind == "reevict":
        Kn, Vn, Q = st["new"][st["turn"] % len(st["new"])]
        st["turn"] += 1
        n = st["n_old"]
        jq.evict_append(st["Kc"], st["Vc"], n, Kn, Vn, Q, s, st["idx"], st["ws"])
        # (the rows behind the kept ones are free space)
        return _kept(st["idx"], st["Kc"][:, :n], st["Vc"][:, :n])
    Kout, Vout, idx = st["out"]
    if kind == "layer":
        jq.evict_layer(st["K"], st["V"], st["Q"], s, Kout, Vout, idx, st["ws"])
    elif kind == "layers":
        jq.evict_layers(st["K"], st["V"], st["Q"], s, Kout, Vout, idx, st["ws"])
    elif kind == "ragged":
        jq.evict_ragged(st["K"], st["V"], st["Q"], s, st["L"], st["budget"], Kout, Vout, idx, st["ws"])
    elif kind == "window":
        jq.evict_layer_window_kept(st["K"], st["V"], st["Q"], st["Kwin"], st["Vwin"], s, Kout, Vout, idx, st["ws"])
    elif kind == "host":
        jq.evict_layer_host(st["K"], st["V"], st["Q"], s, Kout, Vout, idx, st["ws"])
    elif kind == "stages":
        jq.score(st["K"], st["Q"], s, st["scores"], st["ws"])
        jq.select_topk(st["scores"], s, idx, st["ws"], pooled=st["pooled"])
        jq.compact_kv(st["K"], st["V"], idx, s, Kout, Vout)
        return {"scores": st["scores"], "pooled": st["pooled"], **_kept(idx, Kout, Vout)}
    return _kept(idx, Kout, Vout)


# ------------------------------------------------------------------ what a pass cannot do without, and how exact it is

def work(case):
    kind, Hkv, group = case["kind"], case["Hkv"], case["group"]
    row = 2 * D
    if kind == "decode":
        n = case["n"]
        return {"bytes": 2 * Hkv * n * row + Hkv * group * D * 6, "flops": 4 * Hkv * group * n * D}
    R = group * case["w"]
    if kind == "reevict":
        keep, L = case["n_old"], case["n_old"] + case["n_new"]
        # the old and the new keys, the new values, the queries; the kept rows stay in place as far as they can
        return {"bytes": Hkv * (L * row + case["n_new"] * row + R * row + 4 * keep), "flops": 2 * Hkv * R * L * D}
    if kind == "ragged":
        lengths = [n for n in _lengths(case) for _ in range(case["layers"])]
    else:
        lengths = [case["L"]] * case.get("layers", 1)
    nbytes = flops = 0
    for L in lengths:
        keep = min(case["budget"], L)
        # every key once, the queries, the kept rows of V; out: the kept rows of K and V and their indices
        nbytes += Hkv * (L * row + R * row + keep * row + 2 * keep * row + 4 * keep)
        flops += 2 * Hkv * R * L * D
        if kind == "stages":
            nbytes += 8 * Hkv * L
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    if case["kind"] == "decode":
        return {"rel": 1e-5}
    # scores are 32-bit sums of 32-bit exponentials; two such sums may order two keys differently when they are equal to
    # seven digits, and the kept rows between the two then move by one place
    if case["kind"] == "stages":
        return {"rel": 1e-5, "differ": 0.01}
    return {"differ": 0.01}
