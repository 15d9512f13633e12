"""The work a program has this library do, as cases to time and to compare.

A request to a vision-language model meets the library in three places: the
prefill (``tgvkv_prefill``, one layer at a time or every layer in one call),
the eviction at its end (``tgvkv_evict``, or ``tgvkv_evict_with_stats`` when the
prefill kept the rows' statistics; ``tgvkv_score`` where only the ranking is
wanted), and every decode step after it (``tgvkv_decode`` over the compacted
cache, or over the full one for a request that was not evicted).

A case is a dict of plain values:

call        "evict", "score", "prefill", "request" or "decode"
L, H_q, H_kv, d
            layers in the call, query heads, KV heads, head dimension
head, blocks, stamp, frame, tail
            the sequence: `head` text tokens, `blocks` times (`stamp` text and
            `frame` vision tokens), `tail` text tokens
window      "tail" (the last text segment queries) or "all" (every text token)
ratio       the retention budget r
basis, weights, sinks
            options of the eviction; sinks = keep the first 4 and the last token
cache       "compacted" or "full": the rows a decode step reads

Values follow the repository's synthetic workloads: N(0, 1) queries and values,
text keys N(0, I), vision keys around one centre per head (cosine about 0.8),
four outlier channels scaled by 8, rounded to bf16.  K / V caches are handed
over as the 16-bit patterns the library takes (int16), because compaction copies
them bit for bit.
"""
import math

import numpy as np
import torch

from paper_2606_03075_gb300 import api


def _case(call, L, H_q, H_kv, d, head, blocks, stamp, frame, tail, window="tail", ratio=0.05,
          basis="vision", weights="given", sinks=False, cache="compacted", name=None):
    case = dict(call=call, L=L, H_q=H_q, H_kv=H_kv, d=d, head=head, blocks=blocks, stamp=stamp,
                frame=frame, tail=tail, window=window, ratio=ratio, basis=basis, weights=weights,
                sinks=sinks, cache=cache)
    if name is not None:
        case["name"] = name
    return case


def listed():
    return [
        # the smallest call: one layer of eight heads, 112 tokens; launches and host time count
        _case("evict", 1, 8, 8, 64, 16, 1, 0, 64, 32, ratio=0.25, name="evict_tiny"),
        # one image in a 32-layer MHA model: many short heads
        _case("evict", 32, 32, 32, 128, 35, 1, 0, 576, 64, ratio=0.05, name="evict_llava15"),
        # five image tiles, 32-layer MHA, the most rows kept of the usual budgets
        _case("evict", 32, 32, 32, 128, 32, 5, 0, 576, 96, ratio=0.2, name="evict_next"),
        # grouped-query model with every option of the paper's main setting: derived text
        # weights, the all-token budget, sink tokens
        _case("evict", 28, 28, 4, 128, 32, 1, 0, 4096, 224, ratio=0.05, basis="all",
              weights="eq7", sinks=True, name="evict_qwen25_derived"),
        # long video: frames between timestamps, every text token a query row
        _case("evict", 28, 28, 4, 128, 32, 32, 8, 256, 224, window="all", ratio=0.05,
              name="evict_video"),
        # the ranking alone, on a small-head grouped-query model with ragged lengths
        _case("score", 24, 14, 2, 64, 17, 3, 5, 431, 77, window="all", name="score_ragged_d64"),
        # one layer's prefill as a model calls it, at a ragged length
        _case("prefill", 1, 28, 4, 128, 29, 1, 0, 3003, 211, name="prefill_layer_ragged"),
        # a short prompt through every layer in one call
        _case("prefill", 32, 32, 32, 128, 35, 1, 0, 576, 64, name="prefill_llava15"),
        # the largest: a long prompt through every layer of a grouped-query model
        _case("prefill", 28, 28, 4, 128, 32, 1, 0, 4096, 224, name="prefill_qwen25"),
        # a whole request: prefill with statistics, eviction with them, a decode step
        _case("request", 32, 32, 32, 128, 32, 5, 0, 576, 96, ratio=0.1, name="request_next"),
        # a decode step of every layer over the compacted cache
        _case("decode", 32, 32, 32, 128, 32, 5, 0, 576, 96, ratio=0.05, name="decode_next"),
        # a decode step of one layer over a long cache that was not evicted
        _case("decode", 1, 28, 4, 128, 32, 32, 8, 256, 224, cache="full",
              name="decode_layer_full"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """A case of the same ranges: 64 to 8704 tokens, 1 to 32 layers, MHA and grouped-query heads of
    64 and 128, one image or interleaved frames, every option."""
    top = max(_cost(c) for c in listed())
    while True:
        call = rng.choice(["evict", "evict", "score", "prefill", "prefill", "request", "decode",
                           "decode"])
        H_kv = rng.choice([2, 4, 8, 8, 32])
        G = 1 if H_kv == 32 else rng.choice([1, 2, 4, 7])
        blocks = rng.choice([1, 1, 1, 2, 5, 16, 32])
        vision = _log_int(rng, 32, 8192)
        case = _case(call, _log_int(rng, 1, 32), H_kv * G, H_kv, rng.choice([64, 128, 128]),
                     head=rng.randint(1, 64), blocks=blocks,
                     stamp=0 if blocks == 1 else rng.randint(0, 8),
                     frame=max(8, vision // blocks), tail=_log_int(rng, 16, 256),
                     window=rng.choice(["tail", "tail", "all"]),
                     ratio=rng.choice([0.05, 0.05, 0.1, 0.2, round(rng.uniform(0.02, 0.6), 3)]),
                     basis=rng.choice(["vision", "vision", "all"]),
                     weights=rng.choice(["given", "given", "eq7"]),
                     sinks=rng.choice([False, False, True]),
                     cache=rng.choice(["compacted", "compacted", "full"]))
        if call in ("score", "prefill"):     # options of the later steps
            case.update(basis="vision", weights="given", sinks=False)
        if call == "decode":
            case.update(window="tail", weights="given", sinks=False)
        else:
            case.update(cache="compacted")
        if _cost(case) <= top:
            return case


# ---- shapes ------------------------------------------------------------------
def _modality(case):
    parts = [np.zeros(case["head"], np.uint8)]
    for _ in range(case["blocks"]):
        parts += [np.zeros(case["stamp"], np.uint8), np.ones(case["frame"], np.uint8)]
    return np.concatenate(parts + [np.zeros(case["tail"], np.uint8)])


def _layout(case):
    modality = _modality(case)
    N = modality.size
    if case["window"] == "all":
        text_pos = np.flatnonzero(modality == 0)
    else:
        text_pos = np.arange(N - case["tail"], N)
    return modality, text_pos.astype(np.int32), N, int(modality.sum())


def _desc(case):
    _, text_pos, N, N_v = _layout(case)
    return api.make_desc(case["L"], case["H_q"], case["H_kv"], case["d"], N, N_v, text_pos.size,
                         basis=case["basis"], weights=case["weights"],
                         keep_first=4 if case["sinks"] else 0, keep_last=1 if case["sinks"] else 0)


def _rows(case):
    """Rows a decode step reads: retained rows, or the full cache."""
    _, _, N, N_v = _layout(case)
    L, H_kv, r = case["L"], case["H_kv"], case["ratio"]
    if case["cache"] == "full":
        return L * H_kv * N
    if case["basis"] == "all":
        return H_kv * int(math.floor(r * N * L + 0.5))
    return H_kv * (L * (N - N_v) + int(math.floor(r * N_v * L + 0.5)))


def work(case):
    """Each input read once, each output written once; the attention logits counted once."""
    _, text_pos, N, N_v = _layout(case)
    L, H_q, H_kv, d, n_win = case["L"], case["H_q"], case["H_kv"], case["d"], text_pos.size
    kv = 2 * L * H_kv * N * d
    q_win = 2 * L * H_q * n_win * d
    pairs = L * H_q * int((text_pos.astype(np.int64) + 1).sum())
    kept = _rows(dict(case, cache="compacted"))
    total = {"bytes": 0, "flops": 0}

    def add(nbytes, flops):
        total["bytes"] += nbytes
        total["flops"] += flops

    if case["call"] in ("prefill", "request"):
        add(2 * 2 * L * H_q * N * d + 2 * kv + q_win + 12 * L * H_q * n_win,
            4 * d * L * H_q * (N * (N + 1) // 2))
    if case["call"] in ("evict", "score", "request"):
        add(kv + q_win + 4 * L * H_kv * N_v, 2 * d * pairs)
    if case["call"] in ("evict", "request"):
        add(2 * 2 * 2 * kept * d + 4 * kept + 8 * L * H_kv, 0)
    if case["call"] in ("decode", "request"):
        rows = _rows(case)
        add(2 * 2 * rows * d + 6 * L * H_q * d, 4 * d * rows * (H_q // H_kv))
    return total


def _cost(case):
    """A rough time of one pass, to keep drawn cases below the largest listed one."""
    w = work(case)
    return w["bytes"] / 5e12 + w["flops"] / (8e14 if case["call"] in ("prefill", "request") else 3e14)


# ---- inputs ------------------------------------------------------------------
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _bits(x):
    return x.to(torch.bfloat16).view(torch.int16)


def _normal(gen, *shape):
    """bf16 N(0, 1) patterns, drawn a layer at a time."""
    out = torch.empty(shape, dtype=torch.int16, device="cuda")
    for l in range(shape[0]):
        out[l] = _bits(torch.randn(shape[1:], device="cuda", generator=gen))
    return out


def _keys(case, gen, vision, N):
    L, H_kv, d = case["L"], case["H_kv"], case["d"]
    out = torch.empty((L, H_kv, N, d), dtype=torch.int16, device="cuda")
    for l in range(L):
        x = torch.randn((H_kv, N, d), device="cuda", generator=gen)
        centre = torch.randn((H_kv, 1, d), device="cuda", generator=gen)
        x = torch.where(vision[None, :, None], math.sqrt(0.8) * centre + math.sqrt(0.2) * x, x)
        order = torch.rand((H_kv, d), device="cuda", generator=gen).argsort(dim=1)
        scale = torch.where(order < 4, 8.0, 1.0)
        out[l] = _bits(x * scale[:, None, :])
    return out


def _inputs(case, seed):
    """Tensors of one case, from the seed alone."""
    modality, text_pos, N, _ = _layout(case)
    L, H_q, H_kv, d = case["L"], case["H_q"], case["H_kv"], case["d"]
    gen = _generator(seed)
    mod = torch.from_numpy(modality).cuda()
    t = dict(modality=mod, text_pos=torch.from_numpy(text_pos).cuda())
    if case["call"] == "decode":
        t["q_dec"] = _normal(gen, L, H_q, d)
        # retained sets: every layer its own share of the budget, as the statistic splits it
        n_sets, rows = L * H_kv, _rows(case)
        if case["cache"] == "full":
            counts = np.full(n_sets, N, np.int64)
        else:
            share = np.random.default_rng(seed).uniform(0.5, 1.5, L)
            floor_rows = int((modality == 0).sum()) if case["basis"] == "vision" else 0
            free = rows // H_kv - L * floor_rows
            part = np.floor(free * share / share.sum()).astype(np.int64)
            part[: free - int(part.sum())] += 1
            counts = np.repeat(part + floor_rows, H_kv)
        t["offsets"] = torch.from_numpy(np.concatenate([[0], np.cumsum(counts)])).cuda()
        vision = torch.rand(rows, device="cuda", generator=gen) < 0.5
        one = dict(case, L=1, H_kv=1)
        t["k_rows"] = _keys(one, gen, vision, rows).view(rows, d)
        t["v_rows"] = _normal(gen, 1, rows, d).view(rows, d)
        return t
    t["k"] = _keys(case, gen, mod != 0, N)
    if case["call"] != "score":
        t["v"] = _normal(gen, L, H_kv, N, d)
    w = -torch.log(torch.rand((L, text_pos.size), device="cuda", generator=gen).clamp_min(1e-7))
    t["w"] = (w / w.sum(dim=1, keepdim=True)).contiguous()      # Dirichlet(1) text weights
    if case["call"] in ("prefill", "request"):
        t["q"] = _normal(gen, L, H_q, N, d)
    else:
        t["q_text"] = _normal(gen, L, H_q, text_pos.size, d)
    if case["call"] == "request":
        t["q_dec"] = _normal(gen, L, H_q, d)
    return t


def prepare(case, seed):
    """Inputs, the workspace and the output buffers a program keeps."""
    t = _inputs(case, seed)
    desc = _desc(case)
    _, text_pos, N, N_v = _layout(case)
    L, H_q, H_kv, d, n_win = case["L"], case["H_q"], case["H_kv"], case["d"], text_pos.size
    s = dict(t, call=case["call"], ratio=case["ratio"], desc=desc, ws=api.new_workspace(desc))

    def buf(dtype, *shape):
        return torch.zeros(shape, dtype=dtype, device="cuda")

    if case["call"] == "score":
        s["scores"] = buf(torch.float32, L, H_kv, N_v)
        s["tvb_stat"] = buf(torch.float32, L)
    if case["call"] in ("evict", "request"):
        out = api.alloc_outputs(desc, case["ratio"])
        out.k_out = torch.zeros_like(out.k_out).view(torch.int16)
        out.v_out = torch.zeros_like(out.v_out).view(torch.int16)
        out.idx.zero_()
        s["out"] = out
    if case["call"] in ("prefill", "request"):
        s["o"] = buf(torch.bfloat16, L, H_q, N, d)
        s["q_text"] = buf(torch.int16, L, H_q, n_win, d)
        s["row_stats"] = buf(torch.float32, L, H_q, n_win, 3)
    if case["call"] in ("decode", "request"):
        s["o_dec"] = buf(torch.float32, L, H_q, d)
    return s


def run(s):
    desc, ws = s["desc"], s["ws"]
    got = {}
    if s["call"] == "score":
        api.tgvkv_score(desc, s["q_text"], s["k"], s["modality"], s["text_pos"], s["w"],
                        s["scores"], s["tvb_stat"], ws)
        return {"scores": s["scores"], "tvb_stat": s["tvb_stat"]}
    if s["call"] == "decode":
        api.tgvkv_decode(desc, s["q_dec"], s["k_rows"], s["v_rows"], s["offsets"], s["o_dec"], ws)
        return {"o_dec": s["o_dec"]}
    if s["call"] in ("prefill", "request"):
        api.tgvkv_prefill(desc, s["q"], s["k"], s["v"], s["modality"], s["text_pos"], s["o"],
                          s["q_text"], s["row_stats"], ws)
        got.update(o=s["o"], q_text=s["q_text"], row_stats=s["row_stats"])
    if s["call"] == "prefill":
        return got
    out = s["out"]
    if s["call"] == "request":
        api.tgvkv_evict_with_stats(desc, s["q_text"], s["k"], s["v"], s["modality"], s["text_pos"],
                                   s["w"], s["ratio"], s["row_stats"], out, ws)
        api.tgvkv_decode(desc, s["q_dec"], out.k_out, out.v_out, out.offsets, s["o_dec"], ws)
        got["o_dec"] = s["o_dec"]
    else:
        api.tgvkv_evict(desc, s["q_text"], s["k"], s["v"], s["modality"], s["text_pos"], s["w"],
                        s["ratio"], out, ws)
    got.update(scores=out.scores, tvb_stat=out.tvb_stat, budgets=out.budgets, offsets=out.offsets,
               idx=out.idx, k_out=out.k_out, v_out=out.v_out)
    return got


def tolerance(case):
    """About four times the distance from 64 bits that was measured: scores, statistics and decode
    outputs (7e-7, 1e-7, 1.1e-6) are fp32 sums of exact bf16 products under a fast exponential; the
    prefill's output (1.9e-3) is bf16, with bf16 weights in its value product.  Kept rows are
    copied bit for bit; two keys whose scores agree to the last bits may change places in a set,
    which moves the entries between them: the share `differ` is for those."""
    if case["call"] == "decode":
        return {"rel": 5e-6}
    if case["call"] == "prefill":
        return {"rel": 8e-3}
    if case["call"] == "request":
        return {"rel": 8e-3, "differ": 0.01}
    return {"rel": 5e-6, "differ": 0.01}


# ---- the same in 64 bits -----------------------------------------------------
def _f64(bits):
    return bits.view(torch.bfloat16).double()


def _exact_evict(case, t, q_text):
    """Scores and the layers' statistic: attention rows of the text queries over all visible keys,
    their vision columns, text-weighted sums, the mean over each group's heads."""
    L, H_q, H_kv, d = case["L"], case["H_q"], case["H_kv"], case["d"]
    G, N = H_q // H_kv, t["modality"].numel()
    pos, vision = t["text_pos"].long(), t["modality"] != 0
    hidden = torch.arange(N, device="cuda")[None, :] > pos[:, None]
    scores, stat = [], []
    for l in range(L):
        k, q = _f64(t["k"][l]), _f64(q_text[l])
        a = torch.matmul(q.view(H_kv, G, -1, d), k[:, None].transpose(-1, -2)) / math.sqrt(d)
        a = torch.softmax(a.masked_fill_(hidden, -math.inf), dim=-1)
        w = t["w"][l].double()
        if case["weights"] == "eq7":
            tt = a[..., pos].mean(dim=(0, 1))                      # [rows, columns] text to text
            w = tt.tril().sum(dim=0) / torch.arange(pos.numel(), 0, -1, device="cuda")
            w = w / w.sum()
        av = a[..., vision]
        scores.append(torch.einsum("gqiv,i->gv", av, w) / G)
        stat.append(av.sum())
    return torch.stack(scores), torch.stack(stat)


def _exact_decode(case, q_dec, k_rows, v_rows, offsets):
    L, H_q, H_kv, d = case["L"], case["H_q"], case["H_kv"], case["d"]
    G, off = H_q // H_kv, offsets.tolist()
    out = torch.zeros((L, H_q, d), dtype=torch.float64, device="cuda")
    for s in range(L * H_kv):
        l, g = divmod(s, H_kv)
        q = _f64(q_dec[l, g * G:(g + 1) * G])
        k, v = _f64(k_rows[off[s]:off[s + 1]]), _f64(v_rows[off[s]:off[s + 1]])
        if k.shape[0]:
            out[l, g * G:(g + 1) * G] = torch.softmax(q @ k.T / math.sqrt(d), dim=-1) @ v
    return out


def _exact_prefill(case, t):
    L, H_q, H_kv, d = case["L"], case["H_q"], case["H_kv"], case["d"]
    G, N = H_q // H_kv, t["modality"].numel()
    out = torch.empty((L, H_q, N, d), dtype=torch.float32, device="cuda")
    key = torch.arange(N, device="cuda")
    for l in range(L):
        for g in range(H_kv):
            k, v = _f64(t["k"][l, g]), _f64(t["v"][l, g])
            for i in range(0, N, 1024):
                q = _f64(t["q"][l, g * G:(g + 1) * G, i:i + 1024])
                n = min(N, i + 1024)
                a = torch.matmul(q, k[:n].T) / math.sqrt(d)
                a.masked_fill_(key[None, :n] > key[i:n, None], -math.inf)
                out[l, g * G:(g + 1) * G, i:i + 1024] = torch.softmax(a, dim=-1) @ v[:n]
    return out


def exact(case, seed):
    """What run() returns, in 64 bits; None for copies, whole values and the row statistics,
    whose reference maximum is the kernel's to choose."""
    w = work(case)
    if w["flops"] > 8e12:
        return None
    t = _inputs(case, seed)
    if case["call"] == "decode":
        return {"o_dec": _exact_decode(case, t["q_dec"], t["k_rows"], t["v_rows"], t["offsets"])}
    got = {}
    if case["call"] in ("prefill", "request"):
        q_text = t["q"][:, :, t["text_pos"].long()]
        got.update(o=_exact_prefill(case, t), q_text=None, row_stats=None)
        if case["call"] == "prefill":
            return got
        got["o_dec"] = None       # depends on which of two tied rows is kept
    else:
        q_text = t["q_text"]
    got["scores"], got["tvb_stat"] = _exact_evict(case, t, q_text)
    if case["call"] != "score":
        got.update(budgets=None, offsets=None, idx=None, k_out=None, v_out=None)
    return got
