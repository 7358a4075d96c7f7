"""The work that users of this library have it do, as measurable cases: one prune call at a pruning layer (the global
stage with many scored rows, the fine stage with the last token's), chains of fine stages, the positional global rule,
the attention-rollout analysis, and a prune call on host buffers.

Sizes are those of the package's workloads (``workloads.py``), of the tests and of the benchmark, or generic ones of the
same kind; ``draw`` spreads over the same ranges.  Inputs are made on the GPU from the seed.  Attention over audio-visual
prompts is heavy-tailed: a token that one head attends to is attended to by the others as well, and token importance
spans orders of magnitude.  So keys carry a per-token component along a direction that all query rows share, strong
enough to move a token's logits by a normal amount of standard deviation 1.5 in every head, and a few early anchor tokens
carry a large one.
"""
import math
import random

import torch

from paper_2601_13143_b200 import fastav as F
from paper_2601_13143_b200.workloads import MOD_AUDIO, MOD_TEXT, MOD_VIDEO, keep_count, positional_keep_mask

# (query heads, KV heads, head_dim, hidden): the three decoder shapes of the workloads, then two generic ones
TINY = (8, 2, 64, 512)
QWEN2 = (28, 4, 128, 3584)
MISTRAL = (32, 8, 128, 4096)
SHAPES = (TINY, QWEN2, MISTRAL, (16, 16, 64, 1024), (32, 4, 128, 2048))

LOGIT_SPREAD = 1.5  # standard deviation of a token's shared logit shift
SHARED = 0.5        # share of a query that is common to all rows and heads of a KV group


def _case(name, kind, shape, **more):
    hq, hkv, dim, hidden = shape
    c = {"kind": kind, "q_heads": hq, "kv_heads": hkv, "dim": dim, "hidden": hidden, **more}
    return {"name": name, **c} if name else c


def listed():
    return [
        # the smallest call: a short clip on a small decoder, a few scored rows, half the tokens kept (latency)
        _case("tiny_512", "prune", TINY, batch=1, lo=512, hi=512, layout=0, rows=4, keep_lo=0.5, keep_hi=0.5, lse=False),
        # the global stage of one 2k-token prompt at the middle layer, all trailing text rows scored
        _case("global_2048", "prune", QWEN2, batch=1, lo=2048, hi=2048, layout=0, rows=64, keep_lo=0.5, keep_hi=0.5, lse=False),
        # three fine stages on a thousand survivors, last-token query
        _case("fine_chain_3x1024", "chain", QWEN2, tokens=1024, stages=3, keep=0.8),
        # the paper's schedule after its global stage: 744 survivors, 20 % dropped at each of the 13 later layers
        _case("fine_chain_13x744", "chain", QWEN2, tokens=744, stages=13, keep=0.8),
        # the largest scores: four long audio-video clips, 128 scored rows each, 40 % kept
        _case("long_global_4x16384", "prune", MISTRAL, batch=4, lo=16384, hi=16384, layout=0, rows=128, keep_lo=0.4, keep_hi=0.4, lse=False),
        # the fine stage on the survivors of those clips
        _case("long_fine_4x6554", "prune", MISTRAL, batch=4, lo=6554, hi=6554, layout=0, rows=1, keep_lo=0.7, keep_hi=0.7, lse=False),
        # a serving batch of ragged prompts, each with its own keep ratio
        _case("ragged_global_32", "prune", QWEN2, batch=32, lo=1024, hi=8192, layout=4, rows=32, keep_lo=0.3, keep_hi=0.7, lse=False),
        # ... and its fine stage on ragged survivors
        _case("ragged_fine_32", "prune", QWEN2, batch=32, lo=512, hi=4096, layout=5, rows=1, keep_lo=0.8, keep_hi=0.8, lse=False),
        # the global stage beside an attention kernel that hands over its log-sum-exp: odd lengths, one sweep over K
        _case("lse_global_3x8k", "prune", QWEN2, batch=3, lo=8001, hi=9001, layout=2, rows=64, keep_lo=0.4, keep_hi=0.6, lse=True),
        # the paper's deployed global rule: fixed positions, no scores, a batch of its 2,230-token prompts
        _case("positional_8x2230", "positional", QWEN2, batch=8, lo=2230, hi=2230, layout=0),
        # the analysis that fixes that rule: attention rollout up to the middle layer of one prompt
        _case("rollout_2230x14", "rollout", QWEN2, tokens=2230, layers=14),
        # activations kept in host memory: upload, prune, download
        _case("host_2048", "host", QWEN2, batch=1, lo=2048, hi=2048, layout=0, rows=64, keep_lo=0.5, keep_hi=0.5, lse=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("global", "global", "global", "fine", "fine", "chain", "chain", "positional", "rollout", "host"))
    shape = rng.choice(SHAPES)
    layout = rng.randrange(1 << 20)
    if kind == "chain":
        return _case("", "chain", shape, tokens=_log_int(rng, 100, 2000), stages=rng.randint(3, 13), keep=round(rng.uniform(0.7, 0.9), 3))
    if kind == "rollout":
        return _case("", "rollout", shape, tokens=_log_int(rng, 200, 2230), layers=rng.randint(4, 14))
    if kind == "host":
        n = _log_int(rng, 300, 2048)
        return _case("", "host", shape, batch=1, lo=n, hi=n, layout=layout, rows=_log_int(rng, 1, 64), keep_lo=0.3, keep_hi=0.7, lse=False)
    total = _log_int(rng, 300, 60000)  # tokens of the batch
    batch = min(_log_int(rng, 1, 32), max(1, total // 128))
    hi = max(128, total // batch)
    lo = hi if rng.random() < 0.3 else max(64, int(hi * rng.uniform(0.3, 1.0)))
    if kind == "positional":
        return _case("", "positional", shape, batch=batch, lo=lo, hi=hi, layout=layout)
    if kind == "fine":
        rows = rng.choice((1, 1, 1, 2, 4))
        keep_lo = keep_hi = round(rng.uniform(0.6, 0.9), 3)
    else:
        rows = _log_int(rng, 5, 128)
        keep_lo = round(rng.uniform(0.25, 0.5), 3)
        keep_hi = round(keep_lo + rng.uniform(0.0, 0.3), 3)
    return _case("", "prune", shape, batch=batch, lo=lo, hi=hi, layout=layout, rows=rows, keep_lo=keep_lo, keep_hi=keep_hi,
                 lse=kind == "global" and rng.random() < 0.25)


# ---- sizes (a case fixes them; only the values come from the seed) -----------------------------------

def _lengths(case):
    rng = random.Random(case["layout"])
    lens = [rng.randint(case["lo"], case["hi"]) for _ in range(case["batch"])]
    keeps = [keep_count(n, rng.uniform(case["keep_lo"], case["keep_hi"])) for n in lens] if "keep_lo" in case else None
    return lens, keeps


def _chain_lengths(case):
    lens = [case["tokens"]]
    for _ in range(case["stages"]):
        lens.append(keep_count(lens[-1], case["keep"]))
    return lens


def _segments(n):
    """Text prefix, audio, video, text suffix: 5 / 15 / 80 %."""
    text, audio = round(0.05 * n), round(0.15 * n)
    return text // 2, audio, n - text - audio, text - text // 2


def _positional_rule(lens):
    """The mask of "the first tokens of each modality": 10 audio tokens and the first third of the video, text whole."""
    parts, cu = [], [0]
    for n in lens:
        pre, audio, video, suf = _segments(n)
        parts += [torch.full((m,), mod, dtype=torch.uint8) for m, mod in ((pre, MOD_TEXT), (audio, MOD_AUDIO), (video, MOD_VIDEO), (suf, MOD_TEXT))]
        cu.append(cu[-1] + n)
    keep_first = {MOD_AUDIO: 10, MOD_VIDEO: round(0.8 * min(lens)) // 3}
    return positional_keep_mask(torch.cat(parts), torch.tensor(cu, dtype=torch.int32), keep_first)


# ---- values -------------------------------------------------------------------------------------------

def _normal(gen, *shape):
    return torch.randn(shape, generator=gen, device="cuda", dtype=torch.bfloat16)


def _queries_keys(gen, case, rows, tokens, anchors=16):
    """q [rows, Hq, d] and k [tokens, Hkv, d] of one sequence and layer."""
    hq, hkv, dim = case["q_heads"], case["kv_heads"], case["dim"]
    shared = torch.randn(hkv, dim, generator=gen, device="cuda")
    q = torch.randn(rows, hkv, hq // hkv, dim, generator=gen, device="cuda") * math.sqrt(1 - SHARED ** 2) + SHARED * shared[:, None, :]
    shift = torch.randn(tokens, generator=gen, device="cuda")
    quarter = max(1, tokens // 4)
    early = torch.randperm(quarter, generator=gen, device="cuda")[:min(anchors, quarter // 4)]
    shift[early] = 3.0
    k = _normal(gen, tokens, hkv, dim)
    k += (shift * (LOGIT_SPREAD / (SHARED * math.sqrt(dim))))[:, None, None].to(torch.bfloat16) * shared.to(torch.bfloat16)
    return q.reshape(rows, hq, dim).to(torch.bfloat16), k


def _cu(counts):
    cu = [0]
    for c in counts:
        cu.append(cu[-1] + c)
    return torch.tensor(cu, dtype=torch.int32)


def _log_sum_exp(q, k, first):
    """What the layer's attention kernel reports for the rows (tokens first, first + 1, ...): [rows, Hq] fp32, causal."""
    rows, hq, dim = q.shape
    n, hkv, _ = k.shape
    out = torch.empty(rows, hq, device="cuda")
    hidden = torch.arange(n, device="cuda")[None, :] > torch.arange(first, first + rows, device="cuda")[:, None]
    for h in range(hq):
        z = (q[:, h].float() @ k[:, h // (hq // hkv)].float().T) / math.sqrt(dim)
        out[:, h] = torch.logsumexp(z.masked_fill_(hidden, -math.inf), dim=1)
    return out


def _prune_buffers(case, gen, lens, keeps, rows, flags=0, hidden=None, pos=None):
    """Device buffers of one prune call."""
    r_per = [min(rows, n) for n in lens]
    pairs = [_queries_keys(gen, case, r, n) for r, n in zip(r_per, lens)]
    lse = torch.cat([_log_sum_exp(q, k, len(k) - len(q)) for q, k in pairs]) if case.get("lse") else None
    total = sum(lens)
    if hidden is None:
        hidden = _normal(gen, total, case["hidden"])
        pos = torch.cat([torch.randperm(2 * n, generator=gen, device="cuda")[:n].sort().values for n in lens]).to(torch.int32)
    buf = F.make_buffers(
        q=torch.cat([p[0] for p in pairs]), k=torch.cat([p[1] for p in pairs]), v=_normal(gen, total, case["kv_heads"], case["dim"]),
        q_idx=torch.cat([torch.arange(n - r, n, dtype=torch.int32) for n, r in zip(lens, r_per)]).cuda(),
        cu_qlens=_cu(r_per).cuda(), cu_seqlens=_cu(lens).cuda(), keep_counts=torch.tensor(keeps, dtype=torch.int32).cuda(),
        hidden=hidden, pos=pos, softmax_scale=1.0 / math.sqrt(case["dim"]),
        flags=F.FASTAV_CAUSAL | F.FASTAV_PROTECT_QUERY_ROWS | flags, lens=lens, rows=r_per, keeps=keeps)
    return buf, lse


def _survivors(buf):
    return {"scores": buf.scores, "keep_idx": buf.keep_idx, "cu_keep": buf.cu_keep, "hidden": buf.hidden_out, "pos": buf.pos_out,
            "k": buf.k_out, "v": buf.v_out}


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kind = case["kind"]
    state = {"kind": kind}
    if kind == "prune":
        lens, keeps = _lengths(case)
        state["buf"], state["lse"] = _prune_buffers(case, gen, lens, keeps, case["rows"])
    elif kind == "chain":
        # one set of buffers per pruning layer; hidden states and positions run through, every layer has its own q, k, v.
        # The survivor counts are known up front, so the index arrays of all layers are uploaded once.
        lens = _chain_lengths(case)
        layers, hidden, pos = [], None, None
        for n, kept in zip(lens, lens[1:]):
            buf, _ = _prune_buffers(case, gen, [n], [kept], 1, F.FASTAV_CHAIN_CALLS, hidden, pos)
            hidden, pos = buf.hidden_out, buf.pos_out
            layers.append(buf)
        state["layers"] = layers
    elif kind == "positional":
        lens, _ = _lengths(case)
        mask = _positional_rule(lens)
        total, hkv, dim = sum(lens), case["kv_heads"], case["dim"]
        kept = int(mask.sum())
        cu = _cu(lens)
        per = [int(mask[cu[b]:cu[b + 1]].sum()) for b in range(len(lens))]
        new = lambda *shape: torch.empty(shape, dtype=torch.bfloat16, device="cuda")
        state.update(mask=mask.cuda(), cu_seqlens=cu.cuda(), hidden=_normal(gen, total, case["hidden"]), k=_normal(gen, total, hkv, dim),
                     v=_normal(gen, total, hkv, dim), pos=torch.cat([torch.arange(n, dtype=torch.int32) for n in lens]).cuda(),
                     keep_idx=torch.empty(kept, dtype=torch.int32, device="cuda"), cu_keep=torch.empty(len(lens) + 1, dtype=torch.int32, device="cuda"),
                     hidden_out=new(kept, case["hidden"]), k_out=new(kept, hkv, dim), v_out=new(kept, hkv, dim),
                     pos_out=torch.empty(kept, dtype=torch.int32, device="cuda"),
                     workspace=torch.empty(max(256, 4 * len(lens) + 256), dtype=torch.uint8, device="cuda"))
        state["params"] = F.make_params(batch=len(lens), total_tokens=total, max_seqlen=max(lens), total_q=0, max_qlen=0, total_keep=kept,
                                        max_keep=max(per), num_q_heads=case["q_heads"], num_kv_heads=hkv, head_dim=dim, hidden=case["hidden"])
    elif kind == "rollout":
        n = case["tokens"]
        state["qk"] = [_queries_keys(gen, case, n, n) for _ in range(case["layers"])]
        params = F.make_params(batch=1, total_tokens=n, max_seqlen=n, total_q=n, max_qlen=n, total_keep=0, max_keep=0,
                               num_q_heads=case["q_heads"], num_kv_heads=case["kv_heads"], head_dim=case["dim"], hidden=0, flags=F.FASTAV_CAUSAL)
        pre, audio, video, suf = _segments(n)
        protect = torch.zeros(n, dtype=torch.uint8)
        protect[:pre] = 1
        protect[n - suf:] = 1
        state.update(n=n, params=params, protect=protect.cuda(), importance=torch.empty(n, device="cuda"), rollout=torch.empty(n, n, device="cuda"),
                     mask=torch.empty(n, dtype=torch.uint8, device="cuda"), cut=torch.empty(1, dtype=torch.int32, device="cuda"),
                     state=torch.empty(F.fastav_rollout_state_bytes(n), dtype=torch.uint8, device="cuda"),
                     workspace=torch.empty(F.fastav_rollout_workspace_bytes(params), dtype=torch.uint8, device="cuda"))
    else:
        lens, keeps = _lengths(case)
        buf, _ = _prune_buffers(case, gen, lens, keeps, case["rows"])
        host = {name: getattr(buf, name).cpu().pin_memory() for name in ("q", "q_idx", "cu_qlens", "k", "v", "cu_seqlens", "keep_counts", "hidden", "pos")}
        out = {name: torch.empty_like(getattr(buf, name), device="cpu").pin_memory()
               for name in ("scores", "keep_idx", "cu_keep", "hidden_out", "pos_out", "k_out", "v_out")}
        state.update(params=buf.params, host=host, out=out, status=torch.zeros(1, dtype=torch.int32).pin_memory(),
                     arena=torch.empty(F.fastav_host_arena_bytes(buf.params), dtype=torch.uint8, device="cuda"))
    return state


def run(state):
    kind = state["kind"]
    if kind == "prune":
        state["buf"].prune(lse_opt=state["lse"])
        return _survivors(state["buf"])
    if kind == "chain":
        for buf in state["layers"]:
            buf.prune()
        last = state["layers"][-1]
        return {"hidden": last.hidden_out, "pos": last.pos_out,
                "layers": [{"scores": b.scores, "keep_idx": b.keep_idx, "k": b.k_out, "v": b.v_out} for b in state["layers"]]}
    if kind == "positional":
        s = state
        F.fastav_select_mask(s["params"], s["mask"], s["cu_seqlens"], s["keep_idx"], s["cu_keep"], s["workspace"])
        F.fastav_compact(s["params"], s["keep_idx"], s["cu_keep"], s["cu_seqlens"], s["hidden"], s["hidden_out"], s["pos"], s["pos_out"],
                         s["k"], s["k_out"], s["v"], s["v_out"])
        return {name: s[name] for name in ("keep_idx", "cu_keep", "hidden_out", "pos_out", "k_out", "v_out")}
    if kind == "rollout":
        s, n = state, state["n"]
        F.fastav_rollout_begin(n, s["state"])
        for i, (q, k) in enumerate(s["qk"]):
            F.fastav_rollout_layer(s["params"], q, k, 0.5, i, s["state"], s["workspace"])
        F.fastav_rollout_read(n, len(s["qk"]), s["state"], s["importance"], s["rollout"])
        F.fastav_rollout_threshold(n, s["importance"], 0.5 / n, s["protect"], s["mask"], s["cut"])
        return {name: s[name] for name in ("importance", "rollout", "mask", "cut")}
    h, o = state["host"], state["out"]
    F.fastav_prune_host(state["params"], h["q"], h["q_idx"], h["cu_qlens"], h["k"], h["v"], h["cu_seqlens"], h["keep_counts"], None, h["hidden"],
                        h["pos"], o["scores"], o["keep_idx"], o["cu_keep"], o["hidden_out"], o["pos_out"], o["k_out"], o["v_out"],
                        state["status"], state["arena"])
    return o


# ---- what a pass cannot do without ------------------------------------------------------------------------

def _score_work(case, tokens, rows):
    """K and the scored rows read once, one score written per token; 2 d operations per (row, head, key)."""
    hq, hkv, dim = case["q_heads"], case["kv_heads"], case["dim"]
    return (2 * sum(tokens) * hkv * dim + 2 * sum(rows) * hq * dim + 4 * sum(tokens),
            sum(2.0 * n * r * hq * dim for n, r in zip(tokens, rows)))


def _gather_bytes(case, kept):
    """A survivor's hidden state, K, V and position, read and written, and its index."""
    return kept * (4 + 2 * (2 * case["hidden"] + 4 * case["kv_heads"] * case["dim"] + 4))


def work(case):
    kind = case["kind"]
    if kind in ("prune", "host"):
        lens, keeps = _lengths(case)
        size, flops = _score_work(case, lens, [min(case["rows"], n) for n in lens])
        return {"bytes": size + _gather_bytes(case, sum(keeps)), "flops": flops}
    if kind == "chain":
        lens = _chain_lengths(case)
        parts = [(_score_work(case, [n], [1]), _gather_bytes(case, kept)) for n, kept in zip(lens, lens[1:])]
        return {"bytes": sum(s[0] + g for s, g in parts), "flops": sum(s[1] for s, _ in parts)}
    if kind == "positional":
        lens, _ = _lengths(case)
        return {"bytes": sum(lens) + _gather_bytes(case, int(_positional_rule(lens).sum())), "flops": 0}
    n, layers = case["tokens"], case["layers"]
    qk = 2 * n * (case["q_heads"] + case["kv_heads"]) * case["dim"]
    # the causal half of Q K^T per head, and the product of two triangular matrices (the first factor is the identity)
    return {"bytes": layers * qk + 4 * n * n + 4 * n, "flops": layers * case["q_heads"] * n * (n + 1.0) * case["dim"] + (layers - 1) * n ** 3 / 3.0}


def tolerance(case):
    """Four times what the present code is off by against the same path in float64 (2-norm; largest difference).

    Few scored rows: exponentials of the special-function unit and fp32 sums, 3e-7 and 7e-7 seen, the rest is what fp32
    sums of another order may add.  Many scored rows: part of the exponentials are a cubic of relative error 7.5e-5, 1e-5
    and 2e-5 seen.  Rollout: factors of about 16 mantissa bits over up to 14 products, 1.2e-5 and 4e-5 seen.  Whole values: a
    score within rounding of the threshold.
    """
    kind = case["kind"]
    if kind == "positional":
        return "exact"
    if kind == "rollout":
        return {"rel": 5e-5, "max": 1.6e-4, "differ": 0.005}
    if kind == "chain" or case["rows"] <= 4:
        return {"rel": 1e-5, "max": 4e-5, "differ": 0.005}
    return {"rel": 4e-5, "max": 1e-4, "differ": 0.005}
