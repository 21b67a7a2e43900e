"""The work that a user of this package has it do, as timed cases.

A serving program that decodes with a draft calls the package once per decoding step, for whatever requests are in
flight: the whole verify step (attention over the token tree, LM head, acceptance) on inputs that are already on the
device, the same step over an 8-bit cache, or fed from pinned host memory; the target's layers that produce those
inputs, with the roll-forward of the cache behind them; and the early-exit tap or the 8-bit LM head on their own.  All
of it is decoding: the package has no training path, and a prompt goes through the layers like a tree of one chain.

Values: queries, keys and values, hidden rows (they come out of an RMSNorm) and residual rows are N(0, 1); weights keep
unit rows at unit size.  Hidden rows lean towards one token of the vocabulary, whose logit leads by 14 to 24, and the
draft guesses that token most of the time, as a trained target and its draft do: some branches are accepted to some
depth, and no decision hangs on the last bit of a sum.
"""
import math
import random

import torch

from paper_2510_13161_b200 import binding, inputs

# Model shapes of the package's own configurations: hidden, query heads, KV heads, head size, vocabulary.
_TINY = dict(hidden=256, hq=4, hkv=2, d=64, vocab=1024)
_14B = dict(hidden=5120, hq=40, hkv=8, d=128, vocab=152064)
_32B = dict(hidden=5120, hq=64, hkv=8, d=128, vocab=152064)
_66B = dict(hidden=8192, hq=64, hkv=8, d=128, vocab=128256)

_MODES = {"greedy": binding.ACCEPT_GREEDY, "spec_sampling": binding.ACCEPT_SPEC_SAMPLING, "spec_tree": binding.ACCEPT_SPEC_TREE}


def listed():
    return [
        # One short request of a toy model: launch latency and the host's own work are all there is.
        dict(name="tiny_step", kind="step", **_TINY, layers=1, batch=1, lo=128, hi=128, kappa=2, gamma=4, mode="greedy"),
        # A chat turn on a 14B target, one request, greedy: the ordinary call, bound by the weights and the cache.
        dict(name="14b_step", kind="step", **_14B, layers=48, batch=1, lo=2048, hi=2048, kappa=4, gamma=4, mode="greedy"),
        # The same target at the paper's operating point (8 branches of 7) with the lossless rule over the tree.
        dict(name="14b_tree_step", kind="step", **_14B, layers=48, batch=1, lo=2048, hi=2048, kappa=8, gamma=7, mode="spec_tree"),
        # Eight requests of ragged lengths in one batch, sampled: a server under load.
        dict(name="14b_batch8_step", kind="step", **_14B, layers=48, batch=8, lo=512, hi=4096, kappa=8, gamma=6, mode="spec_sampling"),
        # One long document: 32k tokens of context.
        dict(name="32b_long_step", kind="step", **_32B, layers=64, batch=1, lo=32768, hi=32768, kappa=4, gamma=8, mode="greedy"),
        # The largest batch of the largest target: the tensor cores' end of the range.
        dict(name="66b_batch16_step", kind="step", **_66B, layers=80, batch=16, lo=1024, hi=8192, kappa=8, gamma=8, mode="spec_sampling"),
        # Long contexts are what an 8-bit cache is for: four requests that would not fit otherwise.
        dict(name="32b_fp8_cache_step", kind="step_fp8", **_32B, layers=64, batch=4, lo=4096, hi=16384, kappa=4, gamma=4, mode="greedy"),
        # The target's queries and tree K/V arrive in pinned host memory (the target's layers run elsewhere).
        dict(name="14b_host_step", kind="step_host", **_14B, layers=48, batch=1, lo=2048, hi=2048, kappa=4, gamma=4, mode="greedy"),
        # The target's own layers on the tree's tokens, and the accepted path appended to the cache.
        dict(name="14b_layers", kind="layers", **_14B, inter=17408, layers=48, batch=1, lo=2048, hi=2048, kappa=4, gamma=4),
        # The same of a toy model of two layers: many launches, hardly any work.
        dict(name="tiny_layers", kind="layers", **_TINY, inter=512, layers=2, batch=1, lo=100, hi=100, kappa=3, gamma=4),
        # The early-exit message to the draft: the 8 best tokens of each of the window's rows.
        dict(name="14b_early_exit", kind="tap", **_14B, rows=57, topk=8),
        # The LM head with 8-bit weights on a small batch's rows (the rows are quantised on each call).
        dict(name="14b_fp8_head", kind="head_fp8", **_14B, rows=68),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    most = {"s": _seconds(listed()[5]), "gb": 32.0}
    while True:
        kind = rng.choices(["step", "step_fp8", "step_host", "layers", "tap", "head_fp8"], [10, 2, 2, 3, 2, 1])[0]
        c = dict(kind=kind, hidden=256 * _log_int(rng, 2, 32), vocab=_log_int(rng, 8000, 152064))
        c["d"] = 128 if c["hidden"] >= 1024 or kind == "step_fp8" else 64
        c["hkv"] = rng.choice([2, 4, 8])
        c["hq"] = c["hkv"] * rng.choice([2, 4, 5, 7, 8])
        if kind in ("tap", "head_fp8"):
            c["rows"] = _log_int(rng, 1, 1040)
            if kind == "tap":
                c["topk"] = rng.randint(1, 16)
            return c
        c["layers"] = _log_int(rng, 1, 80)
        c["batch"] = _log_int(rng, 1, 16)
        c["lo"] = _log_int(rng, 64, 16384)
        c["hi"] = c["lo"] if c["batch"] == 1 else min(32768, int(c["lo"] * rng.uniform(1.0, 8.0)))
        c["kappa"], c["gamma"] = rng.randint(1, 8), rng.randint(1, 8)
        if kind == "layers":
            c["inter"] = 64 * max(1, int(c["hidden"] * rng.uniform(2.0, 3.6) / 64))
        else:
            c["mode"] = rng.choice(sorted(_MODES))
        if kind == "step_host":
            c["batch"], c["hi"] = min(c["batch"], 4), c["lo"]
        if _seconds(c) <= most["s"] and _gigabytes(c) <= most["gb"]:
            return c


def _nodes(c):
    return 1 + c["kappa"] * c["gamma"]


def _attention(c):
    """(bytes, flops) of the attention of all layers: cache, tree K/V and queries read, outputs written."""
    n, mean = _nodes(c), (c["lo"] + c["hi"]) / 2
    e = 1 if c["kind"] == "step_fp8" else 2
    b = c["layers"] * c["batch"] * (2 * (mean + n) * c["hkv"] * c["d"] * e + 2 * n * c["hq"] * c["d"] * 2)
    f = c["layers"] * c["batch"] * 4 * c["d"] * c["hq"] * n * (mean + 1 + c["gamma"] / 2)
    return b, f


def work(case):
    c = case
    v, h = c["vocab"], c["hidden"]
    if c["kind"] in ("tap", "head_fp8"):
        m = c["rows"]
        out = m * c["topk"] * 6 if c["kind"] == "tap" else m * 12
        return {"bytes": v * h * (1 if c["kind"] == "head_fp8" else 2) + m * h * 2 + out, "flops": 2 * m * v * h}
    b, f = _attention(c)
    m = c["batch"] * _nodes(c)
    if c["kind"] == "layers":
        per = (c["hq"] + 2 * c["hkv"]) * c["d"] * h + h * c["hq"] * c["d"] + 3 * c["inter"] * h
        # weights; embedding rows in, stream and normed rows out; the tree's K/V written once more into the cache
        return {"bytes": b + c["layers"] * (per * 2 + m * 2 * c["hkv"] * c["d"] * 2) + 4 * m * h * 2, "flops": f + c["layers"] * 2 * m * per}
    b += v * h * 2 + m * h * 2
    if c["mode"] != "greedy":
        b += c["batch"] * v * 4                       # at least one row of the draft's distributions per request
    return {"bytes": b, "flops": f + 2 * m * v * h}


def _seconds(c):
    w = work(c)
    return max(w["bytes"] / 6.4e12, w["flops"] / 1.4e15) + (0.0 if c["kind"] != "step_host" else _attention(c)[0] / 6e12)


def _gigabytes(c):
    m = c["batch"] * _nodes(c)
    g = c["layers"] * c["batch"] * 2 * c["hi"] * c["hkv"] * c["d"] * (3 if c["kind"] == "step_fp8" else 2) + 4 * c["layers"] * m * c["hq"] * c["d"] * 2
    g += c["vocab"] * c["hidden"] * 2 + 2 * m * c["vocab"] * 4
    if c["kind"] == "layers":
        g = work(c)["bytes"] + 2 * m * 16 * c["hidden"]
    if c["kind"] == "step_host":
        g += 20 * c["layers"] * m * c["hq"] * c["d"] * 2          # (pinned memory is dear: few and small)
    return g / 1e9


def tolerance(case):
    if case["kind"] == "head_fp8":
        return {"rel": 1e-5, "differ": 0.005}          # exact products, 32-bit sums
    if case["kind"] == "tap":
        return {"rel": 4e-3, "differ": 0.01}           # log-probabilities are sent in bf16
    if case["kind"] == "layers":
        return {"rel": 2e-2, "differ": 0.0}            # bf16 stored between all steps of up to 80 layers
    if case["kind"] == "step_fp8":
        return {"rel": 3e-2, "differ": 0.01}           # softmax weights enter an 8-bit product as e4m3
    return {"rel": 1e-2, "differ": 0.01}               # bf16 outputs


def _config(c):
    return inputs.VerifyConfig("case", c["hidden"], c["hq"], c["hkv"], c["d"], c.get("layers", 1), c.get("batch", 1), c.get("lo", 0), c.get("hi", 0),
                               c.get("kappa", 1), c.get("gamma", 1), c["vocab"], c.get("mode", "greedy"), explicit_hidden=True)


def _mirror(c):
    return binding.Mirror(c["hidden"], c["hq"], c["hkv"], c["d"], c["vocab"])


def _leaning(hidden, W, gen):
    """Hidden rows that lean towards one token each, and those tokens."""
    m, h = hidden.shape
    y = torch.randint(0, W.shape[0], (m,), generator=gen, device="cuda")
    lead = torch.empty((m, 1), device="cuda").uniform_(14.0, 24.0, generator=gen)
    w = W[y].float()
    return (hidden.float() + w * (lead / w.square().sum(1, keepdim=True))).to(torch.bfloat16), y


def _draft(x, y, rng):
    """Tokens of a draft that is right about four times in five: of a node's children one is the target's own token."""
    B, n = x.tokens.shape
    tokens, y = x.tokens.cpu(), y.view(B, n).cpu()
    for b in range(B):
        served = set()
        for c in range(1, n):
            p = x.parent[c]
            if p not in served and rng.random() < 0.8:
                served.add(p)
                tokens[b, c] = y[b, p]
    return tokens.to(torch.int32).cuda()


def _prepare_step(c, seed):
    cfg = _config(c)
    x = inputs.gen_verify_inputs(cfg, seed, "cuda")
    gen = torch.Generator(device="cuda").manual_seed(seed * 7 + 1)
    hidden, y = _leaning(x.hidden, x.W, gen)
    x.tokens = _draft(x, y, random.Random(seed))
    if x.q_probs is not None:
        # the draft's distribution of each node has most of its mass on the token that it proposed
        at = x.tokens[:, 1:].long().unsqueeze(-1)
        boost = torch.empty(at.shape, device="cuda").uniform_(0.6, 0.98, generator=gen)
        x.q_probs.mul_(1.0 - boost).scatter_add_(2, at, boost)
    m = _mirror(c)
    s = dict(kind=c["kind"], m=m, hidden=hidden, W=x.W, attn=torch.empty_like(x.q), argmax=torch.empty(cfg.rows, dtype=torch.int32, device="cuda"))
    s["tree"] = m.tree(x.tokens, cfg.kappa, cfg.gamma)
    s["acc"] = m.accept_in(_MODES[c["mode"]], True, q_probs=x.q_probs, u_accept=x.u_accept, u_resample=x.u_resample)
    s["out"] = binding.AcceptResult(cfg.batch, cfg.gamma, "cuda")
    if c["kind"] == "step_fp8":
        page = inputs.PAGE_SIZE * c["d"]
        s["ks"], s["vs"] = m.mirror_kv_scales_fp8(x.k_pool, page), m.mirror_kv_scales_fp8(x.v_pool, page)
        k8, v8 = m.mirror_kv_quantize_fp8(x.k_pool, page, s["ks"]), m.mirror_kv_quantize_fp8(x.v_pool, page, s["vs"])
        s["kn"], s["vn"] = m.mirror_kv_quantize_fp8(x.k_new, c["d"], s["ks"]), m.mirror_kv_quantize_fp8(x.v_new, c["d"], s["vs"])
        s["kv"], s["q"], s["q_scale"] = m.kv_fp8(k8, v8, x.page_table, x.prefix_len), x.q, 6.0 / 448.0
        return s
    s["kv"] = m.kv(x.k_pool, x.v_pool, x.page_table, x.prefix_len)
    s["q"], s["kn"], s["vn"] = x.q, x.k_new, x.v_new
    if c["kind"] == "step_host":
        s["d_in"] = dict(q=x.q, k_new=x.k_new, v_new=x.v_new, tokens=x.tokens)
        s["h_in"] = {k: t.cpu().pin_memory() for k, t in s["d_in"].items()}
        host = lambda *shape: torch.empty(shape, dtype=torch.int32).pin_memory()  # noqa: E731
        s["h_out"] = dict(n_accepted=host(cfg.batch), best_branch=host(cfg.batch), n_emitted=host(cfg.batch), emitted=host(cfg.batch, cfg.gamma + 1))
    return s


def _prepare_layers(c, seed):
    cfg = _config(c)
    L, B, n, bf = cfg.layers, cfg.batch, cfg.n_nodes, torch.bfloat16
    m = _mirror(c)
    layers, norm_final, _ = inputs.gen_layer_weights(cfg, c["inter"], L, seed, "cuda", w_std=1.4 / math.sqrt(cfg.hidden))
    gen = torch.Generator(device="cuda").manual_seed(seed)
    normal = lambda *shape: torch.empty(shape, dtype=bf, device="cuda").normal_(0, 1.0, generator=gen)  # noqa: E731
    prefix = inputs.draw_prefix_lens(cfg, seed)
    table, pages = inputs.gen_page_table(prefix, seed, headroom=cfg.gamma + 1)
    k_pool, v_pool = normal(L, pages, cfg.n_kv_heads, inputs.PAGE_SIZE, cfg.head_dim), normal(L, pages, cfg.n_kv_heads, inputs.PAGE_SIZE, cfg.head_dim)
    tokens = torch.randint(0, cfg.vocab, (B, n), generator=gen, device="cuda").to(torch.int32)
    # what the acceptance of this step will say: a branch of each request, accepted to some depth
    rng, out = random.Random(seed), binding.AcceptResult(B, cfg.gamma, "cuda")
    depth = [rng.randint(0, cfg.gamma) for _ in range(B)]
    branch = [rng.randrange(cfg.kappa) for _ in range(B)]
    out.n_accepted.copy_(torch.tensor(depth, dtype=torch.int32))
    out.accepted_nodes.copy_(torch.tensor([[1 + k * cfg.gamma + j if j < a else -1 for j in range(cfg.gamma)] for k, a in zip(branch, depth)], dtype=torch.int32))
    s = dict(kind="layers", m=m, embed=normal(cfg.vocab, cfg.hidden), tokens=tokens, x=torch.empty((B * n, cfg.hidden), dtype=bf, device="cuda"), accepted=out)
    s["target"] = m.target(layers, norm_final, c["inter"])
    s["tree"] = m.tree(tokens, cfg.kappa, cfg.gamma)
    s["kv"] = m.kv(k_pool, v_pool, table.cuda(), prefix.cuda())
    s["scratch"] = m.target_scratch(s["tree"], s["target"])
    new = lambda heads: torch.empty((L, B, n, heads, cfg.head_dim), dtype=bf, device="cuda")  # noqa: E731
    s["res"] = dict(q=new(cfg.n_q_heads), k_new=new(cfg.n_kv_heads), v_new=new(cfg.n_kv_heads), attn_out=new(cfg.n_q_heads),
                    x_out=torch.empty_like(s["x"]), hidden=torch.empty_like(s["x"]))
    s["pools"], s["next_len"], s["prefix"] = (k_pool, v_pool), prefix.cuda(), prefix.cuda()
    return s


def prepare(case, seed):
    c = case
    if c["kind"].startswith("step"):
        return _prepare_step(c, seed)
    if c["kind"] == "layers":
        return _prepare_layers(c, seed)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    W = torch.empty((c["vocab"], c["hidden"]), dtype=torch.bfloat16, device="cuda").normal_(0, 0.02, generator=gen)
    hidden, _ = _leaning(torch.empty((c["rows"], c["hidden"]), dtype=torch.bfloat16, device="cuda").normal_(0, 1.0, generator=gen), W, gen)
    m = _mirror(c)
    s = dict(kind=c["kind"], m=m, hidden=hidden)
    if c["kind"] == "tap":
        s["W"], s["topk"] = W, c["topk"]
    else:
        s["W8"], s["ws"] = m.mirror_quantize_rows_fp8(W)
    return s


def run(s):
    m = s["m"]
    if s["kind"] == "tap":
        return m.mirror_early_exit_tap(s["hidden"], s["W"], s["topk"])
    if s["kind"] == "head_fp8":
        h8, hs = m.mirror_quantize_rows_fp8(s["hidden"])
        r = m.mirror_lmhead_reduce_fp8(h8, hs, s["W8"], s["ws"])
        return r["argmax"], r["maxlogit"], r["lse"]
    if s["kind"] == "layers":
        x = m.mirror_embed_rows(s["embed"], s["tokens"], out=s["x"])
        r = m.mirror_target_forward(s["target"], s["kv"], s["tree"], x, scratch=s["scratch"], out=s["res"])
        s["next_len"].copy_(s["prefix"])               # (the request's length before this step: the commit advances it)
        m.mirror_kv_commit(s["kv"], s["tree"], r["k_new"], r["v_new"], s["accepted"], s["next_len"])
        return r["x_out"], r["hidden"], r["q"], r["k_new"], r["v_new"], r["attn_out"], s["pools"], s["next_len"]
    o = s["out"]
    if s["kind"] == "step_fp8":
        m.mirror_verify_step_fp8(s["kv"], s["tree"], s["q"], s["kn"], s["vn"], s["ks"], s["vs"], s["q_scale"], s["hidden"], s["W"], s["acc"], s["attn"],
                                 out=o, argmax_out=s["argmax"])
    elif s["kind"] == "step_host":
        m.mirror_verify_step_host(s["kv"], s["tree"], s["h_in"], s["d_in"], s["hidden"], s["W"], s["acc"], s["attn"], o, h_out=s["h_out"])
    else:
        m.mirror_verify_step(s["kv"], s["tree"], s["q"], s["kn"], s["vn"], s["hidden"], s["W"], s["acc"], s["attn"], out=o, argmax_out=s["argmax"])
    got = (s["attn"], o.n_accepted, o.best_branch, o.n_emitted, o.emitted, o.accepted_nodes, o.decide_row, o.reuse_slot)
    return got + (s["h_out"],) if s["kind"] == "step_host" else got + (s["argmax"],)
