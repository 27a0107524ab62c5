"""The work a user of this library has it do, as measurable cases through the public entry points.

Four kinds of call, the four that a visual on-policy distillation loop makes:

  rollout   hbsjd_rollout / hbsjd_rollout_host: the student's whole rollout of a batch (state init, prefix pre-filling,
            every verification round).  Its outputs are what the call returns: the token rows and the counts of
            its rounds.  The tokens of a free-running rollout are compared exactly: each one is sampled from the logits
            of every round before it, so equal tokens over a whole rollout are the strictest statement about the
            logits that can be made, and an approximate one means nothing (one different token changes all later ones).
  score     hbsjd_score: teacher and student forwards over the finished trajectories and the divergence of Eq. 3.
  verify    hbsjd_verify: one verification step on the caller's logits (probabilities, accept test, commit, refresh).
  probs     hbsjd_probs: the probability pipeline (guidance, temperature, top-k, softmax) on the caller's logits.

Sizes are those of the library's own workloads (synth.WORKLOADS) and ranges around them.  A context is kept for as long
as cases of its size run, as a training loop keeps it: weights do not depend on a case's seed, inputs do.
"""
from __future__ import annotations

import collections
import math

import numpy as np
import torch

from paper_2608_18183_b200 import binding, synth

_W = synth.WORKLOADS
_B, _L, _XL = _W["B"].shape, _W["L"].shape, _W["XL"].shape
MODELS = {
    "tiny": _W["tiny"].shape,   # fp32
    "B": _B,
    "L": _L,
    "XL": _XL,
    # the scoring benchmark's teacher: the XL decoder's width and depth on the student's grid
    "XL_on_L": synth.ModelShape(_XL.n_layers, _XL.dim, _XL.n_heads, _XL.ffn_hidden, _L.vocab, _L.grid_h, _L.grid_w,
                                _L.n_classes, _L.dtype),
}
# committed tokens per image and round that these random-weight models approach with wide windows (for work() only)
ACCEPT = {"tiny": 1.25, "B": 2.6, "L": 2.3, "XL": 1.6}


def _rollout(name, model, batch, window, k_lo, k_hi, cfg=4.0, top_k=1000, temperature=1.0, greedy=False,
             exec_mode="hybrid", host=False):
    c = dict(kind="rollout", model=model, batch=batch, window=window, k_lo=k_lo, k_hi=k_hi, cfg=cfg, top_k=top_k,
             temperature=temperature, greedy=greedy, exec_mode=exec_mode, host=host)
    return dict(c, name=name) if name else c


def _score(name, student, teacher, batch, window, k_lo, k_hi):
    c = dict(kind="score", student=student, teacher=teacher, batch=batch, window=window, k_lo=k_lo, k_hi=k_hi)
    return dict(c, name=name) if name else c


def _verify(name, batch, window, vocab, branches, top_k, temperature=1.0, greedy=False):
    c = dict(kind="verify", batch=batch, window=window, vocab=vocab, branches=branches, top_k=top_k,
             temperature=temperature, greedy=greedy)
    return dict(c, name=name) if name else c


def _probs(name, rows, vocab, guidance, top_k, temperature):
    c = dict(kind="probs", rows=rows, vocab=vocab, guidance=guidance, top_k=top_k, temperature=temperature)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the headline: one training step's rollout of the L student, guidance, wide window, device buffers
        _rollout("rollout_L", "L", 128, 32, 0, 128),
        # the small student without guidance: launch-bound rounds of at most 1024 rows
        _rollout("rollout_B", "B", 64, 16, 0, 64, cfg=1.0),
        # the longest sequences and the deepest model, a handful of images (an evaluation or a small worker)
        _rollout("rollout_XL_few", "XL", 6, 32, 0, 288),
        # one image: an interactive sample, where only latency counts
        _rollout("rollout_L_single", "L", 1, 16, 0, 0),
        # token by token (window 1): the cached autoregressive baseline, a ragged number of images
        _rollout("rollout_L_ar", "L", 24, 1, 0, 128),
        # greedy evaluation through host buffers, odd batch and window, Compact execution
        _rollout("rollout_B_greedy_odd", "B", 37, 11, 5, 90, cfg=1.0, top_k=0, greedy=True, exec_mode="compact",
                 host=True),
        # the fp32 configuration: the smallest rollout
        _rollout("rollout_tiny_fp32", "tiny", 4, 8, 0, 0, cfg=1.0, top_k=0),
        # long real prefixes, few tokens to generate: pre-filling of many rows, an odd batch beyond the headline's
        _rollout("rollout_L_prefill", "L", 200, 32, 176, 240, temperature=0.9),
        # the step after the rollout: full-sequence forwards of student and teacher over a whole batch
        _score("score_L_XL", "L", "XL_on_L", 128, 32, 0, 128),
        # the same for a few trajectories and the small student
        _score("score_B_L_few", "B", "L", 9, 16, 0, 64),
        # one verification step at the headline's sizes, at the paper's commit length
        _verify("verify_L", 128, 32, 16384, 2, 1000),
        # probabilities of an odd number of rows, every option on
        _probs("probs_odd", 1537, 16384, True, 1000, 0.7),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def _seconds(c):
    """A rough time of a rollout, to keep drawn ones below the largest listed one."""
    s = MODELS[c["model"]]
    w = work(c)
    rounds, fills = _rounds(c)
    return (rounds + fills) * (s.n_layers * 70e-6 + 1e-4) + w["flops"] / (0.75e15 if s.dtype == "bf16" else 20e12)


def draw(rng):
    kind = rng.choice(["rollout"] * 6 + ["score", "verify", "verify", "probs"])
    if kind == "rollout":
        most = max(_seconds(c) for c in listed() if c["kind"] == "rollout")
        while True:
            model = rng.choice(["tiny", "B", "B", "L", "L", "L", "XL"])
            T = MODELS[model].T
            batch = _log_int(rng, 1, {"tiny": 32, "B": 96, "L": 160, "XL": 8}[model])
            window = _log_int(rng, 1, min(32, T // 2))
            k_lo = rng.randrange(0, 3 * T // 4)
            k_hi = rng.randrange(k_lo, T - T // 16)
            greedy = rng.random() < 0.25
            c = _rollout(None, model, batch, window, k_lo, k_hi,
                         cfg=1.0 if model == "tiny" or rng.random() < 0.35 else rng.choice([1.5, 3.0, 4.0, 7.5]),
                         top_k=0 if model == "tiny" else rng.choice([0, 100, 1000, 1000, 2000]),
                         temperature=rng.choice([1.0, 1.0, 0.9, 0.7]), greedy=greedy,
                         exec_mode=rng.choice(["hybrid", "hybrid", "compact", "full"]), host=rng.random() < 0.3)
            if _seconds(c) <= most:
                return c
    if kind == "score":
        student, teacher = rng.choice([("B", "L"), ("B", "XL_on_L"), ("L", "XL_on_L")])
        k_lo = rng.randrange(0, 128)
        return _score(None, student, teacher, _log_int(rng, 1, 128), rng.randrange(4, 33), k_lo,
                      rng.randrange(k_lo, 240))
    if kind == "verify":
        vocab = rng.choice([4096, 8192, 16384, 16384, 32768])
        window = rng.randrange(2, 33)
        return _verify(None, _log_int(rng, 1, max(1, 128 * 32 * 16384 // (window * vocab))), window, vocab,
                       rng.choice([1, 2]), rng.choice([0, 100, 1000, 1000]), rng.choice([1.0, 0.9]),
                       rng.random() < 0.2)
    vocab = rng.choice([4096, 8192, 16384, 16384, 32768])
    return _probs(None, _log_int(rng, 1, 4096 * 16384 // vocab), vocab, rng.random() < 0.6,
                  rng.choice([0, 100, 1000, 1000]), rng.choice([1.0, 0.7]))


# ---------------------------------------------------------------------------------------------- contexts

def make_weights(shape, seed):
    """Random weights in the library's flat layout, as synth.make_weights makes them (every matrix N(0, 0.02), gains 1,
    the LM head scaled for a mean next-token entropy of 3 nats), drawn on the GPU."""
    table, total = synth.tensor_table(shape)
    img = np.zeros(total, dtype=np.uint8)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    dt = torch.bfloat16 if shape.dtype == "bf16" else torch.float32
    for name, r, c, off in table:
        if name.endswith("g_attn") or name.endswith("g_ffn") or name == "g_out":
            t = torch.ones(r, c, device="cuda")
        else:
            t = torch.randn(r, c, device="cuda", generator=g) * 0.02
            if name == "w_head":
                d = torch.randn(64, shape.dim, device="cuda", generator=g, dtype=torch.float64)
                base = (d / d.square().mean(1, keepdim=True).sqrt()) @ t.double().T
                lo, hi = 0.0, 4096.0
                for _ in range(24):
                    mid = 0.5 * (lo + hi)
                    lp = torch.log_softmax(mid * base, dim=1)
                    entropy = float(-(lp.exp() * lp).sum(1).mean())
                    lo, hi = (mid, hi) if entropy > min(3.0, 0.7 * math.log(shape.vocab)) else (lo, mid)
                t = t * round(lo, 2)
        img[off:off + r * c * shape.elem_bytes] = t.to(dt).contiguous().view(torch.uint8).reshape(-1).cpu().numpy()
    return img


_contexts = collections.OrderedDict()


def _context(model, batch, window):
    """The context of this size, kept while it is in use: at most two live at once (a student and a teacher)."""
    key = (model, batch, window)
    if key in _contexts:
        _contexts.move_to_end(key)
        return _contexts[key]
    while len(_contexts) >= 2:
        _contexts.popitem(last=False)  # freed with its last state
    if isinstance(model, int):  # the stand-alone entry points use a context's vocabulary, limits and scratch only
        shape = synth.ModelShape(1, 64, 1, 64, model, 4, 4, 3, "bf16")
    else:
        shape = MODELS[model]
    _contexts[key] = binding.Context(shape, make_weights(shape, 1 + len(str(model))), batch, window)
    return _contexts[key]


# ---------------------------------------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _batch_inputs(shape, c, g):
    b = c["batch"]
    toks = torch.randint(0, shape.vocab, (b, shape.T), device="cuda", generator=g, dtype=torch.int32)
    k = torch.randint(c["k_lo"], c["k_hi"] + 1, (b,), device="cuda", generator=g, dtype=torch.int32)
    lab = torch.randint(0, shape.n_classes, (b,), device="cuda", generator=g, dtype=torch.int32)
    return toks, k, lab


def _prepare_rollout(c, seed):
    s = MODELS[c["model"]]
    ctx = _context(c["model"], c["batch"], c["window"])
    toks, k, lab = _batch_inputs(s, c, _gen(seed))
    mode = {"full": binding.EXEC_FULL, "compact": binding.EXEC_COMPACT, "hybrid": binding.EXEC_HYBRID}[c["exec_mode"]]
    # the threshold the library measures for itself: Compact at every live count (see hbsjd_calibrate_gamma)
    p = binding.make_params(c["window"], s.grid_w, c["cfg"], c["temperature"], c["top_k"],
                            binding.VERIFY_GREEDY if c["greedy"] else binding.VERIFY_PROB, mode, c["batch"], seed, -1)
    out = torch.empty(c["batch"], s.T, dtype=torch.int32, device="cuda")
    if c["host"]:
        toks, k, lab, out = (x.cpu().pin_memory() for x in (toks, k, lab, out))
    return dict(kind="rollout", host=c["host"], ctx=ctx, toks=toks, k=k, lab=lab, params=p, out=out)


def _prepare_score(c, seed):
    s = MODELS[c["student"]]
    stu, tea = _context(c["student"], c["batch"], c["window"]), _context(c["teacher"], c["batch"], c["window"])
    toks, k, lab = _batch_inputs(s, c, _gen(seed))
    return dict(kind="score", ctx=stu, teacher=tea, toks=toks, k=k, lab=lab)


def _topk_filter(x, top_k):
    if 0 < top_k < x.shape[-1]:
        kth = torch.topk(x, top_k, dim=-1).values[..., -1:]
        x = x.masked_fill(x < kth, float("-inf"))
    return x


def _prepare_verify(c, seed):
    """Targets p = softmax of the guided logits, proposals q of the same with noise on the logits (sigma 1.49: the
    paper's mean commit of 2.3 tokens at the headline's sizes), drafts drawn from q, 15 % point-mass drafts, ragged
    cursors up to the end of the sequence."""
    B, W, V, T, scale = c["batch"], c["window"], c["vocab"], 256, 4.0
    g = _gen(seed)
    ctx = _context(V, B, W)
    cond = torch.randn(B, W, V, device="cuda", generator=g) * 2.5
    if c["branches"] == 2:
        unc = cond * 0.5 + torch.randn(B, W, V, device="cuda", generator=g)
        logits, guided = torch.stack([cond, unc]), unc + scale * (cond - unc)
    else:
        logits, guided = cond[None].clone(), cond
    cursor = torch.randint(0, T, (B,), device="cuda", generator=g, dtype=torch.int32)
    back = torch.randint(1, 4, (B,), device="cuda", generator=g, dtype=torch.int32)
    qbase = torch.clamp(cursor - back, min=0)
    shift = (cursor - qbase).long()
    noisy = guided / c["temperature"] + 1.49 * torch.randn(B, W, V, device="cuda", generator=g)
    q = torch.softmax(_topk_filter(noisy, c["top_k"]), dim=-1)
    del noisy, guided, cond
    # the proposal of the draft at window position i sits in row i + shift of the previous round's probabilities
    rows = (torch.arange(W, device="cuda")[None, :] - shift[:, None]) % W
    q = torch.gather(q, 1, rows[:, :, None].expand(B, W, V)).contiguous()
    draws = torch.multinomial(q.view(B * W, V), 1, generator=g).view(B, W).to(torch.int32)
    state = torch.zeros(4 * (2 * B + B * (T + 1)) + B * (T + 1), dtype=torch.uint8, device="cuda")
    cur, qb, seq, delta = _state_views(state, B, T)
    cur.copy_(cursor)
    qb.copy_(qbase)
    seq.copy_(torch.randint(0, V, (B, T + 1), device="cuda", generator=g, dtype=torch.int32))
    delta.fill_(1)
    i = torch.arange(W - 1, device="cuda")[None, :]
    t, qi = cursor.long()[:, None] + 1 + i, i + shift[:, None]
    ok = (qi < W) & (t <= T) & (torch.rand(B, W - 1, device="cuda", generator=g) < 0.85)
    b = torch.arange(B, device="cuda")[:, None].expand(B, W - 1)
    seq[b[ok], t[ok]] = draws[b[ok], qi[ok]]
    delta[b[ok], t[ok]] = 0
    work_state = state.clone()
    desc = binding.hbsjd_verify_desc(B, W, T, V, c["branches"], 16, 1 if c["greedy"] else 0, c["top_k"], scale,
                                     c["temperature"], seed, 7, 0)
    return dict(kind="verify", ctx=ctx, desc=desc, logits=logits.contiguous(), q=q,
                p=torch.zeros(B, W, V, device="cuda"), m=torch.zeros(B, dtype=torch.int32, device="cuda"),
                before=state, state=work_state, views=_state_views(work_state, B, T))


def _state_views(buf, B, T):
    """cursor, qbase, seq (int32) and delta (uint8) of a rollout inside one buffer."""
    ints = buf[:4 * (2 * B + B * (T + 1))].view(torch.int32)
    return (ints[:B], ints[B:2 * B], ints[2 * B:].view(B, T + 1), buf[4 * (2 * B + B * (T + 1)):].view(B, T + 1))


def _prepare_probs(c, seed):
    g = _gen(seed)
    ctx = _context(c["vocab"], 2, 4)
    lc = torch.randn(c["rows"], c["vocab"], device="cuda", generator=g) * 3.5
    lu = torch.randn(c["rows"], c["vocab"], device="cuda", generator=g) * 3.5 if c["guidance"] else None
    return dict(kind="probs", ctx=ctx, lc=lc, lu=lu, cfg=4.0 if c["guidance"] else 1.0,
                temperature=c["temperature"], top_k=c["top_k"])


def prepare(case, seed):
    return {"rollout": _prepare_rollout, "score": _prepare_score, "verify": _prepare_verify,
            "probs": _prepare_probs}[case["kind"]](case, seed)


# ---------------------------------------------------------------------------------------------- one pass

_COUNTS = ("rounds", "image_forwards", "committed", "rejects", "full_rounds", "compact_rounds", "prefill_forwards")


def run(state):
    s, ctx = state, state["ctx"]
    if s["kind"] == "rollout":
        call = ctx.hbsjd_rollout_host if s["host"] else ctx.hbsjd_rollout
        tokens, stats = call(s["toks"], s["k"], s["lab"], s["params"], s["out"])
        return {"tokens": tokens, "stats": {n: stats[n] for n in _COUNTS}}
    if s["kind"] == "score":
        pos, per_image, loss = ctx.hbsjd_score(s["teacher"], s["toks"], s["k"], s["lab"])
        return {"pos": pos, "per_image": per_image, "loss": loss}
    if s["kind"] == "verify":
        s["state"].copy_(s["before"])  # the call advances the rollout state in place
        cur, qb, seq, delta = s["views"]
        ctx.hbsjd_verify(s["desc"], s["logits"], s["q"], s["p"], cur, seq, delta, qb, s["m"])
        return {"p": s["p"], "cursor": cur, "qbase": qb, "seq": seq, "delta": delta, "m": s["m"]}
    return ctx.hbsjd_probs(s["lc"], s["lu"], s["cfg"], s["temperature"], s["top_k"])


# ---------------------------------------------------------------------------------------------- what a pass needs

def _rounds(c):
    """(rounds, prefill forwards) of a rollout, from the mean accepted tokens per forward."""
    T, W = MODELS[c["model"]].T, c["window"]
    cap = ACCEPT[c["model"]]
    acc = cap - (cap - 1.0) / W ** 0.8
    k_min = c["k_lo"] + (c["k_hi"] - c["k_lo"]) / (c["batch"] + 1)
    return (T - k_min) / acc, math.ceil(c["k_hi"] / W)


def _block_params(s):
    return s.n_layers * (4 * s.dim * s.dim + 3 * s.dim * s.ffn_hidden)


def work(case):
    c = case
    if c["kind"] == "rollout":
        s = MODELS[c["model"]]
        nb = 2 if c["cfg"] != 1.0 else 1
        rounds, fills = _rounds(c)
        cap = ACCEPT[c["model"]]
        k = 0.5 * (c["k_lo"] + c["k_hi"])
        forwards = c["batch"] * (s.T - k) / (cap - (cap - 1.0) / c["window"] ** 0.8)  # images x rounds
        head = s.dim * s.vocab
        flops = 2.0 * nb * (forwards * c["window"] * (_block_params(s) + head) + c["batch"] * k * _block_params(s))
        kv = 2.0 * s.n_layers * s.dim * s.elem_bytes  # one token's keys and values
        return {"bytes": (rounds + fills) * _block_params(s) * s.elem_bytes + rounds * head * s.elem_bytes +
                nb * forwards * kv * 0.5 * (s.T + k), "flops": flops}
    if c["kind"] == "score":
        flops = nbytes = 0.0
        for m in (c["student"], c["teacher"]):
            s = MODELS[m]
            n = _block_params(s) + s.dim * s.vocab
            flops += 2.0 * n * c["batch"] * s.T
            nbytes += n * s.elem_bytes
        return {"bytes": nbytes + 4.0 * c["batch"] * MODELS[c["student"]].T, "flops": flops}
    if c["kind"] == "verify":
        return {"bytes": 4.0 * c["batch"] * c["window"] * c["vocab"] * (c["branches"] + 1), "flops": 0}
    return {"bytes": 4.0 * c["rows"] * c["vocab"] * (3 if c["guidance"] else 2), "flops": 0}


def tolerance(case):
    if case["kind"] == "rollout":
        return "exact"  # whole numbers; see the head of the file
    if case["kind"] == "score":
        # bf16 activations: the library's two forms of RMSNorm (hbsjd_debug_fold_norm) differ by 3.3e-3 in the 2-norm and
        # 2.0e-2 at one position (score_L_XL; 2.5e-3 and 1.2e-2 at score_B_L_few); four times that
        return {"rel": 1.3e-2, "max": 8e-2}
    # fp32 softmax: 1.1e-6 and 2.1e-5 from the same pipeline in 64 bits (probs_odd; 3.8e-7 and 3.4e-6 at verify_L); four times
    # that.  A draw whose target lies within the last bits of a cumulative sum may fall on its neighbour.
    return {"rel": 5e-6, "max": 1e-4, "differ": 1e-3}
