"""Workloads of prefix-shared preference training on one GPU, for timing.

Every case is one call sequence that a training program makes through the package's public entry
points: attention forward and backward of a pack, the frozen reference model's forward and log-probs,
the loss and its gradient into the logits, a whole small step, an attention layer, or a step on host
buffers.  Sample lengths follow the repository's own workloads (workloads.py); values are N(0, 1)
activations and N(0, variance 3) logits, as in bench.py and the tests.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2410_20305_b200 as psa
from paper_2410_20305_b200 import workloads as wl
from paper_2410_20305_b200.layer import AttentionLayer

RECIPES = {"llama3-8b": 1, "long-prompt": 2, "multi-turn": 3, "short-many": 4}
HEADS = ((32, 8, 128), (8, 2, 128), (16, 16, 64), (8, 2, 64), (32, 8, 64), (4, 4, 64), (8, 8, 128))


def listed():
    full = {"heads": 32, "kv_heads": 8, "head_dim": 128}
    return [
        # The smallest training step (the tiny configuration): planning, attention, log-probs, loss and
        # logits gradient.  Launches and host time are what it consists of.
        {"name": "step-tiny", "kind": "step", "recipe": "tiny", "tokens": 672, "lengths": 0, "heads": 4, "kv_heads": 4,
         "head_dim": 64, "vocab": 1024, "dtype": "f32", "loss": "dpo"},
        # A small step on a fine-tuning box: few short samples, grouped heads of size 64, bf16 logits.
        {"name": "step-small", "kind": "step", "recipe": "short-many", "tokens": 2048, "lengths": 11, "heads": 8,
         "kv_heads": 2, "head_dim": 64, "vocab": 32000, "dtype": "bf16", "loss": "orpo"},
        # Attention of one layer of a training step, forward and backward, on the packs of the benchmark:
        # many short samples (fixed costs per sample and tile),
        {"name": "attention-short-many", "kind": "attention", "recipe": "short-many", "tokens": 8192, "lengths": 1004,
         "grads": "bf16", **full},
        # samples of very different lengths,
        {"name": "attention-llama3-8b", "kind": "attention", "recipe": "llama3-8b", "tokens": 16384, "lengths": 1001,
         "grads": "bf16", **full},
        # and the largest pack (the benchmark's default).
        {"name": "attention-multi-turn", "kind": "attention", "recipe": "multi-turn", "tokens": 32768, "lengths": 1003,
         "grads": "bf16", **full},
        # Head size 64 without grouping, gradients kept in fp32 for accumulation over micro-batches.
        {"name": "attention-d64-f32-grads", "kind": "attention", "recipe": "llama3-8b", "tokens": 8192, "lengths": 7,
         "grads": "f32", "heads": 16, "kv_heads": 16, "head_dim": 64},
        # One long sample and a quarter of the heads: the share of a GPU whose heads are split over four.
        {"name": "attention-one-long-sample", "kind": "attention", "recipe": "one-sample", "tokens": 16700, "lengths": 3,
         "grads": "bf16", "heads": 8, "kv_heads": 2, "head_dim": 128},
        # The frozen reference model: forward only, then the log-probs; long prompts, few scored rows.
        {"name": "reference-long-prompt", "kind": "reference", "recipe": "long-prompt", "tokens": 16384, "lengths": 1002,
         "vocab": 128256, "dtype": "bf16", **full},
        # Log-probs, loss and the gradient into the logits of a whole pack at a large vocabulary.
        {"name": "loss-llama3-8b", "kind": "loss", "recipe": "llama3-8b", "tokens": 16384, "lengths": 1001, "vocab": 128256,
         "dtype": "bf16", "loss": "dpo"},
        # The same in fp32 with a vocabulary that fills no vector: rows padded to the next 16 bytes.
        {"name": "loss-f32-ragged-vocab", "kind": "loss", "recipe": "short-many", "tokens": 4096, "lengths": 21,
         "vocab": 50257, "dtype": "f32", "loss": "simpo"},
        # A whole attention layer, projections and rotary embedding included, forward and backward.
        {"name": "layer-llama3-8b", "kind": "layer", "recipe": "llama3-8b", "tokens": 16384, "lengths": 1001, **full},
        # Inputs and results in pinned host memory: copies in, forward, backward, copies out.
        {"name": "host-short-many", "kind": "host", "recipe": "short-many", "tokens": 8192, "lengths": 1004, **full},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("attention", "attention", "attention", "attention", "step", "reference", "loss", "loss", "layer", "host"))
    recipe = rng.choice(("llama3-8b", "long-prompt", "multi-turn", "short-many", "one-sample"))
    top = {"attention": 32768, "step": 4096, "reference": 16384, "loss": 12288, "layer": 8192, "host": 8192}[kind]
    case = {"kind": kind, "recipe": recipe, "lengths": rng.randrange(1 << 20)}
    hq, hkv, d = rng.choice(HEADS)
    if recipe == "one-sample":   # the work grows with the square of the length
        top = min(top, 16700)
        hq, hkv, d = rng.choice(((8, 2, 128), (4, 4, 64), (8, 2, 64)))
    case["tokens"] = _log_uniform(rng, 256, top)
    if kind != "loss":
        case.update(heads=hq, kv_heads=hkv, head_dim=d)
    if kind in ("step", "reference", "loss"):
        case["dtype"] = rng.choice(("f32", "bf16", "bf16"))
        most = 128256 if kind != "step" else 32768
        case["vocab"] = min(_log_uniform(rng, 1000, most), (1 << 31) // case["tokens"])
    if kind in ("step", "loss"):
        case["loss"] = rng.choice(("dpo", "simpo", "orpo"))
    if kind == "attention":
        case["grads"] = rng.choice(("bf16", "bf16", "f32"))
    return case


def _pack(case):
    """The pack's sample lengths: drawn from the recipe until one does not fit."""
    hq, hkv, d = case.get("heads", 1), case.get("kv_heads", 1), case.get("head_dim", 64)
    tokens = case["tokens"]
    if case["recipe"] == "tiny":
        tiny = wl.config_pack(0)
        lengths = list(zip(tiny.prefix_len, tiny.chosen_len, tiny.rejected_len))
    elif case["recipe"] == "one-sample":
        rng = np.random.default_rng(case["lengths"])
        c, r = (max(1, int(tokens * rng.uniform(0.02, 0.08))) for _ in range(2))
        lengths = [(tokens - c - r, c, r)]
    else:
        lengths, used = [], 0
        for p, c, r in wl.sample_lengths(RECIPES[case["recipe"]], 400, case["lengths"])[0]:
            if used + p + c + r > tokens:
                if lengths:
                    break
                if tokens > 8 * 64:   # nothing placed yet: a sample that does fit comes later
                    continue
                p, c, r = tokens // 2, tokens // 4, tokens // 4
            lengths.append((p, c, r))
            used += p + c + r
        if not lengths:               # a pack shorter than any sample of the recipe holds one cut-down sample
            lengths = [(tokens - 2 * (tokens // 8), tokens // 8, tokens // 8)]
    return wl.pack_from_lengths(case["recipe"], lengths, hq, hkv, d, tokens)


def _normal(gen, *shape, std=1.0):
    return (torch.randn(shape, generator=gen, device="cuda") * std).to(torch.bfloat16)


def _device(a):
    return torch.as_tensor(np.asarray(a, dtype=np.int32)).cuda()


def _lengths_of(pack):
    return pack.cu_seqlens, pack.prefix_len, pack.chosen_len, pack.rejected_len


def _attention_state(s, gen, grads="bf16"):
    pack = s["pack"]
    T, hq, hkv, d = pack.total_tokens, pack.n_q_heads, pack.n_kv_heads, pack.head_dim
    s["plan"] = psa.psa_plan(*_lengths_of(pack), hq, hkv, d)
    s["q"], s["k"], s["v"] = _normal(gen, T, hq, d), _normal(gen, T, hkv, d), _normal(gen, T, hkv, d)
    s["d_o"] = _normal(gen, T, hq, d)
    s["o"] = torch.empty_like(s["q"])
    s["lse"] = torch.empty((hq, T), dtype=torch.float32, device="cuda")
    dtype = torch.float32 if grads == "f32" else torch.bfloat16
    s["grads"] = [torch.empty(s[n].shape, dtype=dtype, device="cuda") for n in ("q", "k", "v")]
    s["workspace"] = torch.empty(max(s["plan"].bwd_workspace_bytes, 256), dtype=torch.uint8, device="cuda")


def _logits_state(s, gen, case, backward):
    pack, vocab = s["pack"], case["vocab"]
    T, n = pack.total_tokens, pack.n_samples
    dtype = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
    stride = (vocab + 7) // 8 * 8          # rows start on 16 bytes
    logits = torch.empty((T, stride), dtype=dtype, device="cuda")
    for lo in range(0, T, 2048):
        hi = min(T, lo + 2048)
        logits[lo:hi] = (torch.randn((hi - lo, stride), generator=gen, device="cuda") * 3.0 ** 0.5).to(dtype)
    s["logits"] = logits[:, :vocab]
    tokens = torch.randint(0, vocab, (T,), generator=gen, device="cuda", dtype=torch.int32).cpu().numpy()
    targets, segments, *forks = psa.logp_labels(tokens, *_lengths_of(pack))
    s["targets"], s["segments"], s["n_segments"] = _device(targets), _device(segments), 2 * n
    s["forks"] = [_device(f) for f in forks]
    if backward:
        scored = np.bincount(segments[segments >= 0], minlength=2 * n) + np.bincount(forks[2], minlength=2 * n)
        s["scored"] = _device(np.maximum(scored, 1))
        # the reference model's log-probs of the same responses: near the policy's, about -(1.5 + log V) a token
        s["reference"] = -(1.5 + math.log(vocab)) * s["scored"] + 5 * torch.randn(2 * n, generator=gen, device="cuda")
        s["d_logits"] = torch.empty_strided(s["logits"].shape, s["logits"].stride(), dtype=dtype, device="cuda")


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    pack, kind = _pack(case), case["kind"]
    s = {"kind": kind, "pack": pack, "loss": case.get("loss"), "f32": case.get("grads") == "f32"}
    T, hq, hkv, d = pack.total_tokens, pack.n_q_heads, pack.n_kv_heads, pack.head_dim
    if kind in ("attention", "step", "reference"):
        _attention_state(s, gen, case.get("grads", "bf16"))
    if kind in ("step", "loss", "reference"):
        _logits_state(s, gen, case, kind != "reference")
    if kind == "layer":
        hidden = hq * d
        s["layer"] = AttentionLayer(_lengths_of(pack), hq, hkv, d, torch.device("cuda"))
        s["x"], s["d_out"] = _normal(gen, T, hidden), _normal(gen, T, hidden)
        std = hidden ** -0.5
        s["w"] = [_normal(gen, hidden, hq * d, std=std), _normal(gen, hidden, hkv * d, std=std),
                  _normal(gen, hidden, hkv * d, std=std), _normal(gen, hq * d, hidden, std=std)]
    if kind == "host":
        s["plan"] = psa.psa_plan(*_lengths_of(pack), hq, hkv, d)
        host = lambda *shape, dtype=torch.bfloat16: torch.empty(shape, dtype=dtype, pin_memory=True)  # noqa: E731
        s["in"] = [host(T, h, d) for h in (hq, hkv, hkv, hq)]
        for t in s["in"]:
            t.copy_(_normal(gen, *t.shape))
        s["out"] = [host(T, hq, d), host(hq, T, dtype=torch.float32), host(T, hq, d), host(T, hkv, d), host(T, hkv, d)]
        s["arena"] = torch.empty(psa.psa_step_host_arena_bytes(s["plan"]), dtype=torch.uint8, device="cuda")
    return s


def _run_loss(s):
    logps = psa.dpo_logp(s["logits"], s["targets"], s["segments"], s["n_segments"], *s["forks"])
    if s["loss"] == "dpo":
        loss, coef = psa.dpo_loss(logps, s["reference"], 0.1)
    elif s["loss"] == "simpo":
        loss, coef = psa.simpo_loss(logps, s["scored"], 2.0, 0.5)
    else:
        loss, coef = psa.orpo_loss(logps, s["scored"], 0.1)
    psa.dpo_logp_bwd(s["logits"], s["targets"], s["segments"], coef, *s["forks"], dlogits=s["d_logits"])
    return [logps, loss, coef, s["d_logits"]]


def run(s):
    kind = s["kind"]
    if kind == "loss":
        return _run_loss(s)
    if kind == "layer":
        out, saved = s["layer"].forward(s["x"], *s["w"])
        return [out, *s["layer"].backward(s["x"], *s["w"], saved, s["d_out"])]
    if kind == "host":
        psa.psa_step_host(s["plan"], *s["in"], *s["out"], s["arena"])
        return s["out"]
    plan, pack = s["plan"], s["pack"]
    if kind == "step":   # one plan per step
        plan = psa.psa_plan(*_lengths_of(pack), pack.n_q_heads, pack.n_kv_heads, pack.head_dim)
    psa.psa_fwd(plan, s["q"], s["k"], s["v"], o=s["o"], lse=s["lse"])
    if kind == "reference":
        return [s["o"], s["lse"], psa.dpo_logp(s["logits"], s["targets"], s["segments"], s["n_segments"], *s["forks"])]
    outs = [s["o"], s["lse"]]
    if kind == "step":
        outs += _run_loss(s)
    backward = psa.psa_bwd_f32 if s["f32"] else psa.psa_bwd
    dq, dk, dv = s["grads"]
    backward(plan, s["d_o"], s["q"], s["k"], s["v"], s["o"], s["lse"], dq=dq, dk=dk, dv=dv, workspace=s["workspace"])
    return outs + s["grads"]


def work(case):
    """Bytes of every input read once and every output written once; flops of the unmasked pairs and the projections."""
    pack, kind = _pack(case), case["kind"]
    T, hq, hkv, d = pack.total_tokens, pack.n_q_heads, pack.n_kv_heads, pack.head_dim
    P, C, R = (x.astype(np.int64) for x in (pack.prefix_len, pack.chosen_len, pack.rejected_len))
    pairs = int(((P + C) * (P + C + 1) // 2 + R * P + R * (R + 1) // 2).sum())
    bytes_, flops = 0, 0
    if kind != "loss":
        training = kind != "reference"
        flops += (14 if training else 4) * d * hq * pairs
        if kind == "layer":
            hidden = hq * d
            weights = hidden * (2 * hq + 2 * hkv) * d
            flops += 6 * T * weights
            bytes_ += 2 * (4 * T * hidden + 2 * weights)             # x, d_out, out, dx; weights and their gradients
        else:
            out = 4 if case.get("grads") == "f32" else 2
            q, kv = T * hq * d, T * hkv * d
            bytes_ += 2 * (2 * q + 2 * kv) + 4 * hq * T                # q, k, v read, o and lse written
            if training:
                bytes_ += 2 * q + out * (q + 2 * kv)                  # d_o read, dq, dk, dv written
    if kind in ("step", "loss", "reference"):
        row = case["vocab"] * (4 if case["dtype"] == "f32" else 2)
        scored = np.maximum(C - (P == 0), 0) + np.maximum(R - 1, 0)    # rows with a label (the fork row is a chosen row)
        live = int(scored.sum() + ((C == 0) & (R > 0) & (P > 0)).sum())
        bytes_ += live * row
        flops += 4 * live * case["vocab"]
        if kind != "reference":
            bytes_ += T * row                                          # every row of the gradient is written
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    # Four times what the present code differs by from the same path in 64 bits.  bf16 outputs and operands: rel 0.0021,
    # max 0.024 (attention), 0.0055 and 0.14 over the seven roundings of a layer.  The loss in fp32: 6e-5 and 1.8e-4, where
    # the loss's coefficients magnify the last bits of log-probs summed over a long response.
    if case["kind"] == "layer":
        return {"rel": 0.022, "max": 0.55}
    if case["kind"] == "loss" and case["dtype"] == "f32":
        return {"rel": 2.5e-4, "max": 7e-4}
    return {"rel": 8.5e-3, "max": 0.1}


def _exact_attention(pack, q, k, v, d_o=None):
    """o, lse and, where d_o is given, dq, dk, dv in 64 bits: dense masked softmax attention, sample by sample."""
    T, hq, d = q.shape
    g = hq // k.shape[1]
    scale = d ** -0.5
    o, lse = torch.zeros_like(q), torch.zeros((hq, T), dtype=torch.float64, device=q.device)
    dq, dk, dv = (torch.zeros_like(t) for t in (q, k, v))
    for start, P, C, R in zip(pack.cu_seqlens, pack.prefix_len, pack.chosen_len, pack.rejected_len):
        rows = slice(int(start), int(start) + int(P + C + R))
        at = torch.arange(int(P + C + R), device=q.device)
        hidden = (at[None, :] > at[:, None]) | ((at[:, None] >= int(P + C)) & (at[None, :] >= int(P)) & (at[None, :] < int(P + C)))
        for h in range(hq):
            qs, ks, vs = q[rows, h], k[rows, h // g], v[rows, h // g]
            scores = (qs @ ks.t() * scale).masked_fill_(hidden, -math.inf)
            lse[h, rows] = torch.logsumexp(scores, 1)
            p = scores.sub_(lse[h, rows, None]).exp_()
            o[rows, h] = p @ vs
            if d_o is not None:
                g_o = d_o[rows, h]
                dv[rows, h // g] += p.t() @ g_o
                ds = (g_o @ vs.t()).sub_((g_o * o[rows, h]).sum(1, keepdim=True)).mul_(p).mul_(scale)
                dq[rows, h] = ds @ ks
                dk[rows, h // g] += ds.t() @ qs
    return o, lse, dq, dk, dv


def _exact_loss(s, backward):
    """logps and, with `backward`, loss, coef and the gradient of the logits in 64 bits."""
    logits, n = s["logits"], s["n_segments"]
    T, vocab = logits.shape
    rows = torch.arange(T, device="cuda")
    label_rows, label_targets, label_segments = (torch.cat([a, b.long()]) for a, b in (
        (rows, s["forks"][0]), (s["targets"].long(), s["forks"][1]), (s["segments"].long(), s["forks"][2])))
    keep = label_segments >= 0
    label_rows, label_targets, label_segments = label_rows[keep], label_targets[keep], label_segments[keep]
    lse = torch.cat([torch.logsumexp(logits[lo:lo + 512].double(), 1) for lo in range(0, T, 512)])
    logps = torch.zeros(n, dtype=torch.float64, device="cuda")
    logps.index_add_(0, label_segments, logits[label_rows, label_targets].double() - lse[label_rows])
    if not backward:
        return [logps]
    x = logps.clone().requires_grad_()
    if s["loss"] == "dpo":
        z = x - s["reference"].double()
        loss = -torch.nn.functional.logsigmoid(0.1 * (z[0::2] - z[1::2])).mean()
    else:
        mean = x / s["scored"].double()
        if s["loss"] == "simpo":
            loss = -torch.nn.functional.logsigmoid(2.0 * (mean[0::2] - mean[1::2]) - 0.5).mean()
        else:
            odds = mean - torch.log(-torch.expm1(mean))
            loss = (-mean[0::2] - 0.1 * torch.nn.functional.logsigmoid(odds[0::2] - odds[1::2])).mean()
    coef, = torch.autograd.grad(loss, x)
    per_row = torch.zeros(T, dtype=torch.float64, device="cuda").index_add_(0, label_rows, coef[label_segments])
    grad = torch.empty((T, vocab), dtype=torch.float64, device="cuda")
    for lo in range(0, T, 512):
        some = slice(lo, lo + 512)
        grad[some] = (logits[some].double() - lse[some, None]).exp_().mul_(-per_row[some, None])
    grad.index_put_((label_rows, label_targets), coef[label_segments], accumulate=True)
    return [logps, loss.detach()[None], coef, grad]


def _exact_layer(pack, x, w, d_out, d):
    """out, dx and the gradients of the four weights in 64 bits."""
    T = x.shape[0]
    x, d_out, (wq, wk, wv, wo) = x.double(), d_out.double(), [t.double() for t in w]
    at = np.concatenate([np.concatenate([np.arange(P + C), P + np.arange(R)])
                         for P, C, R in zip(pack.prefix_len, pack.chosen_len, pack.rejected_len)])
    half = torch.arange(d // 2, dtype=torch.float64, device="cuda")
    angle = torch.as_tensor(at).double().cuda()[:, None, None] * 10000.0 ** (-2 * half / d)

    def turn(t, sign):
        cos, sin, (a, b) = angle.cos(), angle.sin() * sign, t.split(d // 2, 2)
        return torch.cat([a * cos - b * sin, b * cos + a * sin], 2)

    q, k = turn((x @ wq).view(T, -1, d), 1), turn((x @ wk).view(T, -1, d), 1)
    o, _, dq, dk, dv = _exact_attention(pack, q, k, (x @ wv).view(T, -1, d), (d_out @ wo.t()).view(T, -1, d))
    o, dq, dk, dv = o.view(T, -1), turn(dq, -1).view(T, -1), turn(dk, -1).view(T, -1), dv.view(T, -1)
    dx = dq @ wq.t() + dk @ wk.t() + dv @ wv.t()
    return [o @ wo, dx, x.t() @ dq, x.t() @ dk, x.t() @ dv, o.t() @ d_out]


def exact(case, seed):
    s = prepare(case, seed)
    pack, kind = s["pack"], s["kind"]
    if kind == "loss":
        return _exact_loss(s, True)
    if kind == "layer":
        return _exact_layer(pack, s["x"], s["w"], s["d_out"], pack.head_dim)
    q, k, v, d_o = [t.cuda().double() for t in (s["in"] if kind == "host" else (s["q"], s["k"], s["v"], s["d_o"]))]
    if kind == "reference":
        return [*_exact_attention(pack, q, k, v)[:2], *_exact_loss(s, False)]
    outs = _exact_attention(pack, q, k, v, d_o)
    return [*outs[:2], *(_exact_loss(s, True) if kind == "step" else []), *outs[2:]]
