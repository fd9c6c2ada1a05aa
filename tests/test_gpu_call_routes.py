"""The binding's compiled route and its ctypes route are one: same results, same refusals.  And launches that start behind
one another (small packs, the loss chain) see what the kernels before them have written."""
import numpy as np
import pytest
import torch

from paper_2410_20305_b200 import binding as B
from paper_2410_20305_b200 import workloads as wl

from gpu_util import device_plan

pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.as_tensor(np.asarray(a, dtype=np.int32)).cuda()


def _inputs(seed, n, longest, heads, dtype, vocab):
    pack = wl.random_pack(seed, n, longest, *heads)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    q, k, v, d_o = (t.cuda() for t in wl.attention_inputs(pack, seed))
    T = pack.total_tokens
    logits = torch.randn((T, (vocab + 7) // 8 * 8), generator=gen, device="cuda").to(dtype)[:, :vocab]
    tok = np.random.default_rng(seed).integers(0, vocab, T).astype(np.int32)
    labels = B.psa_logp_labels(tok, pack.cu_seqlens, pack.prefix_len, pack.chosen_len, pack.rejected_len)
    lengths = np.maximum(np.bincount(labels[1][labels[1] >= 0], minlength=2 * pack.n_samples), 1)
    return pack, (q, k, v, d_o), logits, [_dev(a) for a in labels], _dev(lengths)


def _step(pack, qkv, logits, labels, lengths, f32):
    """Every call of a training step; all outputs."""
    q, k, v, d_o = qkv
    plan = B.psa_plan(pack.cu_seqlens, pack.prefix_len, pack.chosen_len, pack.rejected_len, pack.n_q_heads, pack.n_kv_heads,
                      pack.head_dim)
    ws = torch.empty(plan.bwd_workspace_bytes, dtype=torch.uint8, device="cuda")
    pos = _dev(B.psa_position_ids(pack.cu_seqlens, pack.prefix_len, pack.chosen_len, pack.rejected_len))
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    qr = B.psa_rope(q, pos, 10000.0, out=torch.empty_like(q))
    o, lse = B.psa_fwd(plan, qr, k, v, o=torch.empty_like(q), lse=None, status=status)
    targets, segments, *forks = labels
    lp = B.dpo_logp(logits, targets, segments, 2 * pack.n_samples, *forks, status=status)
    outs = [qr, o, lse, lp]
    for loss, coef in (B.dpo_loss(lp, lp * 1.01, 0.1), B.simpo_loss(lp, lengths, 2.0, 0.5), B.orpo_loss(lp, lengths, 0.1)):
        d = torch.empty_strided(logits.shape, logits.stride(), dtype=logits.dtype, device="cuda")
        outs += [loss, coef, B.dpo_logp_bwd(logits, targets, segments, coef, *forks, dlogits=d, status=status)]
    backward = B.psa_bwd_f32 if f32 else B.psa_bwd
    g = [torch.empty(t.shape, dtype=torch.float32 if f32 else t.dtype, device="cuda") for t in (q, k, v)]
    outs += backward(plan, d_o, qr, k, v, o, lse, *g, workspace=ws, status=status)
    return outs, status


def _same(got, want):
    """Everything the same to the bit, dq apart.  The fp64 sums of the log-probs come in any order, but 1e-16 of a sum tips its
    rounding to fp32 once in 1e9 sums; loss, coefficients and the logits' gradient follow from them in a fixed order."""
    for i, (a, b) in enumerate(zip(got, want)):
        if i == len(want) - 3:
            # fp32 adds of at most 10 partial sums in any order, and for bf16 one rounding of the output more
            biggest = b.float().abs().max().item()
            assert torch.allclose(a.float(), b.float(), rtol=2.0 ** -7 if a.dtype == torch.bfloat16 else 0.0, atol=64 * 2.0 ** -24 * biggest)
        else:
            assert torch.equal(a, b), i


@pytest.mark.parametrize("heads,f32,dtype", [((4, 2, 64), False, torch.bfloat16), ((8, 2, 128), True, torch.float32)])
def test_both_routes_give_the_same_step(monkeypatch, heads, f32, dtype):
    args = _inputs(3, 3, 200, heads, dtype, 1003)
    assert B.load_library() and B._native is not None
    got, status = _step(*args, f32)
    monkeypatch.setattr(B, "_native", None)
    want, other = _step(*args, f32)
    assert int(status.item()) == int(other.item()) == 0
    _same(got, want)


def test_both_routes_refuse_the_same_calls(monkeypatch):
    pack, (q, k, v, d_o), logits, labels, lengths = _inputs(5, 2, 150, (4, 2, 64), torch.bfloat16, 256)
    plan = device_plan(pack)
    o, lse = B.psa_fwd(plan, q, k, v)
    ws = torch.empty(plan.bwd_workspace_bytes, dtype=torch.uint8, device="cuda")
    g = [torch.empty_like(t) for t in (q, k, v)]
    lp = torch.zeros(2 * pack.n_samples, device="cuda")
    flat = q.transpose(0, 1).contiguous().transpose(0, 1)
    calls = [
        lambda: B.psa_fwd(plan, q[:-1], k, v), lambda: B.psa_fwd(plan, q.float(), k, v), lambda: B.psa_fwd(plan, q, k.cpu(), v),
        lambda: B.psa_fwd(plan, flat, k, v), lambda: B.psa_fwd(plan, q, k, v, lse=lse[:, :-1]),
        lambda: B.psa_bwd(plan, d_o, q, k, v, o, lse, *g, workspace=ws[:-1]),
        lambda: B.psa_bwd(plan, d_o, q, k, v, o, lse, *g, workspace=ws.cpu()),
        lambda: B.psa_bwd_f32(plan, d_o, q, k, v, o, lse, *g, workspace=ws),
        lambda: B.psa_plan(pack.cu_seqlens[:-1], pack.prefix_len, pack.chosen_len, pack.rejected_len, 4, 2, 64),
        lambda: B.psa_plan(pack.cu_seqlens + 1, pack.prefix_len, pack.chosen_len, pack.rejected_len, 4, 2, 64),
        lambda: B.psa_plan(pack.cu_seqlens, pack.prefix_len, pack.chosen_len, pack.rejected_len, 4, 3, 64),
        lambda: B.dpo_logp(logits, labels[0][:-1], labels[1], 4), lambda: B.dpo_logp(logits.cpu(), labels[0], labels[1], 4),
        lambda: B.dpo_logp(logits, labels[0].long(), labels[1], 4), lambda: B.dpo_logp(logits, labels[0], labels[1], -1),
        lambda: B.dpo_logp_bwd(logits, labels[0], labels[1], lp.double(), dlogits=torch.empty_like(logits)),
        lambda: B.dpo_logp_bwd(logits, labels[0], labels[1], lp, dlogits=torch.empty_like(logits).float()),
        lambda: B.dpo_loss(lp, lp[:-1], 0.1), lambda: B.simpo_loss(lp, lp, 0.1, 0.2), lambda: B.orpo_loss(lp.double(), lengths, 0.1),
        lambda: B.psa_rope(q.float(), labels[0], out=q), lambda: B.psa_rope(q, labels[0][:-1], out=q),
    ]
    for route in (B._native, None):
        monkeypatch.setattr(B, "_native", route)
        said = []
        for i, call in enumerate(calls):
            with pytest.raises(Exception) as e:
                call()
            said.append((i, type(e.value), str(e.value)))
        if route is not None:
            first = said
    assert said == first
    plan.close()
    with pytest.raises(B.PsaError):
        B.psa_fwd(plan, q, k, v, o=o, lse=lse)


def test_both_routes_refuse_buffers_that_are_too_small_or_elsewhere(monkeypatch):
    pack, (q, k, v, d_o), logits, (targets, segments, *forks), lengths = _inputs(5, 2, 150, (4, 2, 64), torch.bfloat16, 256)
    plan = device_plan(pack)
    o, lse = B.psa_fwd(plan, q, k, v)
    ws = torch.empty(plan.bwd_workspace_bytes, dtype=torch.uint8, device="cuda")
    g = [torch.empty_like(t) for t in (q, k, v)]
    lp, d = torch.zeros(2 * pack.n_samples, device="cuda"), torch.empty_like(logits)
    byte = torch.zeros(8, dtype=torch.uint8, device="cuda")
    bwd = lambda t=targets, s=segments, f=forks, to=d, status=None: B.dpo_logp_bwd(logits, t, s, lp, *f, dlogits=to, status=status)
    calls = [
        lambda: bwd(t=targets.long()), lambda: bwd(t=targets[:-1]), lambda: bwd(s=segments.cpu()), lambda: bwd(s=segments[:-1]),
        lambda: bwd(f=[forks[0], forks[1][:-1], forks[2]]), lambda: bwd(f=[forks[0], forks[1], forks[2].long()]),
        lambda: bwd(to=d[:-1]), lambda: bwd(to=torch.empty(d.shape, dtype=d.dtype)),
        lambda: B.psa_rope(q, targets, out=torch.empty_like(q)[:-1]), lambda: B.psa_rope(q, targets, out=torch.empty_like(q).cpu()),
        lambda: B.dpo_loss(lp, lp.cpu(), 0.1), lambda: B.simpo_loss(lp, lengths.cpu(), 0.1, 0.2),
        lambda: B.psa_bwd(plan, d_o, q, k, v, o, lse, *g, workspace=byte[:1].clone().expand(ws.numel())),
    ]
    for status in (torch.zeros(1, dtype=torch.int32), byte[:1], byte[1:5]):
        calls += [lambda s=status: bwd(status=s), lambda s=status: B.psa_fwd(plan, q, k, v, status=s),
                  lambda s=status: B.dpo_logp(logits, targets, segments, 2 * pack.n_samples, status=s),
                  lambda s=status: B.psa_bwd(plan, d_o, q, k, v, o, lse, *g, workspace=ws, status=s),
                  lambda s=status: B.simpo_loss(lp, lengths, 0.1, 0.2, status=s), lambda s=status: B.orpo_loss(lp, lengths, 0.1, status=s)]
    for route in (B._native, None):
        monkeypatch.setattr(B, "_native", route)
        for call in calls:
            with pytest.raises((ValueError, AssertionError)):
                call()


@pytest.mark.parametrize("seed,n,longest,heads", [(1, 1, 130, (4, 4, 64)), (2, 2, 400, (8, 2, 128)), (4, 3, 90, (4, 2, 64))])
def test_launches_behind_one_another_see_what_came_before(seed, n, longest, heads):
    """Inputs and labels are rewritten on the stream right before every step, and the same buffers are used again."""
    pack, qkv, logits, labels, lengths = _inputs(seed, n, longest, heads, torch.bfloat16, 504)
    variants = [([t * s for t in qkv], logits * s) for s in (1.0, 0.5, -1.0)]
    want = []
    for x, y in variants:
        torch.cuda.synchronize()
        outs, _ = _step(pack, x, y, labels, lengths, False)
        torch.cuda.synchronize()
        want.append([t.clone() for t in outs])
    live_x, live_y = [torch.empty_like(t) for t in qkv], torch.empty_strided(logits.shape, logits.stride(), dtype=logits.dtype,
                                                                          device="cuda")
    torch.cuda.synchronize()
    for turn in range(30):
        x, y = variants[turn % 3]
        for a, b in zip(live_x, x):
            a.copy_(b)
        live_y.copy_(y)
        outs, status = _step(pack, live_x, live_y, labels, lengths, False)
        kept = [t.clone() for t in outs]
        _same(kept, want[turn % 3])
        assert int(status.item()) == 0


@pytest.mark.parametrize("seed,n,longest,heads", [(1, 1, 130, (4, 4, 64)), (2, 2, 400, (8, 2, 128))])
def test_the_chain_captured_in_a_graph_sees_what_came_before(seed, n, longest, heads):
    """Forward, log-probs, loss, logits' gradient and backward as one graph, in which launches behind one another are edges of
    their own kind: replayed on inputs that change right before."""
    pack, qkv, logits, (targets, segments, *forks), _ = _inputs(seed, n, longest, heads, torch.bfloat16, 504)
    plan = device_plan(pack)
    ws = torch.empty(plan.bwd_workspace_bytes, dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    live = [torch.empty_like(t) for t in qkv]
    live_y = torch.empty_strided(logits.shape, logits.stride(), dtype=logits.dtype, device="cuda")
    grads = [torch.empty_like(t) for t in live[:3]]
    d = torch.empty_strided(logits.shape, logits.stride(), dtype=logits.dtype, device="cuda")

    def chain():
        q, k, v, d_o = live
        o, lse = B.psa_fwd(plan, q, k, v, status=status)
        lp = B.dpo_logp(live_y, targets, segments, 2 * pack.n_samples, *forks, status=status)
        loss, coef = B.dpo_loss(lp, torch.zeros_like(lp), 0.1)
        B.dpo_logp_bwd(live_y, targets, segments, coef, *forks, dlogits=d, status=status)
        B.psa_bwd(plan, d_o, q, k, v, o, lse, *grads, workspace=ws, status=status)
        return [o, lse, lp, loss, coef, d, *grads]

    def fill(scale):
        for a, b in zip(live, qkv):
            a.copy_(b * scale)
        live_y.copy_(logits * scale)

    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        want = []
        for scale in (1.0, 0.5, -1.0):
            fill(scale)
            torch.cuda.synchronize()
            want.append([t.clone() for t in chain()])
            torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        outs = chain()
    with torch.cuda.stream(stream):
        for turn in range(30):
            fill((1.0, 0.5, -1.0)[turn % 3])
            for t in outs:
                t.zero_()
            graph.replay()
            kept = [t.clone() for t in outs]
            _same(kept, want[turn % 3])
    assert int(status.item()) == 0
