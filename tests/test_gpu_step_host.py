"""psa_step_host (host buffers in, host buffers out) against psa_fwd + psa_bwd on device
tensors, and against the fp64 oracle."""
import numpy as np
import pytest
import torch

from paper_2410_20305_b200 import binding as B
from paper_2410_20305_b200 import workloads as wl

from gpu_util import TOL_LSE, TOL_O, device_plan, grad_errors, max_abs, oracle_bwd, oracle_fwd, read_status

pytestmark = pytest.mark.gpu


def _host_step(pack, seed, pinned):
    q, k, v, d_o = wl.attention_inputs(pack, seed)
    plan = device_plan(pack, 0.0)
    host = lambda t: t.pin_memory() if pinned else t.clone()
    hq, hk, hv, hdo = host(q), host(k), host(v), host(d_o)
    T, Hq = pack.total_tokens, pack.n_q_heads
    h_o, h_dq = host(torch.zeros_like(q)), host(torch.zeros_like(q))
    h_dk, h_dv = host(torch.zeros_like(k)), host(torch.zeros_like(k))
    h_lse = host(torch.zeros((Hq, T), dtype=torch.float32))
    n = B.psa_step_host_arena_bytes(plan)
    assert n >= 4 * q.numel() * 2 + 4 * k.numel() * 2 + plan.bwd_workspace_bytes
    arena = torch.empty(n, dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    stream = torch.cuda.Stream()
    B.psa_step_host(plan, hq, hk, hv, hdo, h_o, h_lse, h_dq, h_dk, h_dv, arena, status=status,
                    stream=stream.cuda_stream)
    stream.synchronize()
    assert read_status(status) == 0
    return plan, (q, k, v, d_o), (h_o, h_lse, h_dq, h_dk, h_dv)


@pytest.mark.parametrize("pinned", [True, False])
def test_step_host_matches_device_calls_and_oracle(pinned):
    pack = wl.random_pack(5, 3, 300, 4, 2, 128)
    plan, (q, k, v, d_o), (h_o, h_lse, h_dq, h_dk, h_dv) = _host_step(pack, 3, pinned)
    dq_, dk_, dv_, do_ = q.cuda(), k.cuda(), v.cuda(), d_o.cuda()
    o, lse = B.psa_fwd(plan, dq_, dk_, dv_)
    gq, gk, gv = B.psa_bwd(plan, do_, dq_, dk_, dv_, o, lse)
    torch.cuda.synchronize()
    # same kernels on the same data: everything with a fixed summation order is bit-identical
    assert torch.equal(h_o, o.cpu()) and torch.equal(h_lse, lse.cpu())
    assert torch.equal(h_dk, gk.cpu()) and torch.equal(h_dv, gv.cpu())
    # dq is summed over key tiles with unordered fp32 adds before its rounding to bf16
    assert max_abs(h_dq, gq.float().cpu().numpy().astype(np.float64)) <= 0.0625
    ro, rl = oracle_fwd(pack, q, k, v, None)
    assert max_abs(h_o, ro) <= TOL_O and max_abs(h_lse, rl) <= TOL_LSE
    rdq, rdk, rdv = oracle_bwd(pack, q, k, v, d_o, None)
    for got, ref in ((h_dq, rdq), (h_dk, rdk), (h_dv, rdv)):
        _, raw_small, excess = grad_errors(got, ref)   # the gate of the psa_bwd parity tests
        assert raw_small <= TOL_O and excess <= TOL_O, (raw_small, excess)


def test_step_host_rejects_small_arena_and_null():
    pack = wl.config_pack(0)
    plan = device_plan(pack, 0.0)
    q, k, v, d_o = wl.attention_inputs(pack, 0)
    T, Hq = pack.total_tokens, pack.n_q_heads
    outs = [torch.zeros_like(q), torch.zeros((Hq, T), dtype=torch.float32), torch.zeros_like(q),
            torch.zeros_like(k), torch.zeros_like(k)]
    small = torch.empty(B.psa_step_host_arena_bytes(plan) - 256, dtype=torch.uint8, device="cuda")
    with pytest.raises(B.PsaError) as e:
        B.psa_step_host(plan, q, k, v, d_o, *outs, small)
    assert e.value.code == 1


@pytest.mark.parametrize("lengths,heads", [
    ([(90, 40, 55), (0, 30, 29), (200, 129, 127), (0, 0, 1), (64, 64, 64), (5, 300, 20), (2, 150, 190)] * 2, (32, 8, 64)),
    ([(700, 80, 90)], (32, 8, 128)),             # one sample: one part
    ([(1, 1, 0), (1400, 30, 40), (3, 0, 2)], (16, 16, 128))])
def test_step_host_in_parts_equals_the_device_calls(lengths, heads):
    # packs of more than 2 MB of q go in parts; two calls in a row on two streams share the plan's copy streams
    pack = wl.pack_from_lengths("parts", lengths, *heads)
    assert pack.total_tokens * heads[0] * heads[2] * 2 > 2 << 20
    plan = device_plan(pack)
    sets = []
    for seed in (7, 8):
        t = [x.pin_memory() for x in wl.attention_inputs(pack, seed)]
        q, k = t[0], t[1]
        out = [torch.zeros_like(q).pin_memory(), torch.zeros((heads[0], pack.total_tokens)).pin_memory(),
               torch.zeros_like(q).pin_memory(), torch.zeros_like(k).pin_memory(), torch.zeros_like(k).pin_memory()]
        sets.append((t, out, torch.full((B.psa_step_host_arena_bytes(plan),), 0xff, dtype=torch.uint8, device="cuda"),
                     torch.cuda.Stream()))   # (0xff: every float in it is NaN)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    for t, out, arena, stream in sets:
        B.psa_step_host(plan, *t, *out, arena, status=status, stream=stream.cuda_stream)
    for t, out, arena, stream in sets:
        stream.synchronize()
    assert read_status(status) == 0
    for t, out, arena, stream in sets:
        q, k, v, d_o = (x.cuda() for x in t)
        o, lse = B.psa_fwd(plan, q, k, v)
        grads = B.psa_bwd(plan, d_o, q, k, v, o, lse)
        assert torch.equal(out[0], o.cpu()) and torch.equal(out[1], lse.cpu())
        assert torch.equal(out[3], grads[1].cpu()) and torch.equal(out[4], grads[2].cpu())
        want = grads[0].cpu().double()          # dq: unordered fp32 adds, rounded to bf16
        assert ((out[2].double() - want).abs() <= 2.0 ** -7 * want.abs() + 1e-4).all()


def _host_set(pack, seed, plan, pinned=True):
    place = lambda x: x.pin_memory() if pinned else x.clone()  # noqa: E731
    t = [place(x) for x in wl.attention_inputs(pack, seed)]
    q, k = t[0], t[1]
    out = [place(x) for x in (torch.zeros_like(q), torch.zeros((q.shape[1], q.shape[0])), torch.zeros_like(q),
                              torch.zeros_like(k), torch.zeros_like(k))]
    return t, out, torch.empty(B.psa_step_host_arena_bytes(plan), dtype=torch.uint8, device="cuda")


def _same_as_device_calls(plan, t, out):
    q, k, v, d_o = (x.cuda() for x in t)
    o, lse = B.psa_fwd(plan, q, k, v)
    grads = B.psa_bwd(plan, d_o, q, k, v, o, lse)
    assert torch.equal(out[0], o.cpu()) and torch.equal(out[1], lse.cpu())
    assert torch.equal(out[3], grads[1].cpu()) and torch.equal(out[4], grads[2].cpu())
    want = grads[0].cpu().double()          # dq: unordered fp32 adds, rounded to bf16
    assert ((out[2].double() - want).abs() <= 2.0 ** -7 * want.abs() + 1e-4).all()


PARTS = wl.pack_from_lengths("parts", [(700, 80, 90), (300, 200, 100), (50, 60, 70)] * 2, 32, 8, 64)


def test_a_call_does_not_wait_for_another_stream():
    """The first call's stream is busy; a second call of the same plan, and one of another plan, on idle streams come
    back before that stream has got to the first."""
    plans = [device_plan(PARTS), device_plan(PARTS)]
    sets = [_host_set(PARTS, seed, plans[0]) for seed in (1, 2, 3, 4)]
    busy, idle, third = (torch.cuda.Stream() for _ in range(3))
    a = torch.randn((8192, 8192), device="cuda", dtype=torch.bfloat16)
    b = torch.empty_like(a)
    for plan, stream, (t, out, arena) in ((plans[0], idle, sets[1]), (plans[1], third, sets[2])):   # (once, as warm-up)
        B.psa_step_host(plan, *t, *out, arena, stream=stream.cuda_stream)
    torch.cuda.synchronize()
    with torch.cuda.stream(busy):
        for _ in range(400):
            torch.mm(a, a, out=b)
        passed = torch.cuda.Event()
        passed.record()
    for plan, stream, (t, out, arena) in ((plans[0], busy, sets[0]), (plans[0], idle, sets[1]), (plans[1], third, sets[2]),
                                          (plans[0], idle, sets[3])):
        B.psa_step_host(plan, *t, *out, arena, stream=stream.cuda_stream)
    idle.synchronize()
    third.synchronize()
    assert not passed.query()
    torch.cuda.synchronize()
    for t, out, _ in sets:
        _same_as_device_calls(plans[0], t, out)


def test_many_streams_and_plans_at_once():
    plans = [device_plan(PARTS) for _ in range(3)]
    sets = [_host_set(PARTS, seed, plans[0]) for seed in range(4)]
    streams = [torch.cuda.Stream() for _ in range(4)]
    torch.cuda.synchronize()
    for i in range(24):
        t, out, arena = sets[i % 4]
        B.psa_step_host(plans[i % 3], *t, *out, arena, stream=streams[i % 4].cuda_stream)
    torch.cuda.synchronize()
    for t, out, _ in sets:
        _same_as_device_calls(plans[0], t, out)


@pytest.mark.parametrize("lengths,heads", [([(700, 80, 90), (300, 200, 100), (50, 60, 70)] * 2, (32, 8, 64)),
                                           ([(900, 100, 100)], (16, 16, 128))])
def test_pageable_host_buffers_in_parts(lengths, heads):
    pack = wl.pack_from_lengths("parts", lengths, *heads)
    assert pack.total_tokens * heads[0] * heads[2] * 2 > 2 << 20
    plan = device_plan(pack)
    t, out, arena = _host_set(pack, 5, plan, pinned=False)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    B.psa_step_host(plan, *t, *out, arena, stream=stream.cuda_stream)
    stream.synchronize()
    _same_as_device_calls(plan, t, out)


def test_a_captured_call_is_replayed_with_new_inputs():
    """A call on a capturing stream uses that stream alone; each replay copies what the host buffers then hold."""
    plan = device_plan(PARTS)
    t, out, arena = _host_set(PARTS, 6, plan)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    B.psa_step_host(plan, *t, *out, arena, stream=stream.cuda_stream)   # (the plan has been used on the stream before)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        B.psa_step_host(plan, *t, *out, arena)
    for seed in (7, 8):
        for x, y in zip(t, wl.attention_inputs(PARTS, seed)):
            x.copy_(y)
        for x in out:
            x.zero_()
        graph.replay()
        torch.cuda.synchronize()
        _same_as_device_calls(plan, t, out)
