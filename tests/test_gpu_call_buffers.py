"""Buffers that the binding allocates for one call: they belong to the stream that the call runs on, so neither
another stream's tensors nor a call on another stream get them while the call's kernels still use them."""
import numpy as np
import pytest
import torch

from oracle import psa_oracle as orc
from paper_2410_20305_b200 import binding as B
from paper_2410_20305_b200 import workloads as wl

from gpu_util import device_plan, max_abs, read_status

pytestmark = pytest.mark.gpu


class _Recorder:
    """The library, with the arguments of one entry point's calls written down."""

    def __init__(self, name):
        self._lib, self._name, self.calls = B.load_library(), name, []

    def __getattr__(self, name):
        fn = getattr(self._lib, name)
        if name != self._name:
            return fn
        return lambda *a: (self.calls.append(a), fn(*a))[1]


def _blocks_of(bytes_, n=16):
    """Addresses that the current stream's next tensors of this size get."""
    return [t.data_ptr() for t in [torch.empty(bytes_, dtype=torch.uint8, device="cuda") for _ in range(n)]]


def _device(a):
    return torch.as_tensor(np.asarray(a, dtype=np.int32)).cuda()


def _logp_inputs(rows, vocab, n_segments, seed):
    x, _ = wl.logits_and_tokens(rows, vocab, seed, 3.0 ** 0.5, torch.bfloat16)
    rng = np.random.default_rng(seed)
    targets = rng.integers(0, vocab, rows).astype(np.int32)
    seg = np.where(np.arange(rows) % 5 == 0, -1, rng.integers(0, n_segments, rows)).astype(np.int32)
    return (x.cuda(), _device(targets), _device(seg), n_segments), orc.dpo_logp(wl.to_f64(x), targets, seg, n_segments, [], [], [])


def test_dpo_logp_on_a_stream_that_is_not_current(monkeypatch):
    args, want = _logp_inputs(300, 1024, 6, 1)
    rec = _Recorder("dpo_logp_f64sum")
    monkeypatch.setattr(B, "load_library", lambda: rec)
    side = torch.cuda.Stream()
    a = torch.randn((4096, 4096), device="cuda", dtype=torch.bfloat16)
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        for _ in range(40):
            a @ a                                      # the side stream is busy while the call returns
    out = torch.zeros(6, device="cuda")
    torch.cuda.current_stream().synchronize()
    B.dpo_logp(*args, out=out, stream=side.cuda_stream)
    assert rec.calls[-1][13] not in _blocks_of(8 * 7)
    side.synchronize()
    assert np.abs(out.cpu().double().numpy() - want).max() <= 1e-4 * np.abs(want).max()


def test_dpo_logp_on_two_streams_at_once():
    # policy and reference logits; many calls, so that they overlap
    sets = [_logp_inputs(700, 2048, 6, seed) for seed in (2, 3)]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    torch.cuda.synchronize()
    outs = [[torch.zeros(6, device="cuda") for _ in range(50)] for _ in sets]
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    for i in range(50):
        for (args, _), stream, out in zip(sets, streams, outs):
            B.dpo_logp(*args, out=out[i], status=status, stream=stream.cuda_stream)
    assert read_status(status) == 0
    for (_, want), out in zip(sets, outs):
        got = torch.stack(out).cpu().double().numpy()
        assert np.abs(got - want).max() <= 1e-4 * np.abs(want).max()


def test_dpo_logp_scratch_of_the_caller(monkeypatch):
    args, want = _logp_inputs(300, 1024, 6, 4)
    rec = _Recorder("dpo_logp_f64sum")
    monkeypatch.setattr(B, "load_library", lambda: rec)
    scratch = torch.full((7,), float("nan"), dtype=torch.float64, device="cuda")   # contents on entry do not matter
    got = B.dpo_logp(*args, scratch=scratch).cpu().double().numpy()
    assert rec.calls[-1][13] == scratch.data_ptr()
    assert np.abs(got - want).max() <= 1e-4 * np.abs(want).max()
    for small in (scratch[:6], torch.zeros(7, dtype=torch.float64)):
        with pytest.raises(ValueError):
            B.dpo_logp(*args, scratch=small)


@pytest.mark.parametrize("n_segments", [-1, -2, -100])
def test_a_negative_number_of_responses_is_refused_by_the_library(n_segments):
    (x, targets, seg, _), _ = _logp_inputs(8, 64, 2, 5)
    with pytest.raises(B.PsaError) as e:
        B.dpo_logp(x, targets, seg, n_segments, out=torch.zeros(2, device="cuda"))
    assert e.value.code == 1


@pytest.mark.parametrize("name,at", [("psa_bwd", 10), ("psa_bwd_f32", 10)])
def test_backward_workspace_on_a_stream_that_is_not_current(monkeypatch, name, at):
    pack = wl.random_pack(6, 3, 300, 4, 2, 64)
    plan = device_plan(pack)
    q, k, v, d_o = (t.cuda() for t in wl.attention_inputs(pack, 2))
    o, lse = B.psa_fwd(plan, q, k, v)
    grads = [torch.zeros(t.shape, dtype=torch.float32 if name.endswith("f32") else t.dtype, device="cuda") for t in (q, k, v)]
    want = getattr(B, name)(plan, d_o, q, k, v, o, lse)
    rec = _Recorder(name)
    monkeypatch.setattr(B, "load_library", lambda: rec)
    side = torch.cuda.Stream()
    a = torch.randn((4096, 4096), device="cuda", dtype=torch.bfloat16)
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        for _ in range(40):
            a @ a                                      # the side stream is busy while the call returns
    torch.cuda.current_stream().synchronize()
    getattr(B, name)(plan, d_o, q, k, v, o, lse, *grads, stream=side.cuda_stream)
    assert rec.calls[-1][at] not in _blocks_of(plan.bwd_workspace_bytes, 4)
    side.synchronize()
    assert torch.equal(grads[1], want[1]) and torch.equal(grads[2], want[2])
    # dq: unordered fp32 adds, rounded to bf16
    assert max_abs(grads[0], want[0].cpu().double().numpy()) <= 0.0625


@pytest.mark.parametrize("compiled", [True, False])
def test_what_a_call_allocates_belongs_to_the_current_stream(monkeypatch, compiled):
    """Sums, log-probs, loss and coefficients of a call while a side stream is current: what the main stream allocates and
    writes meanwhile shares no memory with them."""
    args, want = _logp_inputs(300, 1024, 6, 6)
    assert B.load_library() and B._native is not None
    if not compiled:
        monkeypatch.setattr(B, "_native", None)
    ref = torch.zeros(6, device="cuda")
    side = torch.cuda.Stream()
    a = torch.randn((4096, 4096), device="cuda", dtype=torch.bfloat16)
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        for _ in range(40):
            a @ a                                      # the side stream is busy while the calls return
        got = B.dpo_logp(*args)
        loss, coef = B.dpo_loss(got, ref, 0.1)
    held = [torch.full((n,), float("nan"), dtype=t, device="cuda") for n in (1, 6, 7) for t in (torch.float32, torch.float64)
            for _ in range(16)]
    torch.cuda.current_stream().synchronize()
    side.synchronize()
    assert np.abs(got.cpu().double().numpy() - want).max() <= 1e-4 * np.abs(want).max()
    # (of the log-probs as they came: fp32 differences of values of up to 500 times 0.1, 2^-23 500 0.1 = 6e-6 in the exponent)
    want_loss, want_coef = orc.dpo_loss(got.cpu().double().numpy(), np.zeros(6), 0.1)
    assert abs(loss.item() - want_loss) <= 1e-4 * abs(want_loss)
    assert np.abs(coef.cpu().double().numpy() - want_coef).max() <= 1e-4 * np.abs(want_coef).max()
    assert all(t.isnan().all() for t in held)
