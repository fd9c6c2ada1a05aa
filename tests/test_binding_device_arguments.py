"""Device arguments that a kernel would read or write out of range, or as another type: the binding refuses them before
anything is launched.  Host tensors that say they are on a GPU stand in for device ones."""
import pytest
import torch

from paper_2410_20305_b200 import binding as B


class OnDevice(torch.Tensor):
    is_cuda = property(lambda self: True)


def dev(t):
    return t.as_subclass(OnDevice)


def ints(n, dtype=torch.int32):
    return dev(torch.zeros(n, dtype=dtype))


@pytest.fixture
def reached(monkeypatch):
    """The library, whose calls are written down and not made."""
    calls = []

    class Library:
        def __getattr__(self, name):
            return lambda *a: calls.append(name) or 0
    monkeypatch.setattr(B, "load_library", Library)
    return calls


ROWS, VOCAB = 6, 32
HOST = torch.zeros


def logp_bwd(**change):
    a = dict(logits=dev(torch.zeros(ROWS, VOCAB)), targets=ints(ROWS), segment_ids=ints(ROWS), coef=dev(torch.zeros(2)),
             fork_rows=ints(2), fork_targets=ints(2), fork_segments=ints(2), dlogits=dev(torch.zeros(ROWS, VOCAB)), status=ints(1))
    a.update(change)
    return B.dpo_logp_bwd(stream=0, **a)


def logp(**change):
    a = dict(logits=dev(torch.zeros(ROWS, VOCAB)), targets=ints(ROWS), segment_ids=ints(ROWS), n_segments=2,
             out=dev(torch.zeros(2)), status=ints(1), scratch=dev(torch.zeros(3, dtype=torch.float64)))
    a.update(change)
    return B.dpo_logp(stream=0, **a)


def rope(**change):
    a = dict(x=dev(torch.zeros(ROWS, 2, 64, dtype=torch.bfloat16)), position_ids=ints(ROWS),
             out=dev(torch.zeros(ROWS, 2, 64, dtype=torch.bfloat16)))
    a.update(change)
    return B.psa_rope(stream=0, **a)


def loss(**change):
    a = dict(policy_logps=dev(torch.zeros(4)), ref_logps=dev(torch.zeros(4)), beta=0.1)
    a.update(change)
    return B.dpo_loss(stream=0, **a)


BAD_STATUS = [HOST(1, dtype=torch.int32), dev(torch.zeros(1, dtype=torch.uint8)), dev(torch.zeros(9, dtype=torch.uint8))[1:]]


@pytest.mark.parametrize("call,change", [
    *((logp_bwd, {name: bad}) for name in ("targets", "segment_ids")
      for bad in (ints(ROWS, torch.int64), ints(ROWS - 1), HOST(ROWS, dtype=torch.int32), ints(2 * ROWS)[::2])),
    *((logp_bwd, {name: bad}) for name in ("fork_targets", "fork_segments")
      for bad in (ints(2, torch.int64), ints(1), HOST(2, dtype=torch.int32))),
    (logp_bwd, {"fork_rows": ints(2, torch.int64)}),
    (logp_bwd, {"dlogits": dev(torch.zeros(ROWS - 1, VOCAB))}), (logp_bwd, {"dlogits": HOST(ROWS, VOCAB)}),
    (logp_bwd, {"dlogits": dev(torch.zeros(ROWS, VOCAB))[:, :VOCAB - 1]}),
    (logp, {"out": dev(torch.zeros(1))}), (logp, {"out": HOST(2)}), (logp, {"out": dev(torch.zeros(2, dtype=torch.float64))}),
    (logp, {"out": dev(torch.zeros(4))[::2]}), (logp, {"scratch": dev(torch.zeros(1, dtype=torch.float64)).expand(3)}),
    (rope, {"out": dev(torch.zeros(ROWS - 1, 2, 64, dtype=torch.bfloat16))}), (rope, {"out": dev(torch.zeros(ROWS, 2, 64))}),
    (rope, {"out": HOST(ROWS, 2, 64, dtype=torch.bfloat16)}),
    (rope, {"out": dev(torch.zeros(2, ROWS, 64, dtype=torch.bfloat16)).transpose(0, 1)}),
    (loss, {"ref_logps": HOST(4)}),
    *((call, {"status": bad}) for call in (logp_bwd, logp) for bad in BAD_STATUS),
])
def test_refused_before_the_library_is_reached(reached, call, change):
    with pytest.raises(ValueError):
        call(**change)
    assert reached == []


@pytest.mark.parametrize("call,change", [
    (logp_bwd, {}), (logp, {}), (rope, {}), (loss, {}), (logp_bwd, {"status": None}), (logp, {"status": ints(0)}),
    (logp_bwd, {"targets": ints(ROWS + 3), "dlogits": dev(torch.zeros(ROWS + 1, VOCAB))}),   # room to spare
    (logp_bwd, {"fork_rows": None, "fork_targets": None, "fork_segments": None}),
    (rope, {"out": dev(torch.zeros(ROWS, 128, dtype=torch.bfloat16))}),
    (logp, {"scratch": dev(torch.zeros(24, dtype=torch.uint8))}), (logp, {"status": ints(2, torch.int64)}),
])
def test_still_taken(reached, call, change):
    call(**change)
    assert len(reached) == 1


def test_attention_refuses_a_status_and_a_workspace_that_cannot_be_written(reached):
    plan = object.__new__(B.Plan)
    plan._h = None
    plan.total_tokens, plan.n_q_heads, plan.n_kv_heads, plan.head_dim, plan.bwd_workspace_bytes = 4, 2, 1, 64, 64
    q, k = (dev(torch.zeros(4, h, 64, dtype=torch.bfloat16)) for h in (2, 1))
    lse, ws = dev(torch.zeros(2, 4)), dev(torch.zeros(64, dtype=torch.uint8))
    f32 = [dev(torch.zeros(t.shape)) for t in (q, k, k)]
    calls = [lambda **a: B.psa_fwd(plan, q, k, k, o=q, lse=lse, stream=0, **a),
             lambda workspace=ws, **a: B.psa_bwd(plan, q, q, k, k, q, lse, q, k, k, workspace=workspace, stream=0, **a),
             lambda workspace=ws, **a: B.psa_bwd_f32(plan, q, q, k, k, q, lse, *f32, workspace=workspace, stream=0, **a),
             lambda **a: B.psa_bwd_static_scratch(plan, q, q, k, k, q, lse, q, k, k, stream=0, **a)]
    for call in calls:
        for bad in BAD_STATUS:
            with pytest.raises(ValueError):
                call(status=bad)
    for call in calls[1:3]:
        with pytest.raises(ValueError):
            call(workspace=dev(torch.zeros(1, dtype=torch.uint8)).expand(64))
    assert reached == []
    for call in calls:
        call()
    assert len(reached) == 4
