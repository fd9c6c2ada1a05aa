"""The backward's kernel for long tile lists at head size 128 (statistics touched early), on both sides of its line and with
lists longer than the 128 entries kept in shared memory."""
import pytest
import torch

from paper_2410_20305_b200 import binding as B
from paper_2410_20305_b200 import workloads as wl

from gpu_util import TOL_O, device_plan, read_status

pytestmark = pytest.mark.gpu


def _weighted_mean(plan):
    n = plan.export(1)[0][:, 7].astype(float)
    return (n * n).sum() / n.sum()


def _reference(pack, q, k, v, d_o, lse, rows):
    """fp32 gradients of the first sample, one head at a time."""
    P, C = int(pack.prefix_len[0]), int(pack.chosen_len[0])
    i = torch.arange(rows, device="cuda")
    hidden = (i[None] > i[:, None]) | ((i[:, None] >= P + C) & (i[None] >= P) & (i[None] < P + C))
    for h in range(q.shape[1]):
        x, y, z, g = (t[:rows, h].float() for t in (q, k, v, d_o))
        p = torch.exp((x @ y.T * 128 ** -0.5).masked_fill_(hidden, -torch.inf) - lse[h, :rows, None])
        ds = g @ z.T
        ds = p * (ds - (p * ds).sum(1, keepdim=True)) * 128 ** -0.5
        yield h, ds @ y, ds.T @ x, p.T @ g


@pytest.mark.parametrize("long", [(8100, 40, 52), (16300, 60, 70)])   # 64 tiles: a mean of 43, the line; 129 tiles
def test_long_lists_at_head_size_128(monkeypatch, long):
    monkeypatch.setattr(torch.backends.cuda.matmul, "allow_tf32", False)
    pack = wl.pack_from_lengths("long", [long], 8, 8, 128)
    plan, rows = device_plan(pack), sum(long)
    assert _weighted_mean(plan) >= 43 and plan.launch()[1] == 1
    q, k, v, d_o = (t.cuda() for t in wl.attention_inputs(pack, 12))
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    o, lse = B.psa_fwd(plan, q, k, v, status=status)
    f32 = B.psa_bwd_f32(plan, d_o, q, k, v, o, lse, status=status)
    bf16 = B.psa_bwd(plan, d_o, q, k, v, o, lse, status=status)
    assert read_status(status) == 0
    for a, b in zip(f32[1:], bf16[1:]):
        assert torch.equal(a.to(torch.bfloat16), b)
    for h, *want in _reference(pack, q, k, v, d_o, lse, rows):
        for a, w in zip(f32, want):
            assert (a[:, h] - w).abs().max() <= TOL_O


def test_both_sides_of_the_line_give_the_same_sums():
    long, short = (8100, 40, 52), (100, 10, 10)
    pack = wl.pack_from_lengths("below", [long, short], 8, 8, 128)
    plan = device_plan(pack)
    assert _weighted_mean(plan) < 43 and plan.launch()[1] == 1
    q, k, v, d_o = (t.cuda() for t in wl.attention_inputs(pack, 13))
    o, lse = B.psa_fwd(plan, q, k, v)
    late = B.psa_bwd_f32(plan, d_o, q, k, v, o, lse)
    alone = device_plan(wl.pack_from_lengths("above", [long], 8, 8, 128))
    assert _weighted_mean(alone) >= 43 and alone.launch()[1] == 1
    n = sum(long)
    early = B.psa_bwd_f32(alone, *(t[:n].contiguous() for t in (d_o, q, k, v, o)), lse[:, :n].contiguous())
    assert torch.equal(early[1], late[1][:n]) and torch.equal(early[2], late[2][:n])
    # dq: fp32 adds of 64 partial sums in any order
    assert (early[0] - late[0][:n]).abs().max() <= 64 * 2.0 ** -24 * late[0].abs().max()
