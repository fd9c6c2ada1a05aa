"""psa_bwd on packs of few (key tile, kv head) pairs, whose iterations are shared by a cluster of 2, 4 or 8 CTAs:
long and short lists (CTAs of the cluster without an iteration), groups of heads, ragged last tiles, both head sizes."""
import pytest
import torch

from paper_2410_20305_b200 import binding as B
from paper_2410_20305_b200 import workloads as wl

from gpu_util import TOL_O, device_plan, grad_errors, max_abs, oracle_bwd, read_status

pytestmark = pytest.mark.gpu

PACKS = [([(200, 120, 116)], 8, 2, 128, 8),                       # lists of 4 to 16 iterations: CTAs without one
         ([(80, 18, 33)], 16, 2, 64, 8),
         ([(300, 100, 100), (1, 1, 1)], 4, 4, 128, 4),            # lists of 1 to 4: most of a cluster is empty
         ([(700, 333, 251)], 8, 2, 64, 4),
         ([(132, 60, 66)], 32, 16, 64, 2),
         ([(130, 93, 37)], 32, 16, 128, 2),
         ([(130, 60, 1)], 4, 4, 64, 1),                           # lists of 1 and 2: not worth sharing
         ([(64, 200, 190), (128, 128, 128), (90, 37, 300)], 32, 8, 64, 1)]


@pytest.mark.parametrize("lengths,hq,hkv,d,ctas", PACKS)
def test_shared_iterations_match_the_oracle(lengths, hq, hkv, d, ctas):
    pack = wl.pack_from_lengths("split", lengths, hq, hkv, d)
    q, k, v, d_o = wl.attention_inputs(pack, 90)
    plan = device_plan(pack)
    assert plan.launch()[1] == ctas
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    qd, kd, vd, dod = q.cuda(), k.cuda(), v.cuda(), d_o.cuda()
    o, lse = B.psa_fwd(plan, qd, kd, vd, status=status)
    canary = torch.full((pack.total_tokens + 2, hkv, d), 7.0, device="cuda")
    f32 = B.psa_bwd_f32(plan, dod, qd, kd, vd, o, lse, dk=canary[:-2], status=status)
    bf16 = B.psa_bwd(plan, dod, qd, kd, vd, o, lse, status=status)
    assert read_status(status) == 0 and (canary[-2:] == 7.0).all()
    for a, b, ref in zip(f32, bf16, oracle_bwd(pack, q, k, v, d_o)):
        assert max_abs(a, ref) <= TOL_O
        _, small, excess = grad_errors(b, ref)
        assert small <= TOL_O and excess <= TOL_O
    again = B.psa_bwd_f32(plan, dod, qd, kd, vd, o, lse)
    assert torch.equal(again[1], f32[1]) and torch.equal(again[2], f32[2])   # dk, dv: a fixed order of sums


def test_two_entry_points_share_iterations_on_two_streams_at_once():
    """psa_bwd and psa_bwd_static_scratch, both with clusters, on two streams: results as when run alone."""
    sets = []
    for lengths, hq, hkv, d, ctas in (PACKS[0], PACKS[3]):
        pack = wl.pack_from_lengths("both", lengths, hq, hkv, d)
        plan = device_plan(pack)
        assert plan.launch()[1] == ctas > 1
        q, k, v, d_o = (t.cuda() for t in wl.attention_inputs(pack, 91))
        o, lse = B.psa_fwd(plan, q, k, v)
        want = B.psa_bwd(plan, d_o, q, k, v, o, lse)
        workspace = torch.empty(plan.bwd_workspace_bytes, dtype=torch.uint8, device="cuda")
        sets.append((plan, (d_o, q, k, v, o, lse), want, [torch.zeros_like(t) for t in (q, k, v)], workspace, torch.cuda.Stream()))
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    for _ in range(20):
        plan, args, _, out, workspace, stream = sets[0]
        B.psa_bwd(plan, *args, *out, workspace=workspace, status=status, stream=stream.cuda_stream)
        plan, args, _, out, _, stream = sets[1]
        B.psa_bwd_static_scratch(plan, *args, *out, status=status, stream=stream.cuda_stream)
    assert read_status(status) == 0
    for _, _, want, out, _, _ in sets:
        assert torch.equal(out[1], want[1]) and torch.equal(out[2], want[2])
        # dq: unordered fp32 adds, rounded to bf16
        assert ((out[0].double() - want[0].double()).abs() <= 2.0 ** -7 * want[0].double().abs() + 1e-4).all()
