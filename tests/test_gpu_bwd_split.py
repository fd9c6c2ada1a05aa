"""psa_bwd on packs of few (key tile, kv head) pairs, whose iterations are shared by a cluster of 2, 4 or 8 CTAs:
long and short lists (CTAs of the cluster without an iteration), groups of heads, ragged last tiles, both head sizes."""
import pytest
import torch

from paper_2410_20305_b200 import binding as B
from paper_2410_20305_b200 import workloads as wl

from gpu_util import TOL_O, device_plan, grad_errors, max_abs, oracle_bwd, read_status

pytestmark = pytest.mark.gpu

PACKS = [([(200, 120, 116)], 8, 2, 128),                       # lists of 4 to 16 iterations
         ([(130, 60, 1)], 4, 4, 64),                           # lists of 1 and 2: most of the cluster is empty
         ([(300, 100, 100), (1, 1, 1)], 4, 4, 128),
         ([(700, 333, 251)], 8, 2, 64),
         ([(64, 200, 190), (128, 128, 128), (90, 37, 300)], 32, 8, 64)]


@pytest.mark.parametrize("lengths,hq,hkv,d", PACKS)
def test_shared_iterations_match_the_oracle(lengths, hq, hkv, d):
    pack = wl.pack_from_lengths("split", lengths, hq, hkv, d)
    q, k, v, d_o = wl.attention_inputs(pack, 90)
    plan = device_plan(pack)
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
