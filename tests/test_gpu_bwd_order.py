"""The orders in which the backward hands out its (key tile, kv head) pairs: longest first at the end, or as a whole."""
import pytest
import torch

from paper_2410_20305_b200 import binding as B
from paper_2410_20305_b200 import workloads as wl

from gpu_util import device_plan, read_status

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lengths,heads", [
    ([(3000, 300, 301), (900, 200, 252)], (8, 8, 128)),             # 2 waves, accumulator in L2: all or half of it sorted
    ([(2600, 500, 200), (1500, 300, 420), (300, 90, 77)], (32, 8, 128)),   # 2.6 waves, 98 MB: the last wave sorted
    ([(1500, 300, 209)], (32, 8, 128)),                             # clusters, more of them than fit at once
    ([(700, 130, 60), (1, 0, 1), (250, 129, 128)], (16, 16, 64)),   # few pairs, one sample of two tokens
])
def test_every_order_gives_each_sample_its_gradients(lengths, heads):
    pack = wl.pack_from_lengths("order", lengths, *heads)
    q, k, v, d_o = (t.cuda() for t in wl.attention_inputs(pack, 7))
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    plan = device_plan(pack)
    o, lse = B.psa_fwd(plan, q, k, v, status=status)
    got = B.psa_bwd_f32(plan, d_o, q, k, v, o, lse, status=status)
    at = 0
    for one in lengths:   # the same sample alone, whose pairs come in another order and number
        rows = slice(at, at + sum(one))
        at += sum(one)
        alone = device_plan(wl.pack_from_lengths("alone", [one], *heads))
        part = [t[rows].contiguous() for t in (q, k, v, d_o, o)]
        want = B.psa_bwd_f32(alone, part[3], *part[:3], part[4], lse[:, rows].contiguous(), status=status)
        for a, b in zip(got, want):
            # fp32 sums of up to 4 x 3601 products in another order: 2^-24 sqrt(14400) = 7e-6 of the largest partial sum
            assert (a[rows] - b).abs().max() <= 1e-4 * b.abs().max()
    assert read_status(status) == 0
