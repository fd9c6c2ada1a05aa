"""dpo_logp_bwd at the row sizes where it changes its kernel (rows up to 32, 96 and 320 KB, longer), with ragged
ends, rows shorter than one 16-byte vector, labels on the first and the last element, and -inf logits."""
import numpy as np
import pytest
import torch

from oracle import psa_oracle as orc
from paper_2410_20305_b200 import binding as B
from paper_2410_20305_b200 import workloads as wl

from gpu_util import read_status

pytestmark = pytest.mark.gpu

BF16 = (5, 1031, 16384, 16392 + 5, 49152, 49160 + 3, 163840, 163849)      # 32 KB = 16384, 96 KB = 49152, 320 KB = 163840
F32 = (3, 515, 8192, 8196 + 1, 24576, 24580 + 3, 81920, 81925)          # 32 KB = 8192, 96 KB = 24576, 320 KB = 81920


@pytest.mark.parametrize("dtype,vocab", [(torch.bfloat16, v) for v in BF16] + [(torch.float32, v) for v in F32])
def test_gradient_rows_around_the_kernel_limits(dtype, vocab):
    T, stride = 6, (vocab + 7) // 8 * 8
    x, _ = wl.logits_and_tokens(T, stride, vocab, 3.0 ** 0.5, dtype)
    x[2, : vocab // 2] = -float("inf")
    targets = np.array([0, vocab - 1, vocab - 1, vocab // 2, 1, 0], dtype=np.int32)
    seg = np.array([0, 1, 2, -1, 3, -1], dtype=np.int32)
    fr, ft, fs = (np.array(a, dtype=np.int32) for a in ([3, 0], [vocab - 1, 0], [2, 1]))   # row 3 only by its fork
    coef = np.array([0.7, -0.4, 1.0, -0.9], dtype=np.float32)
    dev = lambda a: torch.as_tensor(a).cuda()  # noqa: E731
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    full = torch.full_like(x.cuda(), 7.0)
    B.dpo_logp_bwd(x.cuda()[:, :vocab], dev(targets), dev(seg), dev(coef), dev(fr), dev(ft), dev(fs),
                   dlogits=full[:, :vocab], status=status)
    assert read_status(status) == 0
    x64 = wl.to_f64(x)[:, :vocab]
    with np.errstate(invalid="ignore"):
        want = orc.dpo_logp_grad(x64, targets, seg, coef.astype(np.float64), fr, ft, fs)
    got = full[:, :vocab].cpu().double().numpy()
    # fp32: the log-sum-exp (about 16 in the log2 domain) carries an ulp of 1e-6, which scales every probability <= 1 of
    # the row by as much, times |coef| <= 1; bf16 results add half an ulp (2^-9) of the value.
    tol = 4e-6 + (0 if dtype == torch.float32 else 2.0 ** -8) * np.abs(want)
    assert (np.abs(got - want) <= tol).all(), np.abs(got - want).max()
    assert (got[5] == 0).all() and (full[:, vocab:] == 7.0).all()
