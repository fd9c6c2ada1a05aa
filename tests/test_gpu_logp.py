"""dpo_logp on the GPU against the fp64 oracle."""
import numpy as np
import pytest
import torch

from oracle import psa_oracle as orc
from paper_2410_20305_b200 import binding as B
from paper_2410_20305_b200 import workloads as wl
from paper_2410_20305_b200.labels import logp_labels

from gpu_util import TOL_LOGP, read_status

pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.as_tensor(np.asarray(a, dtype=np.int32)).cuda()


def _run(pack, vocab, seed, std, dtype):
    T = pack.total_tokens
    x, tok = wl.logits_and_tokens(T, vocab, seed, std, dtype)
    targets, seg, fr, ft, fs = logp_labels(tok.numpy(), pack.cu_seqlens, pack.prefix_len, pack.chosen_len,
                                           pack.rejected_len)
    n_seg = 2 * pack.n_samples
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    out = B.dpo_logp(x.cuda(), _dev(targets), _dev(seg), n_seg, _dev(fr), _dev(ft), _dev(fs), status=status)
    assert read_status(status) == 0
    want = orc.dpo_logp(wl.to_f64(x), targets, seg, n_seg, fr, ft, fs)
    got = out.cpu().double().numpy()
    live = np.abs(want) > 0
    assert (got[~live] == 0).all()
    rel = np.abs(got[live] - want[live]) / np.abs(want[live])
    return float(rel.max(initial=0.0))


def test_tiny_config_fp32_logits():
    assert _run(wl.config_pack(0), 1024, 0, 2.0 ** 0.5, torch.float32) <= TOL_LOGP
    assert _run(wl.config_pack(0), 1024, 1, 2.0, torch.float32) <= TOL_LOGP


@pytest.mark.parametrize("vocab", [128256, 32000, 1000, 8, 50257 + 7])
def test_bf16_logits_ragged_vocab(vocab):
    pack = wl.pack_from_lengths("lp", [(20, 9, 13), (0, 5, 4), (7, 0, 3), (3, 4, 0), (1, 1, 1)], 1, 1, 64)
    if vocab % 8:
        # rows must start 16-byte aligned: pad the row stride, keep the vocab ragged
        T = pack.total_tokens
        stride = (vocab + 7) // 8 * 8
        x, tok = wl.logits_and_tokens(T, stride, 3, 3.0 ** 0.5, torch.bfloat16)
        tok = tok % vocab
        targets, seg, fr, ft, fs = logp_labels(tok.numpy(), pack.cu_seqlens, pack.prefix_len, pack.chosen_len,
                                               pack.rejected_len)
        out = B.dpo_logp(x.cuda()[:, :vocab], _dev(targets), _dev(seg), 10, _dev(fr), _dev(ft), _dev(fs))
        want = orc.dpo_logp(wl.to_f64(x)[:, :vocab], targets, seg, 10, fr, ft, fs)
        got = out.cpu().double().numpy()
        live = np.abs(want) > 0
        assert (np.abs(got[live] - want[live]) / np.abs(want[live])).max() <= TOL_LOGP
    else:
        assert _run(pack, vocab, 3, 3.0 ** 0.5, torch.bfloat16) <= TOL_LOGP


def test_plain_gather_without_forks_and_dead_rows():
    x, tok = wl.logits_and_tokens(300, 4096, 5, 1.7, torch.bfloat16)
    seg = np.random.default_rng(1).integers(-1, 7, size=300).astype(np.int32)
    out = B.dpo_logp(x.cuda(), tok.cuda(), _dev(seg), 7)
    want = orc.dpo_logp(wl.to_f64(x), tok.numpy(), seg, 7)
    assert (np.abs(out.cpu().double().numpy() - want) / np.abs(want)).max() <= TOL_LOGP


def test_bad_labels_set_status_bits_and_are_skipped():
    x, tok = wl.logits_and_tokens(6, 64, 5, 1.0, torch.float32)
    targets = np.array([1, 64, 3, -5, 2, 7], dtype=np.int32)      # rows 1 and 3 are out of range
    seg = np.array([0, 0, 1, 1, 9, -1], dtype=np.int32)            # row 4 names a segment >= n_segments
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    out = B.dpo_logp(x.cuda(), _dev(targets), _dev(seg), 2, status=status)
    assert read_status(status) == (B.PSA_DEVSTAT_BAD_TARGET | B.PSA_DEVSTAT_BAD_SEGMENT)
    want = [orc.row_logprob(wl.to_f64(x)[0], 1), orc.row_logprob(wl.to_f64(x)[2], 3)]
    assert np.allclose(out.cpu().numpy(), want, rtol=1e-4)


def test_zero_rows_and_zero_segments():
    x = torch.empty((0, 128), dtype=torch.float32, device="cuda")
    e = torch.empty(0, dtype=torch.int32, device="cuda")
    out = B.dpo_logp(x, e, e, 3)
    assert (out.cpu() == 0).all()


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("vocab", [1, 3, 7, 129])
def test_single_row_of_any_width(vocab, dtype):
    """One row has no stride, so a vocabulary that is not a multiple of 16 bytes is accepted; the
    ragged tail of the row is handled by scalar loads."""
    x, tok = wl.logits_and_tokens(1, vocab, 11, 2.0, dtype)
    seg = np.zeros(1, dtype=np.int32)
    coef = torch.tensor([0.75], dtype=torch.float32, device="cuda")
    out = B.dpo_logp(x.cuda(), tok.cuda(), _dev(seg), 1)
    want = orc.dpo_logp(wl.to_f64(x), tok.numpy(), seg, 1)
    assert abs(out.item() - want[0]) <= TOL_LOGP * max(1.0, abs(want[0]))
    grad = B.dpo_logp_bwd(x.cuda(), tok.cuda(), _dev(seg), coef)
    ref = orc.dpo_logp_grad(wl.to_f64(x), tok.numpy(), seg, [0.75])
    assert np.abs(grad.cpu().double().numpy() - ref).max() <= (2e-6 if dtype == torch.float32 else 2.0 ** -8)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_rows_that_begin_with_a_block_of_minus_infinity(dtype):
    """Banned or padded vocabulary entries are -inf.  A thread whose first chunk of the row is all
    -inf must carry "nothing yet", not a NaN, into the rest of the row; the gradient sweep too."""
    n_rows, vocab = 6, 4096
    x, tok = wl.logits_and_tokens(n_rows, vocab, 21, 2.0, dtype)
    x[0, :1024] = -float("inf")            # every thread's first chunk (and more)
    x[1, :32] = -float("inf")              # exactly one thread's first chunk
    x[2, 100:2100] = -float("inf")         # a block in the middle
    x[3, vocab - 700:] = -float("inf")     # the tail
    x[4, ::2] = -float("inf")              # every other entry
    tok = tok.clone()
    tok[0], tok[1], tok[2], tok[3], tok[4] = 2000, 40, 50, 7, 1
    seg = np.arange(n_rows, dtype=np.int32)
    out = B.dpo_logp(x.cuda(), tok.cuda(), _dev(seg), n_rows)
    want = orc.dpo_logp(wl.to_f64(x), tok.numpy(), seg, n_rows)
    got = out.cpu().double().numpy()
    assert np.isfinite(got).all()
    assert (np.abs(got - want) / np.abs(want)).max() <= TOL_LOGP
    coef = torch.linspace(0.1, 0.6, n_rows, dtype=torch.float32).cuda()
    grad = B.dpo_logp_bwd(x.cuda(), tok.cuda(), _dev(seg), coef).cpu().double().numpy()
    ref = orc.dpo_logp_grad(wl.to_f64(x), tok.numpy(), seg, coef.cpu().double().numpy())
    assert np.isfinite(grad).all()
    assert np.abs(grad - ref).max() <= (2e-6 if dtype == torch.float32 else 2.0 ** -8)


@pytest.mark.parametrize("dtype,vocab,rows", [(torch.float32, 3, 4000), (torch.bfloat16, 515, 3000), (torch.bfloat16, 4096 + 8, 1500),
                                              (torch.float32, 32768, 1024), (torch.float32, 32768, 1025), (torch.float32, 16383, 300),
                                              (torch.bfloat16, 65535, 500), (torch.bfloat16, 65544, 500)])   # 128 MB: the sums are rounded elsewhere
def test_long_responses_are_summed_without_the_rounding_of_a_running_sum(dtype, vocab, rows):
    x, _ = wl.logits_and_tokens(rows, (vocab + 7) // 8 * 8, 31, 3.0 ** 0.5, dtype)
    rng = np.random.default_rng(4)
    targets = rng.integers(0, vocab, rows).astype(np.int32)
    seg = np.where(np.arange(rows) % 7 == 0, -1, np.arange(rows) * 3 // rows).astype(np.int32)
    dev = lambda a: torch.as_tensor(a).cuda()  # noqa: E731
    xd = x.cuda()[:, :vocab]
    got = B.dpo_logp(xd, dev(targets), dev(seg), 4, dev(np.array([0, 7], np.int32)), dev(np.array([1, 2], np.int32)),
                     dev(np.array([0, 2], np.int32))).cpu().double().numpy()
    want = orc.dpo_logp(wl.to_f64(x)[:, :vocab], targets, seg, 4, [0, 7], [1, 2], [0, 2])
    # per row half an ulp of its fp32 log-sum-exp (below 16: 5e-7) and the exponentials' error of the same size, with
    # signs that differ from row to row; then one rounding of the sum (6e-8 of it)
    assert got[3] == 0 and (np.abs(got - want) <= 1e-6 * 4 * np.sqrt(rows) + 6e-8 * np.abs(want)).all()


@pytest.mark.parametrize("n_segments", [1, 31, 33, 70, 1000])
def test_the_last_row_rounds_every_sum(n_segments):
    # small launches: the row that finishes last rounds all sums, a lane for each; every sum has to hold every row's term
    rows, vocab = 900, 512
    x, _ = wl.logits_and_tokens(rows, vocab, 5, 3.0 ** 0.5, torch.bfloat16)
    rng = np.random.default_rng(n_segments)
    targets = rng.integers(0, vocab, rows).astype(np.int32)
    seg = rng.integers(-1, n_segments, rows).astype(np.int32)
    args = x.cuda(), _dev(targets), _dev(seg), n_segments
    want = orc.dpo_logp(wl.to_f64(x), targets, seg, n_segments)
    for got in [B.dpo_logp(*args, out=torch.full((n_segments,), 7.0, device="cuda")) for _ in range(30)]:
        got = got.cpu().double().numpy()
        # up to 900 terms, each off by an ulp of its fp32 log-sum-exp (1e-6); the rounding of a sum of at most 900 x 15
        assert (np.abs(got - want) <= 1e-6 * 4 * np.sqrt(rows) + 6e-8 * np.abs(want)).all()


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("vocab", [1, 7, 1000, 16392])
def test_terms_at_the_ends_of_their_range(dtype, vocab):
    """Responses of tokens that take all of the probability (terms of 0, where rounding must not add up), of a token
    that is impossible (-inf), and with a NaN among the logits; the others keep their values."""
    rows, stride = 400, (vocab + 7) // 8 * 8
    x, _ = wl.logits_and_tokens(rows, stride, 12, 3.0 ** 0.5, dtype)
    targets = np.random.default_rng(1).integers(0, vocab, rows).astype(np.int32)
    seg = (np.arange(rows) // 100).astype(np.int32)
    at = torch.as_tensor(targets[:100]).long()
    x[torch.arange(100), at] = 150 + 7.3 * x[torch.arange(100), at]      # response 0: all certain
    x[150, targets[150]] = -float("inf")                                 # response 1 (vocab 1: no probability left at all)
    x[250, vocab // 2] = float("nan")                                    # response 2
    got = B.dpo_logp(x.cuda()[:, :vocab], _dev(targets), _dev(seg), 5).cpu().double().numpy()
    with np.errstate(invalid="ignore", divide="ignore"):
        want = orc.dpo_logp(wl.to_f64(x)[:, :vocab], targets, seg, 5)
    # per certain row the exponential's error (2^-22), all of the same sign at worst
    assert abs(got[0] - want[0]) <= 100 * 5e-7, (got[0], want[0])
    assert np.isnan(got[1]) if vocab == 1 else got[1] == -np.inf
    assert np.isnan(got[2])
    # (vocab 1: log2 of a sum that should be 1, with the exponential's error)
    assert abs(got[3] - want[3]) <= 1e-6 * 4 * 10 + 6e-8 * abs(want[3]), (got[3], want[3])
    assert got[4] == 0 and (got[[0, 3]] <= 0).all()


@pytest.mark.parametrize("dtype,vocab", [(torch.float32, 1001), (torch.bfloat16, 1003), (torch.bfloat16, 33000), (torch.float32, 17000)])
def test_the_entry_point_without_scratch(dtype, vocab):
    """dpo_logp of the C ABI: fp32 sums added straight into out."""
    rows, stride = 300, (vocab + 7) // 8 * 8
    x, _ = wl.logits_and_tokens(rows, stride, 6, 3.0 ** 0.5, dtype)
    rng = np.random.default_rng(3)
    targets = rng.integers(0, vocab, rows).astype(np.int32)
    seg = rng.integers(-1, 4, rows).astype(np.int32)
    forks = [np.array(a, dtype=np.int32) for a in ([0, 299, 7], [vocab - 1, 0, 5], [3, 0, 1])]
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    out = torch.full((5,), 7.0, device="cuda")
    xd, dev = x.cuda(), [_dev(a) for a in (targets, seg, *forks)]
    code = B.load_library().dpo_logp(xd.data_ptr(), B.PSA_DTYPE_F32 if dtype == torch.float32 else B.PSA_DTYPE_BF16, rows, vocab,
                                     stride, *(a.data_ptr() for a in dev), 3, 4, out.data_ptr(), status.data_ptr(),
                                     torch.cuda.current_stream().cuda_stream)
    assert code == 0 and read_status(status) == 0
    want = orc.dpo_logp(wl.to_f64(x)[:, :vocab], targets, seg, 4, *forks)
    got = out.cpu().double().numpy()
    # per term an ulp of its fp32 log-sum-exp, and half an ulp of the running sum (6e-8 of it) for each of about 60 terms
    assert got[4] == 7.0 and (np.abs(got[:4] - want) <= 300 * 1e-6 + 60 * 6e-8 * np.abs(want)).all()


def test_a_captured_call_is_replayed_with_new_logits():
    rows, vocab = 200, 1000
    rng = np.random.default_rng(8)
    targets, seg = rng.integers(0, vocab, rows).astype(np.int32), rng.integers(-1, 6, rows).astype(np.int32)
    x = torch.zeros((rows, vocab), dtype=torch.bfloat16, device="cuda")
    args = x, _dev(targets), _dev(seg), 6
    out = torch.zeros(6, device="cuda")
    B.dpo_logp(*args, out=out)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        B.dpo_logp(*args, out=out)
    for seed in (1, 2):
        new, _ = wl.logits_and_tokens(rows, vocab, seed, 3.0 ** 0.5, torch.bfloat16)
        x.copy_(new)
        graph.replay()
        torch.cuda.synchronize()
        want = orc.dpo_logp(wl.to_f64(new), targets, seg, 6)
        assert (np.abs(out.cpu().double().numpy() - want) <= TOL_LOGP * np.abs(want)).all()
