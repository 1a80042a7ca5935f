"""Attention of short bf16 sequences: the exponentials are fp32's, not the hardware approximation's."""
import numpy as np
import pytest

import pm_inputs as I

pytestmark = pytest.mark.gpu


def stash(pipe, want):
    """The bf16 tensor in the activation rings that is closest to `want` (all positive), by the exponents at a few places."""
    import torch
    w = want.reshape(-1).log2().float()
    mem = pipe.ring[: pipe.ring.numel() // 256 * 256].view(torch.bfloat16)
    v = mem.view(-1, 128).float().log2()
    n = w.numel() // 128
    m = v.shape[0] - n + 1
    d = sum((v[k:k + m] - w[128 * k:128 * k + 128]).abs().nan_to_num(1e3, 1e3, 1e3).sum(1) for k in range(0, n, n // 40))
    i = int(d.argmin()) * 128
    return mem[i:i + w.numel()].view(want.shape)


# One key of every sequence has the largest score s and the value 0, all others score 0 and have the value 1, so a query's
# output is (S - 1) bf16(e^-s) / (1 + (S - 1) e^-s) in every column.  Scores are products of two bf16 numbers, hence exact.
# A relative error eps of e^-s moves the rounding for a share of about eps / 2^-9.5 of the queries; at s up to 60 that is
# below 1e-4 for expf (2^-23, and as much for the rest of the expression: 3 of 32000) and 1e-3 for the hardware exponential
# (2^-22 + s 2^-24: 30 of 32000).
@pytest.mark.parametrize("seq_len,batch", [(127, 16), (40, 50), (17, 120)])
def test_exponentials(cuda_device, seq_len, batch):
    import torch
    import paper_1910_05124_b200 as pm
    d, heads, vocab, T = 1024, 16, 4096, seq_len * batch
    wl = I.encoder_workload("exponentials", 1, d, heads, 64, seq_len, batch, vocab, compute="bf16", optimizer="sgdm", alpha=0.01, K=4, D=0.5,
                            steps=1, seed=3)
    params = I.init_encoder_params(wl)
    rng = np.random.default_rng(seq_len)
    # columns whose position term is 1 to within 1e-4 at every position: the embedded value is 1 + 32 t for any bf16 sum in [1, 4)
    a, b, c = d - 1, d - 3, d - 5
    grid = np.concatenate([1 + np.arange(128) / 128, 2 + np.arange(128) / 64])
    table = np.zeros((vocab, d), np.float32)
    ub, uc = rng.choice(grid, vocab), rng.choice(grid, vocab)
    table[1:, a], table[:, b], table[:, c] = 1 / 32, (ub - 1) / 32, (uc - 1) / 32
    W, bias = np.zeros((3 * d, d), np.float32), np.zeros(3 * d, np.float32)
    w1, w2, wk = (I.round_to_bf16(rng.uniform(lo, hi, heads)) for lo, hi in ((2, 60), (2, 60), (0.5, 1)))
    q0, k0 = np.arange(heads) * 64, d + np.arange(heads) * 64
    W[q0, b], W[q0, c] = w1, w2
    W[k0, a], bias[k0] = -wk, 2 * wk                         # key: wk where the id is 0, else 0
    W[2 * d:, a], bias[2 * d:] = 1, -1                       # value: 0 where the id is 0, else 1
    params[0] = [table, W, bias]
    ids = rng.integers(1, vocab, (batch, seq_len))
    ids[:, 0] = 0
    pipe = pm.Pipeline(wl, params, loop_order="mb_major")
    dev = torch.from_numpy(ids.astype(np.int32).reshape(-1)).cuda()
    pipe.pm_forward(dev, dev)
    torch.cuda.synchronize()
    q = I.round_to_bf16(ub[ids].reshape(T, 1) * w1 + uc[ids].reshape(T, 1) * w2).astype(np.float64)
    e = np.exp(-q * wk / 8)
    want = (seq_len - 1) * I.round_to_bf16(e).astype(np.float64) / (1 + (seq_len - 1) * e)
    want = torch.from_numpy(I.round_to_bf16(want)).cuda().repeat_interleave(64, 1)
    got = stash(pipe, want).float()
    assert float(((got - want).abs() / want).max()) < 2.0 ** -6
    off = int((got != want)[:, ::64].sum())
    assert off <= 2e-4 * T * heads, (off, T * heads)
