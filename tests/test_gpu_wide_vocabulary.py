"""Vocabularies much larger than the microbatch: the embedding gradient, most of whose rows have no token, and the
cross-entropy that walks long rows of logits."""
import numpy as np
import pytest

import pm_inputs as I

pytestmark = pytest.mark.gpu


# a microbatch of fewer, as many and more tokens than one pass of a warp or a block looks at (32, 256); a quarter of the
# vocabulary and less; widths of one and several column slices, and one that leaves lanes without a column; ids all equal
# (one row summed by eight warps), from a few values (rows of both kinds, every token repeated) and all over the table;
# vocabularies at the ends of the long cross-entropy rows (8192 excluded, 32768, and one beyond it that takes the other kernel)
@pytest.mark.parametrize("d_model,seq,batch,vocab,ids", [(64, 8, 4, 8196, "uniform"), (64, 8, 5, 8200, "equal"), (72, 16, 17, 9000, "few"),
                                                         (264, 16, 16, 16384, "few"), (520, 32, 20, 32768, "uniform"), (128, 16, 8, 33000, "equal")])
@pytest.mark.parametrize("compute", ["f32", "bf16"])
def test_embedding_gradient_and_loss(cuda_device, compute, d_model, seq, batch, vocab, ids):
    import torch
    import paper_1910_05124_b200 as pm
    if compute == "bf16":
        vocab = (vocab + 7) // 8 * 8
    wl = I.encoder_workload("wide", 1, d_model, {264: 6, 520: 13}.get(d_model, 2), 64, seq, batch, vocab, compute=compute, optimizer="sgdm", alpha=0.01,
                            K=4, D=0.5, steps=1, seed=5)
    params0 = I.init_encoder_params(wl)
    pipe = pm.Pipeline(wl, params0, loop_order="mb_major")
    gen = torch.Generator().manual_seed(vocab + d_model)
    T = seq * batch
    tok = {"uniform": torch.randint(0, vocab, (T,), generator=gen), "equal": torch.full((T,), vocab - 1),
           "few": torch.randint(0, 12, (T,), generator=gen) * (vocab // 12)}[ids].int()
    tgt = torch.randint(0, vocab, (T,), generator=gen).int()
    pipe.grad.fill_(7.0)                                             # what an earlier step left in the arena
    pipe.pm_forward(tok.cuda(), tgt.cuda())
    pipe.pm_backward()
    table = pipe.unpack(pipe.grad)[0][0]
    pipe.pm_update()
    hit = np.zeros(vocab, bool)
    hit[tok.numpy()] = True
    assert not table[~hit].any()                                     # rows without a token: zeros, not what was there
    assert np.isfinite(table[hit]).all()
    # the gradient of the table summed over its rows is sqrt(d) times the sum of du over the tokens, whatever the ids: the same
    # network on ids spread over the table, with the embedding of the tokens it replaces, gives the same du
    spread = torch.arange(T).int() * (vocab // T)
    p1 = [list(st) for st in params0]
    p1[0][0] = np.zeros_like(p1[0][0])
    p1[0][0][spread.numpy()] = params0[0][0][tok.numpy()]
    other = pm.Pipeline(wl, p1, loop_order="mb_major")
    other.pm_forward(spread.cuda(), tgt.cuda())
    other.pm_backward()
    rows = torch.from_numpy(other.unpack(other.grad)[0][0][spread.numpy()]).double()
    other.pm_update()
    ref = torch.zeros(vocab, d_model, dtype=torch.float64).index_add_(0, tok.long(), rows)
    # fp32 sums of at most T terms against float64, relative to the terms: T 2^-24; the two runs' du are the same bits
    scale = torch.zeros(vocab, d_model, dtype=torch.float64).index_add_(0, tok.long(), rows.abs())
    assert ((torch.from_numpy(table).double() - ref).abs() <= T * 2.0 ** -24 * scale + 1e-30).all()
    loss = pipe.pm_get_losses(0, 1)[0]
    assert abs(loss - other.pm_get_losses(0, 1)[0]) <= 1e-6 * loss


# rows of logits that leave a thread's registers part empty and fill them, and rows too long for them; more rows than SMs (a block
# walks several), fewer, and an odd number; the whole network in float64, with the same roundings, as the reference
@pytest.mark.parametrize("vocab,batch", [(8200, 25), (16384, 33), (32768, 19), (32768, 40), (33000, 20)])
@pytest.mark.parametrize("compute", ["f32", "bf16"])
def test_cross_entropy_of_long_rows(cuda_device, compute, vocab, batch):
    import torch
    import paper_1910_05124_b200 as pm
    from oracle import transformer
    wl = I.encoder_workload("long", 1, 64, 2, 64, 9, batch, vocab, compute=compute, optimizer="sgdm", alpha=0.0, K=4, D=0.5, steps=1, seed=vocab + batch)
    params0 = I.init_encoder_params(wl)
    params0[-1][2] *= np.float32(3)                                  # logits of a trained network's spread: probabilities up to 1e-2
    data = lambda t: I.token_batch(wl, 0)
    ref_loss, ref = transformer.make_grad_fn(wl.stage_specs, data, 2, 9, vocab, compute)(0, params0, params0)
    pipe = pm.Pipeline(wl, params0, loop_order="mb_major")
    pipe.pm_step(*(torch.from_numpy(a.astype(np.int32)).cuda() for a in data(0)))
    got = pipe.unpack(pipe.grad)
    # fp32: sums of up to V terms in 64-bit against 32-bit order, sqrt(V) 2^-24; bf16: the gradient of the logits is rounded once
    # (2^-9 at most, 2^-10 on average) and its exponentials are the hardware's
    tol = 5e-5 if compute == "f32" else 1e-2
    assert abs(pipe.pm_get_losses(0, 1)[0] - ref_loss) <= (1e-5 if compute == "f32" else 1e-3) * ref_loss
    for p, stage in ((-1, got[-1]), (-2, got[-2])):
        for j, a in enumerate(stage):
            assert np.linalg.norm(a - ref[p][j]) <= tol * np.linalg.norm(ref[p][j]), (p, j)


# the hit list of the embedding gradient grows with the microbatch: just below, at and beyond 48 KB beside the kernel's static
# shared memory (a launch of 46 KB used to be refused)
@pytest.mark.parametrize("batch", [224, 240, 256])
@pytest.mark.parametrize("compute", ["f32", "bf16"])
def test_embedding_gradient_of_long_microbatches(cuda_device, compute, batch):
    import torch
    import paper_1910_05124_b200 as pm
    from oracle import transformer
    wl = I.encoder_workload("hits", 1, 256, 4, 32, 16, batch, 40, compute=compute, optimizer="sgdm", alpha=0.0, K=4, D=0.5, steps=1, seed=batch)
    params0 = I.init_encoder_params(wl)
    data = lambda t: I.token_batch(wl, 0)
    ref_loss, ref = transformer.make_grad_fn(wl.stage_specs, data, 4, 16, 40, compute)(0, params0, params0)
    pipe = pm.Pipeline(wl, params0, loop_order="mb_major")
    pipe.pm_step(*(torch.from_numpy(a.astype(np.int32)).cuda() for a in data(0)))
    table = pipe.unpack(pipe.grad)[0][0]
    assert abs(pipe.pm_get_losses(0, 1)[0] - ref_loss) <= (1e-5 if compute == "f32" else 1e-3) * ref_loss
    # fp32: sums of a hundred tokens behind five Linears; bf16: a dozen roundings of 2^-9 in front of them
    assert np.linalg.norm(table - ref[0][0]) <= (1e-4 if compute == "f32" else 2e-2) * np.linalg.norm(ref[0][0])
