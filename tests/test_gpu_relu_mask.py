"""bf16 networks with many rows: the ReLU mask bits that the forward GEMM leaves for the dgrad that applies them (which microbatch's they are, in
every loop order), and the bias gradients summed beside the weight gradients by CTAs that walk several tiles."""
import numpy as np
import pytest

import pm_inputs as I

pytestmark = pytest.mark.gpu


def network(widths, per_stage, T):
    """Linears widths[i] -> widths[i + 1] in stages of per_stage, ReLU but for the last."""
    n = len(widths) - 1
    lin = [I.LinearSpec(a, b, "relu" if i < n - 1 else "none") for i, (a, b) in enumerate(zip(widths, widths[1:]))]
    wl = I.mlp_workload("mask", n // per_stage, 8, per_stage, "relu", T, compute="bf16", optimizer="sgdm", alpha=0.0, K=4, D=0.5, steps=1, seed=3)
    wl.stages = [lin[p * per_stage:(p + 1) * per_stage] for p in range(n // per_stage)]
    return wl


def check(wl, order, *, entry_period=1, own_launch=False, **options):
    """The gradients each stage's last backward pass left, with a microbatch of its own per step and weights that stand still, against the
    same products in float64 with the same roundings.  own_launch: are there activations whose backward is a launch of its own?"""
    import torch
    import paper_1910_05124_b200 as pm
    P, T = wl.n_stages, wl.microbatch
    lin = [l for st in wl.stages for l in st]
    gen = torch.Generator(device="cuda").manual_seed(T + len(lin))
    rnd = lambda *shape: torch.randn(*shape, generator=gen, device="cuda")
    r16 = lambda v: v.float().bfloat16().double()
    flat = [(rnd(l.n_out, l.n_in).cpu().numpy() * np.float32(1.4 / np.sqrt(l.n_in)), 0.1 * rnd(l.n_out).cpu().numpy()) for l in lin]
    params0 = [flat[p * len(st):(p + 1) * len(st)] for p, st in enumerate(wl.stages)]
    pipe = pm.Pipeline(wl, params0, loop_order=order, entry_period=entry_period, **options)
    E, seen, last = entry_period, [], [-1] * P
    for step in range(4 if order == "mb_major" else E * (4 * P + 3)):       # every ring has come round; phases replayed as graphs
        if step % E:
            pipe.pm_step(None, None)
        else:
            seen.append((rnd(T, lin[0].n_in).bfloat16(), rnd(T, lin[-1].n_out) - 3))      # (a mean, so that column sums are sums of one sign)
            pipe.pm_step(*seen[-1])
        for p in range(P):
            b_mb = pipe.pm_get_bookkeeping(p)[2]
            last[p] = b_mb if b_mb >= 0 else last[p]
    got = pipe.unpack(pipe.grad)
    pipe.pm_profile_enable()
    for _ in range(E):
        pipe.pm_step(*seen[0]) if order == "mb_major" or E == 1 else pipe.pm_step(None, None)
    assert (pipe.pm_profile_read()["act_bwd"][1] > 0) == own_launch
    W = [torch.from_numpy(w).cuda() for w, _ in flat]
    b = [torch.from_numpy(v).cuda().double() for _, v in flat]
    # four roundings of 2^-8 per Linear (z, y, dx, dz; see the products of launches with few tiles) and as much again from units whose
    # sign an earlier rounding decides; the mask of another microbatch, or a missing 64-row block or tile, is 0.2 to 1
    tol = 2 * np.sqrt(4 * len(lin)) * 2.0 ** -8
    rel = lambda a, r: float((torch.from_numpy(a).cuda().double() - r).norm() / r.norm())
    assert min(last) >= 0
    for mb in sorted(set(last)):
        x, y = seen[mb]
        h, zs = [x.double()], []
        for i, l in enumerate(lin):
            zs.append(r16(h[-1] @ r16(W[i]).T + b[i]))
            h.append(r16(torch.relu(zs[-1])) if l.act == "relu" else zs[-1])
        g = r16(2 * (h[-1] - y.double()) / (T * lin[-1].n_out))
        for i in reversed(range(len(lin))):
            if lin[i].act == "relu":
                g = g * (zs[i] > 0)
            p, j = divmod(i, len(wl.stages[0]))
            if last[p] == mb:
                assert rel(got[p][j][0], g.T @ h[i]) <= tol, (p, j, "weights")
                db = torch.from_numpy(got[p][j][1]).cuda().double()
                assert float((db - g.sum(0)).norm() / g.abs().sum(0).norm()) <= tol, (p, j, "bias")
            if i:
                g = r16(g @ r16(W[i]))


# More than 296 tiles of 128 rows x 64 columns per launch, which the kernels for few tiles do not take; remainders in every tile.
def test_ticks_on_pairs(cuda_device):
    check(network([768] * 5, 1, 1030), "tick_major")


def test_ticks_on_pairs_two_linears_per_stage(cuda_device):
    check(network([520] * 9, 2, 1500), "tick_major")


def test_ticks_whose_forward_is_one_cta_and_dgrad_pairs(cuda_device):
    check(network([768, 768, 768, 768, 72], 1, 1030), "tick_major")


def test_microbatches_on_pairs_two_linears_per_stage(cuda_device):
    check(network([520] * 5, 2, 4300), "mb_major")


def test_queued_weights_on_one_cta(cuda_device):
    check(network([200] * 4, 1, 9500), "mb_major", materialize_backward=1)


def test_entry_period(cuda_device):
    check(network([264] * 4, 1, 7700), "tick_major", entry_period=3)


def test_recompute_segments(cuda_device):
    check(network([264] * 5, 1, 7700), "mb_major", recompute_segment=2, own_launch=True)


# Weight gradients of 200 and 180 tiles on 74 pairs and 148 CTAs, summed tiles (the first column) between others; 64-row blocks as
# many as the operand ring has slots (5 and 4), fewer and more.
@pytest.mark.parametrize("T", [130, 256, 300, 380])
def test_bias_gradients_of_several_tiles_per_cta(cuda_device, T):
    check(network([1032] * 9, 1, max(T, 256)), "mb_major", own_launch=False)
    check(network([1032, 248] * 5 + [1032], 1, T), "mb_major", own_launch=False)
