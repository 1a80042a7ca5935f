"""bf16 GEMMs of launches with few output tiles (forward, corrected input gradient with the receiving Linear's activation
derivative) and the column sums of short microbatches, against the same products in float64 with the same roundings."""
import numpy as np
import pytest

import pm_inputs as I
from parity_util import run_gpu_pipeline, run_oracle, compare_params

pytestmark = pytest.mark.gpu


# rows below, at and beyond one 128-row tile; widths that leave remainders in the 32- and 64-column tiles, in the 64-deep
# k-blocks and in the four-way (width >= 512) and two-way (>= 256) split of the reduction; 1024 x 300 walks its operand
# ring more than once; 1024 x 600 and 1024 x 2048 take 64-column tiles, split and not; 513 rows sum their columns in chunks
@pytest.mark.parametrize("width,T", [(8, 1), (72, 16), (40, 128), (264, 129), (328, 72), (520, 100), (1024, 128), (1024, 300), (1024, 600),
                                     (136, 513), (1024, 2048)])
@pytest.mark.parametrize("act", ["relu", "gelu"])
def test_bf16_products(cuda_device, width, T, act):
    import torch
    import paper_1910_05124_b200 as pm
    wl = I.mlp_workload("row_gemm", 2, width, 2, act, T, compute="bf16", optimizer="sgdm", alpha=0.01, K=4, D=0.5, steps=1, seed=7)
    gen = torch.Generator(device="cuda").manual_seed(width * 1000 + T)
    rnd = lambda *shape: torch.randn(*shape, generator=gen, device="cuda")
    r16 = lambda v: v.float().bfloat16().double()
    params0 = [[(rnd(width, width).cpu().numpy() * np.float32(1.5 / np.sqrt(width)), 0.1 * rnd(width).cpu().numpy()) for _ in range(2)] for _ in range(2)]
    pipe = pm.Pipeline(wl, params0, loop_order="mb_major")
    pipe.delta.copy_(0.002 * rnd(pipe.total))
    delta = pipe.unpack(pipe.delta)
    x, y = rnd(T, width).bfloat16(), rnd(T, width)
    pipe.pm_forward(x, y)
    pipe.pm_backward()
    got = pipe.unpack(pipe.grad)
    pipe.pm_update()

    cu = lambda a: torch.from_numpy(a).cuda()
    W = [cu(w) for st in params0 for w, _ in st]
    b = [cu(v).double() for st in params0 for _, v in st]
    D = [cu(w) for st in delta for w, _ in st]
    fn = torch.relu if act == "relu" else torch.nn.functional.gelu
    h, zs = [x.double()], []
    for i in range(4):
        zs.append(r16(h[-1] @ r16(W[i]).T + b[i]))
        h.append(r16(fn(zs[-1])))
    np.testing.assert_allclose(pipe.pm_get_losses(0, 1)[0], float((h[-1] - y.double()).square().mean()), rtol=2e-3)
    g = r16(2 * (h[-1] - y.double()) / (T * width))
    rel = lambda a, r: float((cu(a).double() - r).norm() / r.norm().clamp_min(1e-30))
    # Another order of summation moves a sum of n terms by about sqrt(n) 2^-24; rounding to bf16 turns a relative perturbation
    # eps into one of about sqrt(eps 2^-8) (a share eps / 2^-8 of the values falls on the other side of a tie and moves by
    # 2^-8), so after two or three roundings the perturbation of every stored tensor is of the order of 2^-8 = 3.9e-3 and stays
    # there.  The gradients of the first Linear carry sixteen roundings (z, y, dx, dz of four Linears): 4 x 3.9e-3, and the
    # entries whose ReLU mask changed.  A missing k-block, rank or tile is 1/4 (two of eight blocks) to 1/32 of a sum's norm.
    tol = 2e-2
    for i in reversed(range(4)):
        zz = zs[i].clone().requires_grad_(True)
        fn(zz).sum().backward()
        g = r16(g * zz.grad)
        gw, gb = got[i // 2][i % 2]
        assert rel(gw, g.T @ h[i]) <= tol, (i, "weights")
        assert rel(gb, g.sum(0)) <= tol * max(1.0, float(g.norm() * np.sqrt(T) / g.sum(0).norm().clamp_min(1e-30))), (i, "bias")
        g = r16(g @ r16(W[i] - wl.tau_fwd[i // 2] * D[i]))


# launches over all stages with few tiles: 32-column tiles unsplit, in two and in four parts, 64-column tiles, several row tiles
@pytest.mark.parametrize("P,width,T", [(3, 40, 16), (8, 328, 72), (2, 520, 128), (4, 264, 300), (6, 512, 200)])
def test_bf16_grouped_ticks(cuda_device, P, width, T):
    wl = I.mlp_workload("row_ticks", P, width, 1, "relu", T, compute="bf16", optimizer="sgdm", alpha=0.01, K=4, D=0.5, steps=6, seed=11 + P)
    params0 = I.init_stage_params(wl)
    res = run_oracle(wl, params0, wl.steps)
    pipe, losses, book = run_gpu_pipeline(wl, params0, wl.steps)
    np.testing.assert_allclose(losses, np.array(res.losses), rtol=1e-3)      # the tolerances of the bf16 path up to a dozen layers
    compare_params(pipe, res, 2e-2)
