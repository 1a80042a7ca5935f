"""Microbatches of more rows than a grid's second dimension has blocks of 64."""
import numpy as np
import pytest

import pm_inputs as I

pytestmark = pytest.mark.gpu


# 65535 blocks of 64 rows end at row 4194240
@pytest.mark.parametrize("T", [4194240, 4194240 + 104])
def test_activation_backward_of_one_stage(cuda_device, T):
    import torch
    import paper_1910_05124_b200 as pm
    width = 8
    wl = I.mlp_workload("long", 2, width, 1, "gelu", T, compute="bf16", optimizer="sgdm", alpha=0.01, K=4, D=0.5, steps=1, seed=5)
    gen = torch.Generator(device="cuda").manual_seed(T)
    rnd = lambda *shape: torch.randn(*shape, generator=gen, device="cuda")
    r16 = lambda v: v.float().bfloat16().double()
    params0 = [[(rnd(width, width).cpu().numpy() / np.float32(np.sqrt(width)), 0.1 * rnd(width).cpu().numpy())] for _ in range(2)]
    pipe = pm.Pipeline(wl, params0, loop_order="mb_major")
    x, y = rnd(T, width).bfloat16(), rnd(T, width) + 1
    y[-104:] *= 1e6                                                 # the last rows are most of every gradient
    pipe.pm_forward(x, y)
    pipe.pm_backward()
    got = pipe.unpack(pipe.grad)

    cu = lambda a: torch.from_numpy(a).cuda()
    W = [cu(st[0][0]) for st in params0]
    fn = torch.nn.functional.gelu
    h, zs = [x.double()], []
    for i in range(2):
        zs.append(r16(h[-1] @ r16(W[i]).T + cu(params0[i][0][1]).double()))
        h.append(r16(fn(zs[-1])))
    g = r16(2 * (h[-1] - y.double()) / (T * width))
    for i in (1, 0):
        zz = zs[i].clone().requires_grad_(True)
        fn(zz).sum().backward()
        g = r16(g * zz.grad)
        gw, gb = got[i][0]
        # A sum of T values in fp32 whose partial sums stay below the sum of magnitudes: T/64 additions of sums over 64 rows, each off by
        # 2^-24 of it at most; a tenth of a percent besides for the roundings to bf16 of z, y and dz that fall on the other side of a tie.
        tol = T / 64 * 2.0 ** -24 + 1e-3
        assert float((cu(gb).double() - g.sum(0)).abs().max() / g.abs().sum(0).max()) <= tol, (i, "bias")
        assert float((cu(gw).double() - g.T @ h[i]).abs().max() / (g.abs().T @ h[i].abs()).max()) <= 4 * tol, (i, "weights")   # 16 rows per product
        g = r16(g @ r16(W[i]))
