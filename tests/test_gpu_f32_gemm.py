"""The fp32 GEMM kernels (forward, corrected input gradient, weight gradient) at the edges of their tiles, against the same
products in float64."""
import numpy as np
import pytest

import pm_inputs as I

pytestmark = pytest.mark.gpu


# widths and rows around the 16- and 32-wide tiles, rows that do not start on 16 bytes (width % 4), reductions of less than one
# 16-deep chunk, of a ragged last chunk and of more chunks than the eight warps keep in flight (16 * 8 * 4); 400 x 300 and
# 530 x 70 have more 32 x 32 tiles than the chip has SMs and take the larger tile
@pytest.mark.parametrize("width,T", [(1, 1), (7, 5), (16, 16), (17, 31), (36, 33), (130, 20), (200, 50), (400, 300), (530, 70), (1100, 9)])
@pytest.mark.parametrize("act", ["none", "gelu"])
def test_f32_products(cuda_device, width, T, act):
    import torch
    import paper_1910_05124_b200 as pm
    wl = I.mlp_workload("f32_gemm", 2, width, 2, act, T, compute="f32", optimizer="sgdm", alpha=0.01, K=4, D=0.5, steps=1, seed=7)
    gen = torch.Generator().manual_seed(width * 1000 + T)
    rnd = lambda *shape: torch.randn(*shape, generator=gen, dtype=torch.float64).float()
    params0 = [[(rnd(width, width).numpy() / np.sqrt(width), 0.1 * rnd(width).numpy()) for _ in range(2)] for _ in range(2)]
    pipe = pm.Pipeline(wl, params0, loop_order="mb_major")
    pipe.delta.copy_(0.01 * rnd(pipe.total))
    delta = pipe.unpack(pipe.delta)
    x, y = rnd(T, width), rnd(T, width)
    pipe.pm_forward(x.cuda(), y.cuda())
    pipe.pm_backward()
    got = pipe.unpack(pipe.grad)
    pipe.pm_update()

    W = [torch.from_numpy(w).double() for st in params0 for w, _ in st]
    b = [torch.from_numpy(v).double() for st in params0 for _, v in st]
    D = [torch.from_numpy(w).double() for st in delta for w, _ in st]
    gap = [wl.tau_fwd[i // 2] for i in range(4)]
    h, zs = [x.double()], []
    for i in range(4):
        zs.append(h[-1] @ W[i].T + b[i])
        h.append(torch.nn.functional.gelu(zs[-1]) if act == "gelu" else zs[-1])
    g = 2 * (h[-1] - y.double()) / (T * width)
    np.testing.assert_allclose(pipe.pm_get_losses(0, 1)[0], float((h[-1] - y.double()).square().mean()), rtol=1e-5)
    # a sum of n terms in fp32 is off by about sqrt(n) 2^-24 of its terms' size; four layers and their backward chain such errors
    tol = 16 * np.sqrt(max(width, T)) * 2.0 ** -24
    rel = lambda a, r: float((torch.from_numpy(a).double() - r).norm() / r.norm().clamp_min(1e-30))
    for i in reversed(range(4)):
        if act == "gelu":
            zz = zs[i].clone().requires_grad_(True)
            torch.nn.functional.gelu(zz).sum().backward()
            g = g * zz.grad
        gw, gb = got[i // 2][i % 2]
        # the cancellation in a sum of few terms can leave less than the terms: measured against the terms' norm
        assert rel(gw, g.T @ h[i]) <= tol + 1e-6, (i, "weights")
        assert rel(gb, g.sum(0)) <= (tol + 1e-6) * max(1.0, float(g.norm() * np.sqrt(T) / g.sum(0).norm())), (i, "bias")
        g = g @ (W[i] - gap[i] * D[i])
