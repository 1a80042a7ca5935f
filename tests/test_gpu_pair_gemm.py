"""bf16 GEMMs of launches with many output tiles (CTA pairs): the products, the corrected weights they read, the ReLU mask and the bias
gradients summed beside the weight gradients, at sizes that leave remainders in every tile."""
import numpy as np
import pytest

import pm_inputs as I
from test_gpu_row_gemm import test_bf16_products as check_products

pytestmark = pytest.mark.gpu


# 13 x 24 and 17 x 33 tiles of 128 rows x 64 columns: more than the kernel for few tiles takes; rows and columns beyond whole tiles of
# 256, boxes of 32 x 64 and k-blocks of 64
@pytest.mark.parametrize("width,T", [(776, 3000), (1032, 4100)])
@pytest.mark.parametrize("act", ["relu", "gelu"])
def test_bf16_products_on_pairs(cuda_device, width, T, act):
    check_products(cuda_device, width, T, act)


# A column of ones in the input makes one column of dW the sum that the bias gradient is.  Both add the same T products or values in
# fp32; an order of n additions is within n 2^-24 of the exact sum of magnitudes, and both chains are at most T long.
@pytest.mark.parametrize("order", ["tick_major", "mb_major"])
@pytest.mark.parametrize("width,T,n_micro", [(8, 1, 1), (72, 63, 1), (136, 65, 1), (264, 512, 1), (264, 300, 2), (1032, 130, 1), (1032, 257, 4)])
def test_bias_gradient_is_the_weight_gradient_of_ones(cuda_device, order, width, T, n_micro):
    import torch
    import paper_1910_05124_b200 as pm
    if order == "tick_major" and n_micro > 1:
        pytest.skip("several microbatches per update are microbatch-major")
    wl = I.mlp_workload("bias", 2, width, 1, "relu", T, compute="bf16", optimizer="sgdm", alpha=0.01, K=4, D=0.5, steps=1, seed=3)
    gen = torch.Generator(device="cuda").manual_seed(width + T)
    rnd = lambda *shape: torch.randn(*shape, generator=gen, device="cuda")
    params0 = [[(rnd(width, width).cpu().numpy() / np.float32(np.sqrt(width)), rnd(width).cpu().numpy())] for _ in range(2)]
    pipe = pm.Pipeline(wl, params0, loop_order=order, n_micro=n_micro)
    x = rnd(T, width).bfloat16()
    x[:, 0] = 1.0
    for _ in range(n_micro if order == "mb_major" else 4):          # tick-major: stage 1 has had its backward after 2P ticks
        pipe.pm_forward(x, rnd(T, width))
        pipe.pm_backward()
        pipe.pm_update()
    dw, db = pipe.unpack(pipe.grad)[0][0]
    scale = np.abs(dw).max() * np.sqrt(T) + np.abs(db).max()        # |sum of magnitudes| of a column is about sqrt(T) of its sum
    assert np.abs(db).max() > 0
    np.testing.assert_allclose(dw[:, 0], db, rtol=0, atol=n_micro * T * 2.0 ** -24 * scale)
