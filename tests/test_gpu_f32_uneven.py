"""fp32 networks whose Linears differ much in size: launches over all stages and over one, against the oracle."""
import numpy as np
import pytest

import pm_inputs as I
from parity_util import run_gpu_pipeline, run_oracle, compare_params

pytestmark = pytest.mark.gpu


# a vocabulary of many tiles beside narrow Linears (its own, and all tiles together, on both sides of 148 tiles of 32 x 32:
# 148 row tiles times one column tile, one more, and a ragged one), and widths that change from Linear to Linear
@pytest.mark.parametrize("order", ["tick_major", "mb_major"])
@pytest.mark.parametrize("d_model,vocab", [(16, 33), (16, 4736), (16, 4737), (40, 3000)])
def test_vocabulary(cuda_device, order, d_model, vocab):
    wl = I.encoder_workload("uneven", 1, d_model, 2, 24, 8, 3, vocab, compute="f32", optimizer="sgdm", alpha=0.01, K=4, D=0.5, steps=5, seed=vocab)
    params0 = I.init_encoder_params(wl)
    res = run_oracle(wl, params0, wl.steps)
    pipe, losses, book = run_gpu_pipeline(wl, params0, wl.steps, loop_order=order)
    np.testing.assert_allclose(losses, np.array(res.losses), rtol=1e-5)
    compare_params(pipe, res, 1e-5, bias_per_stage=True)


@pytest.mark.parametrize("order", ["tick_major", "mb_major"])
def test_widths(cuda_device, order):
    wl = I.mlp_workload("uneven", 3, 24, 2, "gelu", 19, compute="f32", optimizer="sgdm", alpha=0.01, K=4, D=0.5, steps=6, seed=9)
    widths = [24, 5, 330, 17, 64, 700, 24]
    wl.stages = [[I.LinearSpec(widths[2 * p + j], widths[2 * p + j + 1], "gelu") for j in range(2)] for p in range(3)]
    params0 = I.init_stage_params(wl)
    res = run_oracle(wl, params0, wl.steps)
    pipe, losses, book = run_gpu_pipeline(wl, params0, wl.steps, loop_order=order)
    np.testing.assert_allclose(losses, np.array(res.losses), rtol=1e-5)
    compare_params(pipe, res, 1e-5)
