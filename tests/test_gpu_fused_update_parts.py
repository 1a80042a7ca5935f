"""The update kernel beside the fused update: a launch over the parts of the stages that the weight-gradient GEMM has left."""
import numpy as np
import pytest

import pm_inputs as I
from parity_util import run_gpu_pipeline

pytestmark = pytest.mark.gpu


# tables whose rows end inside a chunk of the launch, of few chunks (half as large) and of many; a single stage; stages that are a
# matrix and eight biases
@pytest.mark.parametrize("order", ["tick_major", "mb_major"])
@pytest.mark.parametrize("kind", ["small table", "large table", "one stage", "narrow"])
def test_same_bits_as_unfused(cuda_device, order, kind):
    import torch
    opt = dict(compute="bf16", optimizer="adam", alpha=1e-3, K=3, D=0.5, steps=4, seed=8)
    if kind.endswith("table"):
        wl = I.encoder_workload("parts", 1, 256, 4, 128, 16, 3, 1000 if kind == "small table" else 10008, **opt)
        params0 = I.init_encoder_params(wl)
    else:
        wl = I.mlp_workload("parts", 1, 264, 1, "relu", 24, **opt) if kind == "one stage" else I.mlp_workload("parts", 7, 8, 1, "gelu", 24, **opt)
        params0 = I.init_stage_params(wl)
    runs = [run_gpu_pipeline(wl, params0, wl.steps, loop_order=order, fuse_update=f) for f in (0, 1)]
    (plain, loss0, book0), (fused, loss1, book1) = runs
    np.testing.assert_array_equal(loss0, loss1)
    assert book0 == book1                                                    # the update counters
    for name in ("w", "m", "s", "delta"):
        assert torch.equal(getattr(plain, name), getattr(fused, name)), name
    if order == "tick_major":
        assert torch.equal(plain.w_lp, fused.w_lp)
