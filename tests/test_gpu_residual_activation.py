"""bf16 residual stages whose Linear has an activation: out = bf16(skip + bf16(act(z))), on every forward kernel."""
import numpy as np
import pytest

import pm_inputs as I
from parity_util import run_gpu_pipeline, run_oracle, compare_params


def workload(heads, batch, act, steps):
    wl = I.encoder_workload("resact", 1, 64 * heads, heads, 128 * heads, 128, batch, 264, compute="bf16", optimizer="sgdm", alpha=0.05,
                            beta1=0.9, K=4, D=0.5, steps=steps, seed=191005124 + 61)
    for sp in wl.stage_specs:
        if sp.post == "residual":
            sp.act = act
    return wl


# Tiles of 128 rows x 64 columns decide (296 is the most the kernel for few tiles takes): of all five stages in a tick, of one in
# microbatch-major order.  2 sequences: few tiles; 3 heads: one-CTA kernel, widths of 192; 4 heads: CTA pairs.
@pytest.mark.gpu
@pytest.mark.parametrize("order,heads,batch,steps", [("tick_major", 3, 2, 6), ("tick_major", 3, 13, 6), ("tick_major", 4, 13, 6), ("mb_major", 3, 2, 6),
                                                     ("mb_major", 3, 100, 2), ("mb_major", 4, 76, 2)])
@pytest.mark.parametrize("act", ["relu", "gelu"])
def test_against_oracle(cuda_device, order, heads, batch, steps, act):
    wl = workload(heads, batch, act, steps)
    params0 = I.init_encoder_params(wl)
    res = run_oracle(wl, params0, wl.steps)
    pipe, losses, _ = run_gpu_pipeline(wl, params0, wl.steps, loop_order=order)
    np.testing.assert_allclose(losses, np.array(res.losses), rtol=1e-3)      # the bf16 path's tolerances up to a dozen layers
    compare_params(pipe, res, 2e-2, bias_per_stage=True)                     # (biases are a few steps in size)
