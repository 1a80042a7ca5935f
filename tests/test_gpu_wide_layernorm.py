"""LayerNorm stages wider than the fused backward kernel holds (1024), with rows enough for partial sums: their gradients
and the bias gradients, which are summed by column as well, against the oracle."""
import numpy as np
import pytest

import pm_inputs as I
from oracle import transformer

pytestmark = pytest.mark.gpu


# widths just above 1024 and of whole 256-column blocks; ten row chunks and a ragged eighteenth
@pytest.mark.parametrize("d_model,n_heads,batch", [(1032, 12, 40), (1280, 20, 69)])
@pytest.mark.parametrize("order,segment", [("mb_major", 0), ("mb_major", 2), ("tick_major", 0)])
def test_gradients(cuda_device, d_model, n_heads, batch, order, segment):
    import torch
    import paper_1910_05124_b200 as pm
    wl = I.encoder_workload("wide_ln", 1, d_model, n_heads, 256, 16, batch, 96, compute="bf16", optimizer="sgdm", alpha=0.0, K=4, D=0.5,
                            steps=1, seed=d_model)
    params0 = I.init_encoder_params(wl)
    data = lambda t: I.token_batch(wl, 0)
    ref_loss, ref = transformer.make_grad_fn(wl.stage_specs, data, n_heads, 16, 96, "bf16")(0, params0, params0)
    pipe = pm.Pipeline(wl, params0, loop_order=order, recompute_segment=segment)
    ids, tg = (torch.from_numpy(a.astype(np.int32)).cuda() for a in data(0))
    P = wl.n_stages
    for _ in range(1 if order == "mb_major" else 2 * P):      # the same microbatch in every slot, and weights that do not move
        pipe.pm_step(ids, tg)
    got = pipe.unpack(pipe.grad)
    assert abs(pipe.pm_get_losses(0, 1)[0] - ref_loss) <= 1e-3 * ref_loss
    for p, sp in enumerate(wl.stage_specs):
        for j, a in enumerate(got[p]):
            r = np.asarray(ref[p][j], dtype=np.float64)
            if sp.post == "attention" and j == len(got[p]) - 1:
                r[d_model:2 * d_model] = a[d_model:2 * d_model]          # the key bias: exactly zero but for rounding noise
            # a gradient passes at most a dozen roundings of 2^-9 in five stages; sums in another order flip some of them
            assert np.linalg.norm(a - r) <= 2e-2 * np.linalg.norm(r), (p, j)
