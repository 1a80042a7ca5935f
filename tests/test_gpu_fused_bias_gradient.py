"""fuse_update: the bias gradients are in the gradient arena after pm_backward, with the bits of an unfused run, and the update takes what
stands there then (a program may change them between the two phases)."""
import numpy as np
import pytest

import pm_inputs as I

pytestmark = pytest.mark.gpu


# rows below, at and beyond 64 and 512 (one 64-row block, eight of them); widths that leave remainders in blocks of 32 and tiles of 128 and 256
@pytest.mark.parametrize("order", ["tick_major", "mb_major"])
@pytest.mark.parametrize("width,T", [(8, 1), (40, 63), (136, 65), (264, 512), (328, 577), (1032, 1100)])
def test_bias_gradients_after_the_backward_phase(cuda_device, order, width, T):
    import torch
    import paper_1910_05124_b200 as pm
    wl = I.mlp_workload("fb", 3, width, 1, "relu", T, compute="bf16", optimizer="sgdm", alpha=0.01, K=4, D=0.5, steps=9, seed=191005124 + width)
    params0 = I.init_stage_params(wl)
    gen = torch.Generator(device="cuda").manual_seed(width + T)
    rnd = lambda *shape: torch.randn(*shape, generator=gen, device="cuda")
    pipes = [pm.Pipeline(wl, params0, loop_order=order, fuse_update=f) for f in (0, 1)]
    seen = 0
    for step in range(wl.steps):                                    # beyond the two steps that run as plain launches
        x, y = rnd(T, width).bfloat16(), rnd(T, width)
        for pipe in pipes:
            pipe.pm_forward(x, y)
            pipe.pm_backward()
        plain, fused = (pipe.unpack(pipe.grad) for pipe in pipes)
        for p in range(wl.n_stages):
            np.testing.assert_array_equal(fused[p][0][1], plain[p][0][1])
            seen += int(np.abs(plain[p][0][1]).max() > 0)
        for pipe in pipes:
            for p in range(wl.n_stages):                            # the program doubles the bias gradients before the update
                o = pipe.stage_desc[p].param_offset + pipe.layout[p][1][1]
                pipe.grad[o:o + width] *= 2
            pipe.pm_update()
        assert torch.equal(pipes[0].w, pipes[1].w) and torch.equal(pipes[0].m, pipes[1].m)
    assert seen >= wl.n_stages
