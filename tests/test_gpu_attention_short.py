"""Attention of bf16 sequences shorter than the 128-row tile, with heads of 64: self-, causal and cross-attention."""
import numpy as np
import pytest

import pm_inputs as I
from parity_util import run_gpu_pipeline, run_oracle, compare_params

pytestmark = pytest.mark.gpu


# one token; a row group of the swizzle (8) and one past it; around the 32-row groups of the accumulator and the
# two 64-key halves; one below the full tile
@pytest.mark.parametrize("seq_len", [1, 8, 9, 31, 33, 64, 65, 96, 127])
def test_short_sequences(cuda_device, seq_len):
    wl = I.cfg5_small(compute="bf16", n_enc=1, n_dec=1, d_model=128, n_heads=2, d_ff=128, seq_len=seq_len, batch=3, vocab=64, steps=6)
    params0 = I.init_encoder_params(wl)
    res = run_oracle(wl, params0, wl.steps)
    pipe, losses, book = run_gpu_pipeline(wl, params0, wl.steps)
    np.testing.assert_allclose(losses, np.array(res.losses), rtol=1e-3)
    compare_params(pipe, res, 2e-2, per_stage=True)
