"""Training of the learned classifier is a fixed sequence of sums: every run on the same keys gives
the same parameters and losses, bit for bit, whatever the order in which CTAs and warps finish."""
import numpy as np
import pytest

import bsp_inputs as gen
import oracle

from .gpu_util import run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, p, s", [(1 << 18, 256, 16), (40_000, 8, 3)])
def test_trained_parameters_repeat(n, p, s):
    keys = gen.gmm(n, seed=4)
    first = run_gpu(keys, p, s, 0, oracle.RANDOM, 8, classify=1, debug=False)
    assert np.isfinite(first.mlp_params).all() and first.mlp_loss[1] <= first.mlp_loss[0]
    for _ in range(40):
        again = run_gpu(keys, p, s, 0, oracle.RANDOM, 8, classify=1, debug=False)
        assert again.mlp_params.tobytes() == first.mlp_params.tobytes()
        assert again.mlp_loss.tobytes() == first.mlp_loss.tobytes()
        assert (again.stats.mispredicted, again.stats.correction_steps) == (first.stats.mispredicted, first.stats.correction_steps)
