"""A batch's call does not wait for the stream's earlier work."""
import time

import numpy as np
import pytest

import bsp_inputs as gen
from .gpu_util import lib, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[3000] * 3000, [40_000] * 150], ids=["on_chip", "larger"])
def test_the_call_does_not_wait_for_the_stream(sizes):
    import torch
    bsps = lib()
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    keys = gen.uniform(int(off[-1]), 1, 3)
    kin = to_dev(keys)
    kout, prm, tune = torch.empty_like(kin), bsps.make_params(1, sampling=bsps.BSPS_RANDOM, seed=5), bsps.bsps_tune_default()
    ws = torch.empty(bsps.bsps_batch_workspace_size(off, bsps.BSPS_I32, prm, tune), dtype=torch.uint8, device="cuda:0")
    assert bsps.bsps_sort_batched(kin, kout, off, bsps.BSPS_I32, prm, tune, None, ws) == 0
    torch.cuda.synchronize()
    kout.zero_()
    torch.cuda._sleep(400_000_000)  # about 0.2 s
    t = time.perf_counter()
    assert bsps.bsps_sort_batched(kin, kout, off, bsps.BSPS_I32, prm, tune, None, ws) == 0
    took = time.perf_counter() - t
    torch.cuda.synchronize()
    out = kout.cpu().numpy()
    for i in range(0, len(sizes), 17):
        assert out[off[i]:off[i + 1]].tobytes() == np.sort(keys[off[i]:off[i + 1]]).tobytes()
    assert took < 0.1, took
