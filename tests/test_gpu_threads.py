"""Calls from several host threads, each with its own stream, buffers and workspace, whose sizes ask
for different amounts of shared memory of the same kernels."""
import threading

import numpy as np
import pytest

from .gpu_util import code_of, lib, to_dev

pytestmark = pytest.mark.gpu

# (n, p, s, sampling, pairs): samples of one CTA and of many, few and many buckets, one and both block sizes
CALLS = [(20_000, 2, 40, 1, False), (300_000, 8, 3000, 1, False), (120_000, 2000, 8, 1, False),
         (60_000, 2, 64, 0, False), (60_000, 600, 600, 0, False), (60_000, 16, 0, 1, True), (200_000, 1500, 6, 1, True)]


def test_threads_do_not_lower_each_others_limits():
    import torch
    bsps, rng = lib(), np.random.default_rng(1)
    calls = []
    for n, p, s, sampling, pairs in CALLS:
        keys = rng.integers(0, 2**31, n).astype(np.int32)
        kin, code, prm = to_dev(keys), code_of(keys), bsps.make_params(p, s=s, sampling=sampling, seed=2)
        val = torch.arange(n, dtype=torch.int32, device="cuda:0") if pairs else None
        ws = torch.empty(bsps.bsps_workspace_size(n, code, prm, pairs), dtype=torch.uint8, device="cuda:0")
        calls.append((keys, kin, torch.empty_like(kin), val, torch.empty_like(kin), code, prm,
                      torch.empty(p, dtype=torch.int64, device="cuda:0"), ws, torch.cuda.Stream()))
    torch.cuda.synchronize()
    bad, start = [], threading.Barrier(len(calls))

    def work(c):
        keys, kin, kout, val, vout, code, prm, sizes, ws, stream = c
        start.wait()
        for _ in range(300):
            if val is None:
                rc = bsps.bsps_sort_keys(kin, kout, len(keys), code, prm, sizes, ws, stream=stream)
            else:
                rc = bsps.bsps_sort_pairs(kin, val, kout, vout, len(keys), code, prm, sizes, ws, stream=stream)
            if rc:
                bad.append((len(keys), prm.p, rc))
                return

    threads = [threading.Thread(target=work, args=(c,)) for c in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not bad, bad
    for keys, _, kout, val, vout, _, _, _, ws, _ in calls:
        assert bsps.bsps_read_stats(ws).status == 0
        assert kout.cpu().numpy().tobytes() == np.sort(keys).tobytes()
        assert val is None or np.array_equal(vout.cpu().numpy(), np.argsort(keys, kind="stable"))
