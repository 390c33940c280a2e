"""Batches whose instances go through several launches: few on-chip instances of mixed sizes, waves that
reuse one workspace, regular sampling's recorded graph on later calls, and a call that does not wait for
the stream's earlier work."""
import time

import numpy as np
import pytest

import bsp_inputs as gen
import oracle

from .gpu_util import lib, to_dev
from .test_gpu_batched import _batch, _check, _run_batched

pytestmark = pytest.mark.gpu


# one launch for few instances, one per shape for many; short lists of jobs and uploaded ones
@pytest.mark.parametrize("count", [1, 2, 31, 32, 33, 150, 153, 200])
@pytest.mark.parametrize("hi", [9, 12, 13, 14])
def test_on_chip_instances(count, hi):
    bsps, rng = lib(), np.random.default_rng(count)
    sizes = [int(2 ** rng.uniform(0, hi)) for _ in range(count - 1)] + [1 << hi]
    keys, off = _batch(sizes, count)
    prm, tune = bsps.make_params(1, sampling=bsps.BSPS_RANDOM, seed=5), bsps.bsps_tune_default()
    tune.p[9], tune.p[11], tune.p[13] = 3, 8, 16
    out, bsz, base, _ = _run_batched(keys, off, prm, tune)
    for i in range(count):
        a, b = off[i], off[i + 1]
        p = base[i + 1] - base[i]
        ref = oracle.sort(keys[a:b], p, 0, 0, oracle.RANDOM, seed=5 + i, want_sample=False)
        assert out[a:b].tobytes() == ref.keys.tobytes() and np.array_equal(bsz[base[i]:base[i + 1]], ref.bucket_sizes)


def test_few_mixed_instances_run_in_one_launch_s_time():
    """As many CTAs as instances, none waiting for another shape's: a few of mixed sizes take about as long as the largest."""
    import torch
    bsps = lib()

    def least_us(sizes):
        off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
        kin = to_dev(gen.uniform(int(off[-1]), 1, 3))
        kout, prm, tune = torch.empty_like(kin), bsps.make_params(1, sampling=bsps.BSPS_RANDOM, seed=5), bsps.bsps_tune_default()
        ws = torch.empty(bsps.bsps_batch_workspace_size(off, bsps.BSPS_I32, prm, tune), dtype=torch.uint8, device="cuda:0")
        best = float("inf")
        for _ in range(20):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda._sleep(200_000)  # the launches are queued behind it: no host time between the events
            a.record()
            assert bsps.bsps_sort_batched(kin, kout, off, bsps.BSPS_I32, prm, tune, None, ws) == 0
            b.record()
            torch.cuda.synchronize()
            best = min(best, 1e3 * a.elapsed_time(b))
        return best

    mixed, one = least_us([300, 2000, 3500, 4097, 6000, 8000, 9000, 16_000] * 3), least_us([16_000])
    print(f"24 instances of mixed sizes {mixed:.0f} us, the largest alone {one:.0f} us")
    assert mixed <= 1.5 * one, (mixed, one)


def test_waves_reuse_the_workspace():
    """One lane: its workspace holds one wave of some of the instances, so later waves start on what earlier ones left."""
    bsps = lib()
    rng = np.random.default_rng(4)
    sizes = [1 << 20] * 6 + [1 << 22, 300_000, 1 << 21, 17_000, 5000] + [int(2 ** rng.uniform(17, 21)) for _ in range(24)]
    keys, off = _batch(sizes, 71)
    prm, tune = bsps.make_params(1, sampling=bsps.BSPS_RANDOM, seed=7), bsps.bsps_tune_default()
    tune.lanes, tune.learned_min_log2 = 1, 20
    need = [bsps.bsps_workspace_size(n, bsps.BSPS_I32, bsps.make_params(tune.p[20], sampling=bsps.BSPS_RANDOM, classify=1)) for n in sizes]
    assert sum(need) > 2.5 * bsps.bsps_batch_workspace_size(off, bsps.BSPS_I32, prm, tune)
    out, bsz, base, bufs = _run_batched(keys, off, prm, tune)
    _check(keys, off, out, bsz, base, prm, tune, oracle_max=0)
    keys2, _ = _batch(sizes, 81)
    out, bsz, base, _ = _run_batched(keys2, off, prm, tune, reuse=bufs)
    _check(keys2, off, out, bsz, base, prm, tune, oracle_max=0)


def test_an_early_wave_s_overflow_is_reported():
    """Regions 4 % above the mean: some of the first instance's 64 buckets overflow, the later ones' only bucket cannot."""
    import torch
    bsps = lib()
    prm, tune = bsps.make_params(1, sampling=bsps.BSPS_RANDOM, seed=7, capacity_pct=104), bsps.bsps_tune_default()
    tune.lanes, tune.p[16], tune.p[20] = 1, 1, 64
    for first, overflow in ((1 << 20, 1), (60_000, 0)):
        off = np.concatenate([[0], np.cumsum([first] + [60_000] * 400)]).astype(np.int64)
        need = bsps.bsps_batch_workspace_size(off, bsps.BSPS_I32, prm, tune)
        assert need < 0.7 * 400 * bsps.bsps_workspace_size(60_000, bsps.BSPS_I32, prm)  # several waves
        ws = torch.empty(need, dtype=torch.uint8, device="cuda:0")
        kin = to_dev(gen.uniform(int(off[-1]), 1, 3))
        assert bsps.bsps_sort_batched(kin, torch.empty_like(kin), off, bsps.BSPS_I32, prm, tune, None, ws) == 0
        st = bsps.bsps_read_stats(ws)
        assert (st.status, st.overflow) == (bsps.BSPS_ERR_BUCKET_OVERFLOW if overflow else 0, overflow)


def test_regular_batch_graph_sees_new_keys_and_offsets():
    bsps = lib()
    prm, tune = bsps.make_params(1, sampling=bsps.BSPS_REGULAR), bsps.bsps_tune_default()
    for c in range(32):
        tune.p[c] = 4
    sizes = [3000, 70_000, 20_000, 0, 1, 150_000, 9000, 40_000, 5, 12_345]
    keys, off = _batch(sizes, 41)
    out, bsz, base, bufs = _run_batched(keys, off, prm, tune)
    _check(keys, off, out, bsz, base, prm, tune)
    keys2, _ = _batch(sizes, 51)  # the same call on new keys: the recorded graph again
    out, bsz, base, _ = _run_batched(keys2, off, prm, tune, reuse=bufs)
    _check(keys2, off, out, bsz, base, prm, tune, oracle_max=0)
    sizes[1], sizes[2] = sizes[2], sizes[1]  # other offsets in the same buffers: recorded anew
    keys3, off3 = _batch(sizes, 61)
    out, bsz, base, _ = _run_batched(keys3, off3, prm, tune, reuse=bufs)
    _check(keys3, off3, out, bsz, base, prm, tune, oracle_max=0)


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
