"""The out-of-core tiers of the final sort and what slow_buckets counts: a sub-bucket past a cluster's
shared memory, sorted in parts by the counting sort, and what that gives back (more than 65,535 keys in
one of its bins) and a cluster cannot hold, sorted by radix passes."""
import numpy as np
import pytest

import oracle

from .gpu_util import code_of, lib, to_dev

pytestmark = pytest.mark.gpu


def call(keys, p, vals=None, **kw):
    """(keys, payloads, statistics, sub-buckets on the list of the radix passes: DevStatus::slow_count of csrc/common.cuh)"""
    import torch
    bsps, n, code = lib(), len(keys), code_of(keys)
    prm = bsps.make_params(p, sampling=bsps.BSPS_RANDOM, seed=9, refine=1, **kw)
    ws = torch.empty(bsps.bsps_workspace_size(n, code, prm, vals is not None), dtype=torch.uint8, device="cuda:0")
    kin = to_dev(keys)
    kout, vout = torch.empty_like(kin), None
    if vals is None:
        assert bsps.bsps_sort_keys(kin, kout, n, code, prm, None, ws) == 0
    else:
        vin = to_dev(vals)
        vout = torch.empty_like(vin)
        assert bsps.bsps_sort_pairs(kin, vin, kout, vout, n, code, prm, None, ws) == 0
    st = bsps.bsps_read_stats(ws)
    return (kout.cpu().numpy().view(keys.dtype), None if vals is None else vout.cpu().numpy().view(np.uint32), st,
            int(ws[:64].view(torch.int32)[15].item()))


def check(keys, vals, got):
    order = np.argsort(keys, kind="stable")
    assert got[2].status == 0 and got[0].tobytes() == keys[order].tobytes()
    assert vals is None or np.array_equal(got[1], vals[order])


@pytest.mark.parametrize("pairs", [False, True], ids=["keys", "pairs"])
@pytest.mark.parametrize("dt", [np.int32, np.float64])
def test_even_bucket_in_parts(dt, pairs):
    keys = np.random.default_rng(1).permutation(300_000).astype(dt)
    vals = np.arange(len(keys), dtype=np.uint32) if pairs else None
    got = call(keys, 1, vals)
    check(keys, vals, got)
    assert got[2].slow_buckets == 1
    assert got[3] == (1 if pairs and dt == np.float64 else 0)  # doubles with payloads have no counting sort


@pytest.mark.parametrize("pairs", [False, True], ids=["keys", "pairs"])
@pytest.mark.parametrize("dt", [np.int32, np.float64])
def test_radix_passes(dt, pairs):
    rng = np.random.default_rng(2)
    keys = np.where(rng.random(400_000) < 0.4, 12_345, rng.integers(-2**31, 2**31, 400_000)).astype(dt)
    vals = np.arange(len(keys), dtype=np.uint32) if pairs else None
    got = call(keys, 1, vals)
    check(keys, vals, got)
    assert (got[2].slow_buckets, got[3]) == (1, 1)


def test_a_bucket_that_a_cluster_holds_is_not_counted():
    rng = np.random.default_rng(3)
    keys = np.where(rng.random(100_000) < 0.3, 77, rng.integers(-2**31, 2**31, 100_000)).astype(np.int32)
    vals = np.arange(len(keys), dtype=np.uint32)
    got = call(keys, 8, vals, duplicates=1, capacity_pct=500)
    check(keys, vals, got)
    assert got[2].max_vbucket > 40_000 and got[2].slow_buckets == 0


def test_expired_look_back_wait_of_doubles_with_payloads():
    """On the route that a plain call of doubles with payloads takes: the wait that runs out is reported, and the
    same call without the hooks, on the same workspace, is exact."""
    import torch
    bsps, n, p = lib(), 300_000, 16
    keys, vals = np.random.default_rng(4).normal(0, 1, n), np.arange(n, dtype=np.uint32)
    prm = bsps.make_params(p, sampling=bsps.BSPS_RANDOM, seed=3, refine=1)
    pl = bsps.bsps_get_plan(n, bsps.BSPS_F64, prm, True)
    assert pl.route_tiles >= 3
    ws = torch.empty(pl.workspace_bytes, dtype=torch.uint8, device="cuda:0")
    kin, vin = to_dev(keys), to_dev(vals)
    kout, vout, sizes = torch.empty_like(kin), torch.empty_like(vin), torch.empty(p, dtype=torch.int64, device="cuda:0")
    assert bsps.bsps_sort_debug(kin, vin, kout, vout, n, bsps.BSPS_F64, prm, sizes, ws, stall_tile=2, wait_polls=2000) == 0
    st = bsps.bsps_read_stats(ws)
    assert st.status == bsps.BSPS_ERR_DEVICE_TIMEOUT and st.timeouts >= 1
    assert bsps.bsps_sort_pairs(kin, vin, kout, vout, n, bsps.BSPS_F64, prm, sizes, ws) == 0
    st = bsps.bsps_read_stats(ws)
    assert (st.status, st.timeouts) == (0, 0)
    ref = oracle.sort(keys, p, 0, 0, oracle.RANDOM, seed=3, vals=vals, want_sample=False)
    assert kout.cpu().numpy().tobytes() == ref.keys.tobytes() and np.array_equal(vout.cpu().numpy().view(np.uint32), ref.vals)
    assert np.array_equal(sizes.cpu().numpy(), ref.bucket_sizes)
