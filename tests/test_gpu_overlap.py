"""Pairs whose outputs take the place of an input.  Input equal to its own output is refused; any
other overlap was always sorted exactly, because every input is read before an output is written:
the paths that read an input late (payloads fetched by position, whole sorts on chip) leave such
calls to those that do not."""
import numpy as np
import pytest

import oracle

from .gpu_util import code_of, lib, to_dev

pytestmark = pytest.mark.gpu

# where each buffer starts in one arena, in units of n words: keys in, payloads in, keys out, payloads out
PLACES = {
    "keys_out_is_vals_in": (0, 1, 1, 2),
    "vals_out_is_keys_in": (0, 1, 2, 0),
    "exchanged": (0, 1, 1, 0),
    "keys_out_half_on_vals_in": (0, 1, 1.5, 3),
    "vals_out_half_on_vals_in": (0, 1, 2.5, 1.5),
    "keys_out_half_on_keys_in": (0, 2, 0.5, 3),
}


def arena(n, places, arrays):
    import torch
    a = torch.zeros(5 * n + 64, dtype=torch.int32, device="cuda:0")
    views = [a[int(at * n) // 4 * 4:][:n] for at in places]
    for v, x in zip(views, arrays):
        v.copy_(to_dev(x).view(torch.int32))
    return views


@pytest.mark.parametrize("classify", [0, 1])
@pytest.mark.parametrize("n, p, values", [(3000, 4, 2**31), (16_384, 16, 50), (60_000, 8, 2**31), (700_000, 64, 2**31), (300_000, 8, 9)])
@pytest.mark.parametrize("place", sorted(PLACES))
def test_pairs(place, n, p, values, classify):
    import torch
    if classify and n < 50_000:
        pytest.skip("the learned classifier is compared at the larger sizes")
    bsps, rng = lib(), np.random.default_rng(n)
    keys, vals = rng.integers(0, values, n).astype(np.int32), rng.integers(0, 2**32, n).astype(np.uint32)
    prm = bsps.make_params(p, sampling=bsps.BSPS_RANDOM, seed=9, classify=classify)
    ws = torch.empty(bsps.bsps_workspace_size(n, code_of(keys), prm, True), dtype=torch.uint8, device="cuda:0")
    sizes = torch.full((p,), -1, dtype=torch.int64, device="cuda:0")
    kin, vin, kout, vout = arena(n, PLACES[place], (keys, vals))
    assert bsps.bsps_sort_pairs(kin, vin, kout, vout, n, code_of(keys), prm, sizes, ws) == 0
    ref = oracle.sort(keys, p, 0, 0, oracle.RANDOM, seed=9, vals=vals, want_sample=False)
    assert bsps.bsps_read_stats(ws).status == 0
    assert kout.cpu().numpy().tobytes() == ref.keys.tobytes()
    assert np.array_equal(vout.cpu().numpy().view(np.uint32), ref.vals)
    assert np.array_equal(sizes.cpu().numpy(), ref.bucket_sizes)


@pytest.mark.parametrize("n, p", [(3000, 4), (16_384, 1), (60_000, 8)])
def test_keys(n, p):
    import torch
    bsps, rng = lib(), np.random.default_rng(n)
    keys = rng.integers(0, 2**31, n).astype(np.int32)
    prm = bsps.make_params(p, sampling=bsps.BSPS_RANDOM, seed=9)
    ws = torch.empty(bsps.bsps_workspace_size(n, code_of(keys), prm), dtype=torch.uint8, device="cuda:0")
    sizes = torch.full((p,), -1, dtype=torch.int64, device="cuda:0")
    kin, kout = arena(n, (0, 0.5), (keys,))
    assert bsps.bsps_sort_keys(kin, kout, n, code_of(keys), prm, sizes, ws) == 0
    ref = oracle.sort(keys, p, 0, 0, oracle.RANDOM, seed=9, want_sample=False)
    assert bsps.bsps_read_stats(ws).status == 0
    assert kout.cpu().numpy().tobytes() == ref.keys.tobytes()
    assert np.array_equal(sizes.cpu().numpy(), ref.bucket_sizes)


@pytest.mark.parametrize("n", [3000, 60_000])
def test_bucket_sizes_on_vals_in(n):
    import torch
    bsps, rng, p = lib(), np.random.default_rng(n), 8
    keys, vals = rng.integers(0, 2**31, n).astype(np.int32), rng.integers(0, 2**32, n).astype(np.uint32)
    prm = bsps.make_params(p, sampling=bsps.BSPS_RANDOM, seed=9)
    ws = torch.empty(bsps.bsps_workspace_size(n, code_of(keys), prm, True), dtype=torch.uint8, device="cuda:0")
    kin, vin, kout, vout = arena(n, (0, 1, 2, 3), (keys, vals))
    sizes = vin[n // 2 & ~1:][:2 * p].view(torch.int64)
    assert bsps.bsps_sort_pairs(kin, vin, kout, vout, n, code_of(keys), prm, sizes, ws) == 0
    ref = oracle.sort(keys, p, 0, 0, oracle.RANDOM, seed=9, vals=vals, want_sample=False)
    assert bsps.bsps_read_stats(ws).status == 0
    assert np.array_equal(vout.cpu().numpy().view(np.uint32), ref.vals)
    assert np.array_equal(sizes.cpu().numpy(), ref.bucket_sizes)
