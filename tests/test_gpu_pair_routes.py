"""Random pairs of 4-byte keys at the sizes where both routes are queued and the device takes one by
how often the sample's keys repeat: each route's inputs, the edge between them, sub-buckets of one value
and of many, and those that only the out-of-core sort takes, stably."""
import numpy as np
import pytest

import bsp_inputs as gen
import oracle

from .gpu_util import assert_same, run_gpu

pytestmark = pytest.mark.gpu


def values(n, kind, seed):
    rng = np.random.default_rng(seed)
    if kind == "distinct":
        return rng.permutation(n).astype(np.int64) * 17 - 5
    if kind == "one":
        return np.full(n, -7)
    if kind == "zipf":
        return gen.zipf(n, seed=seed)
    share, count = kind  # a share of the keys on `count` values
    return np.where(rng.random(n) < share, rng.integers(0, count, n) * 1_000_003, rng.integers(-2**31, 2**31, n))


@pytest.mark.parametrize("n, p", [(65_536, 2), (70_001, 1), (300_003, 8), (1 << 23, 2048)])
@pytest.mark.parametrize("kind", ["distinct", "one", "zipf", (1.0, 3), (0.94, 20), (0.955, 20), (0.97, 20)], ids=str)
def test_both_routes(n, p, kind):
    keys = values(n, kind, n).astype(np.int32)
    vals = np.random.default_rng(1).integers(0, 2**32, n).astype(np.uint32)
    for dt, classify in ((np.int32, 0), (np.float32, 0), (np.uint32, 1)):
        k = keys.astype(dt) if dt == np.float32 else keys.view(dt)
        ref = oracle.sort(k, p, 0, 0, oracle.RANDOM, seed=5, vals=vals, want_sample=False)
        assert_same(run_gpu(k, p, 0, 0, oracle.RANDOM, 5, vals, debug=False, classify=classify), ref)
        if n >= 1 << 23:
            return  # one type is enough there


@pytest.mark.parametrize("kind", ["distinct", (1.0, 3), (1.0, 200_000), "zipf"], ids=str)
def test_out_of_core(kind):
    n = 400_000
    keys = values(n, kind, 3).astype(np.int32)
    vals = np.arange(n, dtype=np.uint32)
    ref = oracle.sort(keys, 2, 0, 0, oracle.RANDOM, seed=5, vals=vals, want_sample=False)
    assert_same(run_gpu(keys, 2, 0, 0, oracle.RANDOM, 5, vals, refine=1, debug=False), ref)


def test_regular_sample_with_the_learned_classifier():
    n = 1 << 18
    for kind in ("distinct", "zipf"):
        keys, vals = values(n, kind, 4).astype(np.int32), np.arange(n, dtype=np.uint32)
        ref = oracle.sort(keys, 4, 64, 0, oracle.REGULAR, seed=5, vals=vals, want_sample=False)
        assert_same(run_gpu(keys, 4, 64, 0, oracle.REGULAR, 5, vals, debug=False, classify=1), ref)
