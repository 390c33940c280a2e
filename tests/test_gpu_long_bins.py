"""The counting sort's bins that hold one value many times and a few other keys, or two such values:
around the sizes at which a warp, its registers, the CTA and the CTA's pivots take over."""
import numpy as np
import pytest

import oracle

from .gpu_util import assert_same, run_gpu

pytestmark = pytest.mark.gpu

V = 1 << 29


def keys_of(c, others, seed, second=0):
    """c copies of V, `others` keys next to it (in V's bin), `second` copies of a value between, and 2000 spread keys."""
    rng = np.random.default_rng(seed)
    near = V + np.setdiff1d(np.arange(-others, others + 1), [0])[rng.permutation(2 * others)[:others]]
    k = np.concatenate([np.full(c, V), near, np.full(second, V + 1), rng.integers(0, 1 << 30, 2000), [0, (1 << 30) - 1]])
    return rng.permutation(k)


@pytest.mark.parametrize("c", [20, 60, 250, 300, 1020, 8000, 8300, 30_000])
@pytest.mark.parametrize("others", [0, 1, 31, 32, 33, 200, 511, 512, 513, 900])
def test_one_value_and_others(c, others):
    keys = keys_of(c, others, c + others)
    for dt in (np.int32, np.float64):
        k = keys.astype(dt)
        ref = oracle.sort(k, 1, 0, 0, oracle.RANDOM, seed=5, want_sample=False)
        got = run_gpu(k, 1, 0, 0, oracle.RANDOM, 5, refine=1, debug=False)
        assert got.keys.tobytes() == ref.keys.tobytes()


@pytest.mark.parametrize("c, second", [(40, 30), (200, 200), (600, 300), (3000, 3000), (5000, 2900), (5000, 9000), (20_000, 18_000)])
@pytest.mark.parametrize("pairs", [False, True], ids=["keys", "pairs"])
def test_two_values_in_a_bin(c, second, pairs):
    keys = keys_of(c, 40, c, second).astype(np.int32)
    vals = np.random.default_rng(c).integers(0, 2**32, len(keys)).astype(np.uint32) if pairs else None
    ref = oracle.sort(keys, 1, 0, 0, oracle.RANDOM, seed=5, vals=vals, want_sample=False)
    assert_same(run_gpu(keys, 1, 0, 0, oracle.RANDOM, 5, vals, refine=1, debug=False), ref)


# samples that repeat records (more draws than keys), around the one-CTA size
@pytest.mark.parametrize("n, p, s", [(30, 3, 900), (500, 8, 1024), (2000, 2, 4096), (9, 2, 4000)])
def test_sample_of_repeated_records(n, p, s):
    keys = np.random.default_rng(n).integers(0, 2**31, n).astype(np.int32)
    ref = oracle.sort(keys, p, s, 0, oracle.RANDOM, seed=3, want_sample=True)
    assert_same(run_gpu(keys, p, s, 0, oracle.RANDOM, 3), ref)


# ... of far more draws than keys, bins of one record and of several past 65,535 copies, and bins that take radix passes
@pytest.mark.parametrize("n, p, s, dt", [(10, 2, 1_000_000, np.int32), (10, 2, 1_000_000, np.float64), (40, 1, 8_000_000, np.int32),
                                         (3000, 16, 100_000, np.int32), (3000, 16, 100_000, np.float64), (700, 2, 13_000_000, np.float64)])
def test_sample_much_larger_than_the_input(n, p, s, dt):
    keys = np.random.default_rng(n).integers(-2**31, 2**31, n).astype(dt)
    keys[: n // 3] = keys[0]
    ref = oracle.sort(keys, p, s, 0, oracle.RANDOM, seed=3, want_sample=False)
    got = run_gpu(keys, p, s, 0, oracle.RANDOM, 3, debug=False)
    assert got.keys.tobytes() == ref.keys.tobytes() and np.array_equal(got.bucket_sizes, ref.bucket_sizes)
