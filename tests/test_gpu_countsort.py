"""The streamed counting sort of the keys-only final step (Fig. 2 step 12) at the sizes and
value distributions where it can go wrong: part edges, several CTAs per bucket, bins that hold
many keys, repeated keys, and keys of every type, each against the oracle, element by element."""
import numpy as np
import pytest

import oracle

from .gpu_util import assert_same, run_gpu

pytestmark = pytest.mark.gpu


def same(gpu, ref):
    assert gpu.keys.tobytes() == ref.keys.tobytes()
    assert np.array_equal(gpu.bucket_sizes, ref.bucket_sizes)


def check(keys, p, s=0):
    ref = oracle.sort(keys, p, s, 0, oracle.RANDOM, seed=5, want_sample=False)
    same(run_gpu(keys, p, s, 0, oracle.RANDOM, 5, refine=1, debug=False), ref)


# around a shape's stage (8192, 18944 and 38912 keys of 4 bytes, half of 8), one part more, 16-byte remainders
@pytest.mark.parametrize("dt", [np.int32, np.float64])
@pytest.mark.parametrize("n", [1, 2, 255, 1023, 4088, 4097, 8184, 8193, 9464, 9473, 18936, 18945, 38904, 38913, 77_817, 120_003])
def test_one_bucket(n, dt):
    rng = np.random.default_rng(n)
    keys = rng.integers(-2**31, 2**31, n).astype(np.int32) if dt == np.int32 else rng.normal(0, 1, n)
    check(keys, 1)


# half-word stages: few units of 2^15 (2^31) values, one and two parts, most keys in one half of the bins,
# windows over more than two units
@pytest.mark.parametrize("n", [38_905, 65_001, 65_540, 77_816, 77_821, 150_000])
@pytest.mark.parametrize("span_log2", [16, 18, 21, 23])
@pytest.mark.parametrize("shape", ["even", "low", "high", "gaps"])
def test_half_word_stage(n, span_log2, shape):
    rng = np.random.default_rng(n + span_log2)
    j = rng.integers(0, 1 << span_log2, n)
    if shape == "low":
        j = np.where(rng.random(n) < 0.97, j >> 2, j)
    elif shape == "high":
        j = (1 << span_log2) - 1 - np.where(rng.random(n) < 0.97, j >> 2, j)
    elif shape == "gaps":
        j = j & ~(1 << (span_log2 - 2)) & ~(1 << (span_log2 - 4))
    check((j - 5_000_000).astype(np.int32), 1)
    check(3.0 + j * 2.0**-37, 1)  # 2^15 consecutive doubles from one to the next


@pytest.mark.parametrize("p", [2, 7, 200])
def test_several_ctas_per_bucket(p):
    check(np.random.default_rng(p).integers(0, 2**31, 200_003).astype(np.int32), p)


SHAPES = {
    "two_values": lambda r, n: r.choice([7, 2**30], n),
    "one_heavy_value": lambda r, n: np.where(r.random(n) < 0.6, 12345, r.integers(0, 2**31, n)),
    "repeats_of_17_to_2000": lambda r, n: np.repeat(r.integers(0, 2**31, n), r.choice([1, 17, 40, 300, 1500, 2000], n))[:n],
    "dense_runs": lambda r, n: (r.integers(0, 64, n) << 24) + r.integers(0, 300, n),
    "halving": lambda r, n: (2.0**31 * 2.0 ** -(20 * r.random(n))).astype(np.int64) - 1,
    "consecutive": lambda r, n: np.arange(n),
    "descending": lambda r, n: 2**31 - 1 - 3 * np.arange(n),
    "all_ones_bits": lambda r, n: r.choice([-1, -2, 2**31 - 1, -(2**31)], n),
}


@pytest.mark.parametrize("p", [1, 3])
@pytest.mark.parametrize("n", [5000, 30_011, 90_000])
@pytest.mark.parametrize("name", sorted(SHAPES))
def test_skewed_bins(name, n, p):
    keys = SHAPES[name](np.random.default_rng(n), n)
    check(keys.astype(np.int32), p)
    check(keys.astype(np.float64) * 2.0**-20, p)


# blocks of the regular sample (Fig. 1 step 3): block sizes that are no multiple of 4, one and several CTAs a block
@pytest.mark.parametrize("n, p, s", [(10_007, 1, 50), (65_536, 8, 64), (150_001, 2, 30), (163_839, 2, 4096), (400_003, 100, 100)])
@pytest.mark.parametrize("dt", [np.int32, np.float32])
def test_blocks(n, p, s, dt):
    rng = np.random.default_rng(n)
    keys = rng.integers(0, 2**31, n).astype(np.int32) if dt == np.int32 else rng.normal(0, 1, n).astype(np.float32)
    ref = oracle.sort(keys, p, s, 0, oracle.REGULAR, seed=0, want_sample=True)
    assert_same(run_gpu(keys, p, s, 0, oracle.REGULAR, 0), ref)


@pytest.mark.parametrize("n", [4000, 50_000])
def test_floats_around_zero(n):
    rng = np.random.default_rng(n)
    keys = rng.normal(0, 1, n).astype(np.float32)
    keys[::50], keys[1::50], keys[2::60], keys[3::60] = 0.0, -0.0, np.inf, -np.inf
    keys[4::70], keys[5::90] = np.nan, -np.float32(np.nan)
    check(keys, 2)
