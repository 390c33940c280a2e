"""The streamed counting sort of the keys-only final step (Fig. 2 step 12) at the sizes and
value distributions where it can go wrong: part edges, several CTAs per bucket, bins that hold
many keys, repeated keys, and keys of every type, each against the oracle, element by element."""
import numpy as np
import pytest

import oracle

from .gpu_util import assert_same, code_of, lib, run_gpu, to_dev

pytestmark = pytest.mark.gpu


def same(gpu, ref):
    assert gpu.keys.tobytes() == ref.keys.tobytes()
    assert np.array_equal(gpu.bucket_sizes, ref.bucket_sizes)


def check(keys, p, s=0):
    ref = oracle.sort(keys, p, s, 0, oracle.RANDOM, seed=5, want_sample=False)
    same(run_gpu(keys, p, s, 0, oracle.RANDOM, 5, refine=1, debug=False), ref)


# around a shape's stage (7680, 17408 and 37376 keys of 4 bytes, half of 8), one part more, 16-byte remainders
@pytest.mark.parametrize("dt", [np.int32, np.float64])
@pytest.mark.parametrize("n", [1, 2, 255, 1023, 3832, 3841, 7672, 7681, 8696, 8705, 17400, 17409, 37368, 37377, 74_745, 120_003])
def test_one_bucket(n, dt):
    rng = np.random.default_rng(n)
    keys = rng.integers(-2**31, 2**31, n).astype(np.int32) if dt == np.int32 else rng.normal(0, 1, n)
    check(keys, 1)


# half-word stages: few units of 2^15 (2^31) values, one and two parts, most keys in one half of the bins,
# windows over more than two units
@pytest.mark.parametrize("n", [37_369, 65_001, 65_540, 74_744, 74_749, 150_000])
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


# the sample sort (Fig. 1 step 5): around the one-CTA size, one and more records per bin of the larger form, tiles
# of both sizes, keys that repeat (ties by tag) and skewed doubles; every record is compared
@pytest.mark.parametrize("n, p, s", [(300, 3, 2), (9000, 1, 8193), (9000, 1, 8194), (20_000, 2, 4500), (60_000, 64, 1100), (50_000, 16, 70_000)])
@pytest.mark.parametrize("kind", ["uniform", "few_values", "skewed_doubles"])
def test_sample_sort(n, p, s, kind):
    rng = np.random.default_rng(n)
    if kind == "skewed_doubles":
        keys = rng.choice([-700.0, 3.0, 512.5], n, p=[0.1, 0.2, 0.7]) + rng.normal(0, 1, n) * rng.choice([1e-9, 0.01, 50.0], n)
    else:
        keys = rng.integers(0, 5 if kind == "few_values" else 2**31, n).astype(np.int32)
    ref = oracle.sort(keys, p, s, 0, oracle.RANDOM, seed=3, want_sample=True)
    assert_same(run_gpu(keys, p, s, 0, oracle.RANDOM, 3), ref)


def plain_call(keys, vals, p, s, **kw):
    """bsps_sort_keys or bsps_sort_pairs (run_gpu goes through bsps_sort_debug)."""
    import torch
    bsps, n, code = lib(), len(keys), code_of(keys)
    prm = bsps.make_params(p, s=s, sampling=bsps.BSPS_RANDOM, seed=9, **kw)
    ws = torch.empty(bsps.bsps_workspace_size(n, code, prm, vals is not None), dtype=torch.uint8, device="cuda:0")
    kin, sizes = to_dev(keys), torch.full((p,), -1, dtype=torch.int64, device="cuda:0")
    out = torch.empty_like(kin)
    if vals is None:
        assert bsps.bsps_sort_keys(kin, out, n, code, prm, sizes, ws) == 0
    else:
        vin = to_dev(vals)
        vout = torch.empty_like(vin)
        assert bsps.bsps_sort_pairs(kin, vin, out, vout, n, code, prm, sizes, ws) == 0
    st = bsps.bsps_read_stats(ws)
    return (out.cpu().numpy().view(keys.dtype), None if vals is None else vout.cpu().numpy().view(np.uint32),
            sizes.cpu().numpy(), st)


# single calls of up to 2^14 keys run on chip in one launch (no diagnostics asked for): the shapes' ends, several
# bucket counts and sample sizes, equal keys, payloads, and the status block, against the multi-kernel path's oracle
@pytest.mark.parametrize("dt", [np.uint32, np.int32, np.float32])
@pytest.mark.parametrize("n", [1, 2, 31, 600, 4095, 4096, 4097, 8192, 8193, 16_383, 16_384, 16_385])
@pytest.mark.parametrize("p, s", [(1, 0), (3, 0), (16, 0), (256, 20), (5, 1)])
def test_small_calls(n, p, s, dt):
    rng = np.random.default_rng(n + p)
    for few in (False, True):
        keys = (rng.integers(0, 7, n) if few else rng.integers(0, 2**32, n)).astype(np.uint32).view(dt)
        if dt == np.float32:
            keys = rng.integers(0, 7, n).astype(np.float32) if few else rng.normal(0, 1, n).astype(np.float32)
        vals = rng.integers(0, 2**32, n).astype(np.uint32)
        for v in (None, vals):
            ref = oracle.sort(keys, p, s, 0, oracle.RANDOM, seed=9, vals=v, want_sample=False)
            out, vout, sizes, st = plain_call(keys, v, p, s)
            assert out.tobytes() == ref.keys.tobytes() and np.array_equal(sizes, ref.bucket_sizes)
            assert v is None or np.array_equal(vout, ref.vals)
            assert (st.status, st.slow_buckets, st.max_bucket) == (0, 0, ref.bucket_sizes.max())


def test_small_call_reports_overflow():
    keys = np.random.default_rng(1).integers(0, 2**31, 10_000).astype(np.int32)
    st = plain_call(keys, None, 8, 4, capacity_pct=50)[3]
    assert (st.status, st.overflow) == (-4, 1)


# 4-byte keys with payloads as words of key and position: the shapes above through the counting sort, the cluster sort
# (values too heavy for a part) and the out-of-core sort, payloads of equal keys in input order
@pytest.mark.parametrize("n, p", [(20_000, 1), (90_000, 1), (90_001, 3), (300_000, 40), (700_000, 1)])
@pytest.mark.parametrize("name", sorted(SHAPES) + ["uniform"])
def test_pairs_as_words(name, n, p):
    rng = np.random.default_rng(n)
    keys = (rng.integers(-2**31, 2**31, n) if name == "uniform" else SHAPES[name](rng, n)).astype(np.int32)
    vals = rng.integers(0, 2**32, n).astype(np.uint32)
    for dt in (np.int32, np.uint32):
        ref = oracle.sort(keys.view(dt), p, 0, 0, oracle.RANDOM, seed=5, vals=vals, want_sample=False)
        assert_same(run_gpu(keys.view(dt), p, 0, 0, oracle.RANDOM, 5, vals, refine=1, debug=False), ref)


# keys that crowd in a small part of a bucket's range, so that 256 bins hold more than half a stage: nested widths,
# values with thousands of copies (below and past the 16 bits of a bin's count), one and several CTAs a bucket
CROWDS = {
    "narrow_component": lambda r, n: np.where(r.random(n) < 0.7, 1e6 + r.normal(0, 1e-3, n), r.normal(0, 1e6, n)),
    "nested": lambda r, n: r.normal(0, 1, n) * 10.0 ** -r.integers(0, 12, n),
    "two_heavy_values": lambda r, n: r.choice([3.0, 3.0 + 2.0**-30, 1e5], n, p=[0.45, 0.15, 0.4]) + (r.random(n) < 0.1) * r.normal(0, 1, n),
    "edge": lambda r, n: np.where(r.random(n) < 0.8, 2.0**30 - 1 - r.integers(0, 50, n), r.integers(0, 2**30, n)).astype(np.float64),
}


@pytest.mark.parametrize("n, p", [(24_000, 1), (60_000, 1), (160_001, 1), (450_000, 2)])
@pytest.mark.parametrize("name", sorted(CROWDS))
def test_crowded_ranges(name, n, p):
    rng = np.random.default_rng(n)
    keys = CROWDS[name](rng, n)
    check(keys, p)
    check(keys.astype(np.float32), p)
    k32 = keys.astype(np.float32)
    vals = rng.integers(0, 2**32, n).astype(np.uint32)
    ref = oracle.sort(k32, p, 0, 0, oracle.RANDOM, seed=9, vals=vals, want_sample=False)
    got = plain_call(k32, vals, p, 0, refine=1)
    assert got[0].tobytes() == ref.keys.tobytes() and np.array_equal(got[1], ref.vals)
    assert np.array_equal(got[2], ref.bucket_sizes)


# a few hundred values: one run of 256 one-value bins as large as a stage or larger, on several CTAs a bucket
@pytest.mark.parametrize("n", [65_536, 130_000, 400_000])
@pytest.mark.parametrize("values, p", [(180, 1), (375, 1), (3000, 8)])
def test_few_values_several_ctas(n, values, p):
    keys = np.random.default_rng(n).integers(0, values, n)
    check(keys.astype(np.int32), p)
    check(keys.astype(np.float64), p)
