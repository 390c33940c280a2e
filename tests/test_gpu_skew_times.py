"""Inputs with repeated keys cost a bounded multiple of the same call on distinct keys.  Times are
CUDA events around a phase of the call, the least of several runs, so that only the kernels count;
the bounds leave room for what the repeats cost by themselves."""
import numpy as np
import pytest

from .gpu_util import code_of, lib, to_dev

pytestmark = pytest.mark.gpu

SAMPLE, SAMPLE_SORT, SPLITTERS, ROUTE, SORT = range(5)


def phase_us(keys, p, phases, pairs=False, s=0):
    """Least time of the given phases (one after the other) over ten runs, and the call's statistics."""
    import torch
    bsps, n, code = lib(), len(keys), code_of(keys)
    prm = bsps.make_params(p, s=s, sampling=bsps.BSPS_RANDOM, seed=9)
    ws = torch.empty(bsps.bsps_workspace_size(n, code, prm, pairs), dtype=torch.uint8, device="cuda:0")
    kin, sizes = to_dev(keys), torch.empty(p, dtype=torch.int64, device="cuda:0")
    out, val = torch.empty_like(kin), torch.arange(n, dtype=torch.int32, device="cuda:0") if pairs else None
    vout = torch.empty_like(val) if pairs else None
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(6)]
    for e in ev:
        e.record()
    best = float("inf")
    for _ in range(10):
        assert bsps.bsps_sort_debug(kin, val, out, vout, n, code, prm, sizes, ws, phase_events=ev) == 0
        torch.cuda.synchronize()
        best = min(best, 1e3 * ev[phases[0]].elapsed_time(ev[phases[-1] + 1]))
    assert out.cpu().numpy().tobytes() == np.sort(keys).tobytes()
    return best, bsps.bsps_read_stats(ws), ws


def uniform(n, seed=1):
    return np.random.default_rng(seed).integers(0, 2**31, n).astype(np.int32)


def copies(n, c, seed=2):
    """About c copies of every value, the values spread over the range."""
    v = np.random.default_rng(seed).integers(0, max(1, n // c), n).astype(np.int64)
    return (v * 2654435761 % 2**31).astype(np.int32)


# every key equals splitters, whose tags are then searched: log2 of their number more reads a key
# (pairs at a size that only moves as words)
@pytest.mark.parametrize("pairs", [False, True], ids=["keys", "pairs"])
def test_routing_few_values(pairs):
    n, p = (1 << 22, 1024) if pairs else (1 << 25, 1024)
    few, base = phase_us(copies(n, n // 100), p, [ROUTE], pairs)[0], phase_us(uniform(n), p, [ROUTE], pairs)[0]
    print(f"routing: few values {few:.0f} us, uniform {base:.0f} us")
    assert few <= 2.5 * base, (few, base)


def given_back(ws):
    """Sub-buckets the counting sort left to the cluster sort (DevStatus::retry_count of csrc/common.cuh)."""
    import torch
    return int(ws[:64].view(torch.int32)[14].item())


# values of a few dozen copies fill more bins past the window sort's reach than the scan lists
@pytest.mark.parametrize("n, p, c", [(1 << 20, 16, 20), (1 << 20, 16, 33), (300_000, 4, 24), (200_000, 1, 40), (16_000, 1, 25), (1 << 22, 256, 18)])
@pytest.mark.parametrize("dt", [np.int32, np.float64])
def test_many_long_bins_are_not_given_back(n, p, c, dt):
    keys = copies(n, c).astype(dt)
    assert given_back(phase_us(keys, p, [SORT])[2]) == 0


# ... and where the list holds them, finding the few that need the whole CTA costs little
@pytest.mark.parametrize("c", [10, 19])
def test_many_listed_bins(c):
    n, p = 1 << 26, 1024
    some, base = phase_us(copies(n, c), p, [SORT])[0], phase_us(uniform(n), p, [SORT])[0]
    print(f"bucket sort: {c} copies of every key {some:.0f} us, uniform {base:.0f} us")
    assert some <= 3 * base, (some, base)


def heavy(n, c, share, seed=3):
    """Distinct keys, and a share of the keys on values of about c copies each."""
    rng = np.random.default_rng(seed)
    return np.where(rng.random(n) < share, copies(n, c, seed + 1), uniform(n, seed + 2))


# values with thousands of copies, each sharing its bin with a few other keys
@pytest.mark.parametrize("c, share", [(5000, 0.3), (5000, 0.9), (40_000, 0.5)])
def test_heavy_values_among_distinct_keys(c, share):
    n, p = 1 << 24, 256
    some, base = phase_us(heavy(n, c, share), p, [SORT])[0], phase_us(uniform(n), p, [SORT])[0]
    print(f"bucket sort: {share} of the keys on values of {c} copies {some:.0f} us, uniform {base:.0f} us")
    assert some <= 6 * base, (some, base)


# a few values a bucket, of tens of thousands of copies each: every range of bins that holds one is crowded
def test_few_values_a_bucket():
    n, p = 1 << 24, 256
    some, base = phase_us(copies(n, 30_000).astype(np.float64), p, [SORT])[0], phase_us(uniform(n).astype(np.float64), p, [SORT])[0]
    print(f"bucket sort: values of 30000 copies {some:.0f} us, uniform {base:.0f} us")
    assert some <= 1.5 * base, (some, base)


# pairs of few values: the payloads travel along and one-value buckets are copied, where distinct keys' payloads are gathered
def test_pairs_of_few_values():
    n, p = 1 << 26, 1024
    phases = [ROUTE, SORT]
    few, base = phase_us(copies(n, n // 256), p, phases, pairs=True)[0], phase_us(uniform(n), p, phases, pairs=True)[0]
    print(f"routing and bucket sort of pairs: 256 values {few:.0f} us, uniform {base:.0f} us")
    assert few <= 0.95 * base, (few, base)


# large samples of doubles, whose 128-bit records fill a stage sooner
def test_sample_sort_of_many_doubles():
    n, p, s = 1 << 22, 1024, 1 << 16
    k = uniform(n)
    wide, base = phase_us(k.astype(np.float64), p, [SAMPLE_SORT], s=s)[0], phase_us(k, p, [SAMPLE_SORT], s=s)[0]
    print(f"sample sort of 2^26 records: doubles {wide:.0f} us, int32 {base:.0f} us")
    assert wide <= 4 * base, (wide, base)
