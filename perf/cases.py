"""What a user of this library has it do, as cases to time and compare.

Every case goes through the C ABI's Python binding: bsps_sort_keys, bsps_sort_pairs or
bsps_sort_batched, on inputs, outputs, parameters and a workspace that the caller holds.
The distributions are those of the paper's benchmarks (Sec. 6.3: uniform, Gaussian,
staggered, bucket-sorted), Zipf-distributed duplicates, a Gaussian mixture of doubles and
normally distributed floats.
"""
import math
import random

import numpy as np
import torch

import paper_1408_6729_gb300 as bsps

INT_MAX = 2**31
DTYPE = {"u32": bsps.BSPS_U32, "i32": bsps.BSPS_I32, "f32": bsps.BSPS_F32, "f64": bsps.BSPS_F64}
TORCH = {"u32": torch.int32, "i32": torch.int32, "f32": torch.float32, "f64": torch.float64}
KEY_BYTES = {"u32": 4, "i32": 4, "f32": 4, "f64": 8}
PIECE = 1 << 25  # keys generated at a time


def listed():
    """s = 0, runs = 0: the paper's defaults.  learned: the learned classifier (in a batch:
    from instances of 2^learned keys up).  merge: the paper's merge as the final step."""
    keys = {"op": "keys", "sampling": "random", "s": 0, "learned": False, "merge": False}
    regular = dict(keys, sampling="regular")
    return [
        # a small sort on the latency path of a larger program (a query's candidates, a batch's
        # lengths): launches are what counts
        dict(keys, name="keys_i32_3k_random", dtype="i32", dist="uniform", n=3000, p=4),
        # deterministic sampling at the size of the paper's smaller experiments: 2^20 keys over
        # the full unsigned range, p = 64, 8 samples per run
        dict(regular, name="keys_u32_1m_regular", dtype="u32", dist="uniform32", n=1 << 20, p=64, s=8),
        # keys with a 32-bit payload (a permutation, row ids), ragged size
        dict(keys, name="pairs_i32_4m_random", op="pairs", dtype="i32", dist="gaussian", n=4000037, p=256),
        # the randomized sort of the paper's distributions, 2^26 keys in 1024 buckets
        dict(keys, name="keys_i32_64m_random", dtype="i32", dist="gaussian", n=1 << 26, p=1024),
        # bulk sort of one large array: 2^28 uniform keys in 4096 buckets
        dict(keys, name="keys_i32_256m_random", dtype="i32", dist="uniform", n=1 << 28, p=4096),
        # the same array when the bucket sizes must be bounded (deterministic sampling)
        dict(regular, name="keys_i32_256m_regular", dtype="i32", dist="uniform", n=1 << 28, p=4096, s=4096),
        # grouping records by a duplicate-heavy column, stably: 256 values, Zipf, index payloads
        dict(regular, name="pairs_i32_256m_zipf", op="pairs", dtype="i32", dist="zipf", n=1 << 28, p=4096, s=4096),
        # skewed doubles (measurements, scores) with the learned classifier
        dict(keys, name="keys_f64_256m_learned", dtype="f64", dist="gmm", n=1 << 28, p=4096, s=16, learned=True),
        # skewed doubles with the splitter tree, ragged size
        dict(keys, name="keys_f64_16m_tree", dtype="f64", dist="gmm", n=16000033, p=1024),
        # the paper's own last step, the merge of the sorted blocks' segments
        dict(regular, name="keys_i32_16m_merge", dtype="i32", dist="uniform", n=1 << 24, p=1024, s=1024, merge=True),
        # many independent sorts of very uneven sizes (segments of a table), the learned
        # classifier on the large ones
        {"name": "batch_i32_mixed", "op": "batch", "count": 150, "lo_log2": 8, "hi_log2": 22, "learned": 18, "sizes": 1},
        # many short sorts (per-request or per-row), all within one SM's reach
        {"name": "batch_i32_small", "op": "batch", "count": 4096, "lo_log2": 8, "hi_log2": 14, "learned": 0, "sizes": 2},
    ]


def log_uniform(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def draw(rng):
    kind = rng.choice(["keys", "keys", "keys", "pairs", "pairs", "regular", "regular", "f64", "f64", "batch", "batch", "merge"])
    if kind == "batch":
        lo = rng.choice([8, 8, 10])
        hi = rng.randint(lo + 2, 22)
        mean = (2.0**hi - 2.0**lo) / ((hi - lo) * math.log(2.0))
        count = log_uniform(rng, 8, min(8192, max(16, 2.0**26 / mean)))
        return {"op": "batch", "count": count, "lo_log2": lo, "hi_log2": hi,
                "learned": rng.choice([0, 0, 18]) if hi > 18 else 0, "sizes": rng.randint(3, 1 << 20)}
    case = {"op": "pairs" if kind == "pairs" else "keys", "sampling": "random", "s": 0, "learned": False,
            "merge": kind == "merge"}
    if kind == "f64":
        n = log_uniform(rng, 1000, 1 << 26)
        case.update(dtype="f64", dist="gmm", learned=rng.random() < 0.5)
    else:
        n = log_uniform(rng, 1000, 1 << 27)
        case.update(dtype=rng.choice(["u32", "i32", "i32", "f32"]))
        case["dist"] = {"u32": "uniform32", "f32": "normal"}.get(case["dtype"]) or rng.choice(
            ["uniform", "gaussian", "staggered", "bucket_sorted", "zipf"])
    if kind in ("regular", "merge") or (kind == "pairs" and rng.random() < 0.4):
        case["sampling"] = "regular"
    # buckets of 2^10 to 2^16 keys, sometimes a number of buckets that is no power of two
    p = max(1, min(4096, round(n / 2.0 ** rng.uniform(10, 16))))
    if rng.random() < 0.7:
        p = 1 << max(0, (p - 1).bit_length())
    if case["sampling"] == "regular":
        p = max(p, -(-n // 65536))
        m = -(-n // p)
        if rng.random() < 0.5:
            case["s"] = max(1, min(p, m))
        else:
            case["s"] = max(1, min(4 * p, m // 4))
    if rng.random() < 0.5:
        n |= 1
    case.update(n=n, p=p)
    return case


# ------------------------------------------------------------------ inputs

def generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def zipf_table():
    """Zipf(1.1) over 256 values, each an injective scramble of its rank."""
    w = np.arange(1, 257, dtype=np.float64) ** -1.1
    cdf = np.cumsum(w / w.sum())
    cdf[-1] = 1.0
    k = np.arange(1, 257, dtype=np.uint64)
    values = ((k * np.uint64(2654435761)) & np.uint64(0xFFFFFFFF)).astype(np.uint32).view(np.int32)
    return torch.from_numpy(cdf).cuda(), torch.from_numpy(values).cuda()


def gmm_table(seed, components=8):
    """A skewed mixture: weights Dirichlet(0.3), means U[-1000, 1000], sigma 10^U[-2, 2]."""
    g = np.random.Generator(np.random.Philox(int(seed)))
    cdf = np.cumsum(g.dirichlet(np.full(components, 0.3)))
    cdf[-1] = 1.0
    mean, sigma = g.uniform(-1e3, 1e3, components), 10.0 ** g.uniform(-2.0, 2.0, components)
    return tuple(torch.from_numpy(v).cuda() for v in (cdf, mean, sigma))


def piece_of(dist, a, b, n, p, g, table):
    """Keys [a, b) of n."""
    c, kw = b - a, {"device": "cuda", "generator": g}
    if dist == "uniform":
        return torch.randint(0, INT_MAX, (c,), dtype=torch.int32, **kw)
    if dist == "uniform32":
        return torch.randint(-INT_MAX, INT_MAX, (c,), dtype=torch.int32, **kw)
    if dist == "gaussian":  # the mean of four uniform draws
        return (sum(torch.randint(0, INT_MAX, (c,), dtype=torch.int64, **kw) for _ in range(4)) // 4).to(torch.int32)
    if dist in ("staggered", "bucket_sorted"):
        at = torch.arange(a, b, dtype=torch.int64, device="cuda")
        m = -(-n // p)
        if dist == "staggered":  # block i holds one slice of the range, the slices out of order
            i = at // m
            k = torch.where(i < p // 2, 2 * i + 1, i - p // 2) % p
        else:  # every block holds p runs in ascending slices
            k = at % m * p // m
        width = max(1, INT_MAX // p)
        return (k * width + torch.randint(0, width, (c,), dtype=torch.int64, **kw)).to(torch.int32)
    if dist == "normal":
        return torch.randn(c, dtype=torch.float32, **kw)
    u = torch.rand(c, dtype=torch.float64, **kw)
    at = torch.searchsorted(table[0], u, right=True).clamp_(max=len(table[0]) - 1)
    if dist == "zipf":
        return table[1][at]
    assert dist == "gmm"
    return table[1][at] + table[2][at] * torch.randn(c, dtype=torch.float64, **kw)


def make_keys(case, seed):
    n = case["n"]
    g, out = generator(seed), torch.empty(n, dtype=TORCH[case["dtype"]], device="cuda")
    table = {"zipf": zipf_table, "gmm": lambda: gmm_table(seed)}.get(case["dist"], lambda: None)()
    for a in range(0, n, PIECE):
        b = min(n, a + PIECE)
        out[a:b] = piece_of(case["dist"], a, b, n, case["p"], g, table)
    return out


def batch_sizes(case):
    """Instance sizes, log-uniform on [2^lo, 2^hi]."""
    rng = random.Random(case["sizes"])
    return [int(2.0 ** rng.uniform(case["lo_log2"], case["hi_log2"])) for _ in range(case["count"])]


def make_batch_keys(case, seed):
    """Instances alternately uniform and Zipf."""
    sizes = batch_sizes(case)
    offsets = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    n, g, table = int(offsets[-1]), generator(seed), zipf_table()
    out = torch.empty(n, dtype=torch.int32, device="cuda")
    ends = torch.from_numpy(offsets[1:]).cuda()
    for a in range(0, n, PIECE):
        b = min(n, a + PIECE)
        odd = torch.searchsorted(ends, torch.arange(a, b, device="cuda"), right=True) % 2 == 1
        out[a:b] = torch.where(odd, piece_of("zipf", a, b, n, 1, g, table), piece_of("uniform", a, b, n, 1, g, None))
    return out, offsets


# ------------------------------------------------------------------ the call

def prepare(case, seed):
    if case["op"] == "batch":
        keys, offsets = make_batch_keys(case, seed)
        params = bsps.make_params(p=1, sampling=bsps.BSPS_RANDOM, seed=seed)
        tune = bsps.bsps_tune_default()
        tune.learned_min_log2 = case["learned"]
        ws = bsps.bsps_batch_workspace_size(offsets, bsps.BSPS_I32, params, tune)
        return {"op": "batch", "keys": keys, "out": torch.empty_like(keys), "offsets": offsets, "params": params, "tune": tune,
                "sizes": torch.empty(bsps.bsps_batch_bucket_base(offsets, tune)[-1], dtype=torch.int64, device="cuda"),
                "ws": torch.empty(ws, dtype=torch.uint8, device="cuda")}
    keys = make_keys(case, seed)
    n, pairs, dtype = case["n"], case["op"] == "pairs", DTYPE[case["dtype"]]
    params = bsps.make_params(
        p=case["p"], s=case["s"], sampling=bsps.BSPS_RANDOM if case["sampling"] == "random" else bsps.BSPS_REGULAR,
        classify=bsps.BSPS_LEARNED if case["learned"] else bsps.BSPS_TREE, seed=seed,
        final_step=bsps.BSPS_FINAL_MERGE if case["merge"] else bsps.BSPS_FINAL_SORT)
    state = {"op": case["op"], "n": n, "dtype": dtype, "params": params, "keys": keys, "out": torch.empty_like(keys),
             "sizes": torch.empty(case["p"], dtype=torch.int64, device="cuda"),
             "ws": torch.empty(bsps.bsps_workspace_size(n, dtype, params, pairs), dtype=torch.uint8, device="cuda")}
    if pairs:
        state.update(vals=torch.arange(n, dtype=torch.int32, device="cuda"), vals_out=torch.empty(n, dtype=torch.int32, device="cuda"))
    return state


def run(state):
    s = state
    if s["op"] == "batch":
        rc = bsps.bsps_sort_batched(s["keys"], s["out"], s["offsets"], bsps.BSPS_I32, s["params"], s["tune"], s["sizes"], s["ws"])
    elif s["op"] == "pairs":
        rc = bsps.bsps_sort_pairs(s["keys"], s["vals"], s["out"], s["vals_out"], s["n"], s["dtype"], s["params"], s["sizes"], s["ws"])
    else:
        rc = bsps.bsps_sort_keys(s["keys"], s["out"], s["n"], s["dtype"], s["params"], s["sizes"], s["ws"])
    if rc:
        raise RuntimeError(bsps.bsps_strerror(rc))
    outputs = {"keys": s["out"], "bucket_sizes": s["sizes"]}
    if s["op"] == "pairs":
        outputs["vals"] = s["vals_out"]
    return outputs


def work(case):
    """Every key (and payload) read once and written once; a sort does no floating-point work."""
    if case["op"] == "batch":
        return {"bytes": 8 * sum(batch_sizes(case)), "flops": 0}
    return {"bytes": 2 * case["n"] * (KEY_BYTES[case["dtype"]] + (4 if case["op"] == "pairs" else 0)), "flops": 0}


def exact(case, seed):
    """The sorted keys and, with payloads, the stable permutation; a bucket's size follows from
    the sample's own random or regular draw and has no value but the library's."""
    if case["op"] == "batch":
        keys, offsets = make_batch_keys(case, seed)
        # one sort of (instance, key) words; the keys are not negative or wrap alike in both halves
        at = torch.from_numpy(offsets[1:]).cuda()
        out = torch.empty_like(keys)
        ids = torch.searchsorted(at, torch.arange(len(keys), device="cuda"), right=True)
        words = (ids << 32) + (keys.to(torch.int64) + INT_MAX)
        out = ((torch.sort(words).values & 0xFFFFFFFF) - INT_MAX).to(torch.int32)
        return {"keys": out, "bucket_sizes": None}
    keys = make_keys(case, seed)
    if case["dtype"] == "u32":
        keys = keys ^ -INT_MAX  # unsigned order as signed order
    if case["op"] == "keys":
        out, at = torch.sort(keys).values, None
    else:
        out, at = torch.sort(keys, stable=True)
    if case["dtype"] == "u32":
        out = out ^ -INT_MAX
    outputs = {"keys": out, "bucket_sizes": None}
    if at is not None:
        outputs["vals"] = at.to(torch.int32)
    return outputs
