// pairs.cu -- the final step (Fig. 2 step 12) of 4-byte keys with payloads that
// were routed as words phi << 32 | input position (route_keys.cu).
//
// The words are unique and their order is the stable order of the keys
// (Sec. 5.1.1: ties by position), so routing need not keep any order and the
// sort need not be stable: the counting sort of countsort.cuh, which keys alone
// take, puts a sub-bucket's words in order, and the payload of each is fetched
// by its position as the word is written.  The tiers are those of bucket.cu:
// what the counting sort gives back goes to the cluster sort, what that cannot
// hold to an LSD sort between the region and the two output arrays.
//
// Bound by instruction issue, then by the gather of the payloads (a 32-byte
// sector for 4 bytes of each).  2^22 pairs in 256 sub-buckets: the whole call
// takes 213 us, with the stable cluster sort and the look-back route 631; 2^28
// uniform pairs 13.9 ms and 33.0.  Where the sample's keys repeat (few values) the
// look-back route was taken beside it (api.cu): its regions hold keys and
// payloads in input order, sub-buckets of one value are copied here and the
// others listed for the stable cluster sort.
#include "countsort.cuh"
#include "many.cuh"
#include "segsort.cuh"

namespace bsps {

struct PairArgs {
    const uint64_t *words;     // region v at v * cap
    const uint32_t *vals_in;
    const uint32_t *vsize;
    const uint64_t *voff;
    const uint32_t *vphi;
    int64_t cap, P;
    uint32_t last;             // n - 1
    int G;
    uint32_t *out_keys, *out_vals;
    uint32_t *retry_flag, *retry_list, *slow_list;
    DevStatus *st;
    int64_t slow_above;        // a larger sub-bucket, sorted in several parts, counts as out of core
    uint64_t *words_rw;
    uint32_t few_above;        // the sample's keys repeat more often: the look-back route was taken
    uint32_t *reg_keys, *reg_vals;  // ... whose regions these are
    __device__ bool repeats() const { return st->repeats > few_above; }
};

template <int DT> struct PairSink {
    uint32_t *keys, *vals;
    const uint32_t *vals_in;
    uint32_t last;
    static constexpr bool kApart = false;
    __device__ int pad(uint32_t p) const { return (int)(((uintptr_t)(keys + p) >> 2) & 3); }
    __device__ uint32_t val(uint64_t w) const { return vals_in[min((uint32_t)w, last)]; }
    __device__ void one(int64_t p, uint64_t w) const {
        keys[p] = KeyTraits<DT>::inv((uint32_t)(w >> 32));
        vals[p] = val(w);
    }
    template <typename Key> __device__ void eight(int64_t p, Key key) const {
        uint32_t v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = val(key(j));
#pragma unroll
        for (int j = 0; j < 8; j += 4)
            *reinterpret_cast<uint4 *>(keys + p + j) =
                make_uint4(KeyTraits<DT>::inv((uint32_t)(key(j) >> 32)), KeyTraits<DT>::inv((uint32_t)(key(j + 1) >> 32)),
                           KeyTraits<DT>::inv((uint32_t)(key(j + 2) >> 32)), KeyTraits<DT>::inv((uint32_t)(key(j + 3) >> 32)));
        if (((uintptr_t)(vals + p) & 15) == 0) {  // (the same for a whole sub-bucket)
            *reinterpret_cast<uint4 *>(vals + p) = make_uint4(v[0], v[1], v[2], v[3]);
            *reinterpret_cast<uint4 *>(vals + p + 4) = make_uint4(v[4], v[5], v[6], v[7]);
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) vals[p + j] = v[j];
        }
    }
};

template <int DT, int SIZE>
__global__ void __launch_bounds__(CountShape<SIZE>::T, CountShape<SIZE>::kPerSm) pair_count_kernel(const Many<PairArgs> many) {
    const PairArgs &a = many.one;
    using CS = typename CountShape<SIZE>::template Sort<uint64_t>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if (a.st->overflow) return;  // a region holds slots that were never written
    const int64_t v = blockIdx.x / a.G;
    const int g = (int)(blockIdx.x % a.G);
    const int64_t cnt = a.vsize[v];
    if (cnt == 0) return;
    if (a.repeats()) {  // in input order by sub-bucket: those of one value are copied, the others listed (bucket.cuh)
        if (v > 0 && v < a.P - 1 && a.vphi[v - 1] == a.vphi[v]) {
            const uint32_t key = KeyTraits<DT>::inv(a.vphi[v]), *vals = a.reg_vals + v * a.cap;
            uint32_t *out_k = a.out_keys + a.voff[v], *out_v = a.out_vals + a.voff[v];
#pragma unroll 8
            for (int64_t e = g * blockDim.x + threadIdx.x; e < cnt; e += a.G * blockDim.x) {
                out_k[e] = key;
                out_v[e] = vals[e];
            }
        } else if (g == 0 && threadIdx.x == 0) {
            a.retry_list[atomicAdd(&a.st->retry_count, 1)] = (uint32_t)v;
        }
        return;
    }
    auto same = [](uint64_t w) { return w; };
    const KeySource<uint64_t, CountShape<SIZE>::T, decltype(same)> src{a.words + v * a.cap, same};
    // between two splitters; exact where one side has none or only positions differ
    const bool inner = v > 0 && v < a.P - 1;
    const bool one_value = inner && a.vphi[v - 1] == a.vphi[v];
    uint64_t lo, hi;
    if (!inner || one_value) {
        CS::bounds(smem_raw, src, (int)cnt, lo, hi);
    } else {
        lo = (uint64_t)a.vphi[v - 1] << 32;
        hi = (uint64_t)a.vphi[v] << 32 | 0xffffffffu;
    }
    const int64_t off = (int64_t)a.voff[v];
    const bool done = CS::run(smem_raw, src, (int)cnt, lo, hi,
                              PairSink<DT>{a.out_keys + off, a.out_vals + off, a.vals_in, a.last}, g, a.G);
    if (done && !one_value && cnt > a.slow_above && g == 0 && threadIdx.x == 0) atomicAdd(&a.st->slow_buckets, 1);
    if (!done && threadIdx.x == 0 && atomicExch(&a.retry_flag[v], 1u) == 0u)
        a.retry_list[atomicAdd(&a.st->retry_count, 1)] = (uint32_t)v;
}

// Tier 2: what the counting sort gave back, on a cluster of eight CTAs.
template <int DT>
__global__ void __cluster_dims__(8, 1, 1) __launch_bounds__(1024, 1) pair_listed_kernel(const Many<PairArgs> many) {
    const PairArgs &a = many.one;
    if (a.repeats()) return;
    using SS = SegSort<uint64_t, false, 8, kBucketItems64>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    typename SS::Smem &sm = *reinterpret_cast<typename SS::Smem *>(smem_raw);
    uint64_t *buf = reinterpret_cast<uint64_t *>(smem_raw + ((sizeof(typename SS::Smem) + 15) & ~size_t(15)));
    const int64_t nitems = a.st->retry_count, clusters = gridDim.x / 8;
    for (int64_t it = blockIdx.x / 8; it < nitems; it += clusters) {
        const int64_t v = a.retry_list[it], off = (int64_t)a.voff[v];
        const uint64_t *src = a.words + v * a.cap;
        const PairSink<DT> sink{a.out_keys + off, a.out_vals + off, a.vals_in, a.last};
        const bool done = SS::run(sm, buf, nullptr, (int64_t)a.vsize[v], [&](int64_t e) { return src[e]; },
                                  [&](uint32_t pos, uint64_t w, uint32_t) { sink.one(pos, w); });
        if (!done && blockIdx.x % 8 == 0 && threadIdx.x == 0) {
            atomicAdd(&a.st->slow_buckets, 1);
            a.slow_list[atomicAdd(&a.st->slow_count, 1)] = (uint32_t)v;
        }
        cg::this_cluster().sync();  // the next sub-bucket reuses every CTA's shared memory
    }
}

// Tier 3: one CTA sorts one oversized sub-bucket by LSD passes between its
// region and its output, where a word lies as its two halves (key and payload,
// in input order and sorted by key, after the look-back route).
template <int DT> __global__ void __launch_bounds__(kSlowThreads) pair_slow_kernel(const Many<PairArgs> many) {
    const PairArgs &a = many.one;
    using Rank = BlockRank<kSlowThreads, kSlowItems, 8>;
    constexpr int CH = kSlowThreads * kSlowItems;
    __shared__ typename Rank::Smem rsm;
    __shared__ uint32_t hist[256], run[256], tmp[40];
    __shared__ unsigned long long red[2];
    const int nslow = a.st->slow_count;
    for (int idx = blockIdx.x; idx < nslow; idx += gridDim.x) {
        const int64_t v = a.slow_list[idx], cnt = a.vsize[v], off = (int64_t)a.voff[v];
        uint64_t *reg = a.words_rw + v * a.cap;
        uint32_t *ok = a.out_keys + off, *ov = a.out_vals + off;
        const bool rep = a.repeats();
        uint32_t *rk = a.reg_keys + v * a.cap, *rv = a.reg_vals + v * a.cap;
        auto get = [&](int buf, int64_t e) {
            return buf == 0 && !rep ? reg[e] : (uint64_t)(buf ? ok : rk)[e] << 32 | (buf ? ov : rv)[e];
        };
        auto put = [&](int buf, int64_t e, uint64_t w) {
            if (buf == 0 && !rep) {
                reg[e] = w;
            } else {
                (buf ? ok : rk)[e] = (uint32_t)(w >> 32);
                (buf ? ov : rv)[e] = (uint32_t)w;
            }
        };
        if (threadIdx.x == 0) {
            red[0] = ~0ull;
            red[1] = 0ull;
        }
        __syncthreads();
        uint64_t mn = ~0ull, mx = 0ull;
        for (int64_t e = threadIdx.x; e < cnt; e += kSlowThreads) {
            const uint64_t w = get(0, e);
            mn = w < mn ? w : mn;
            mx = w > mx ? w : mx;
        }
        atomicMin(&red[0], (unsigned long long)mn);
        atomicMax(&red[1], (unsigned long long)mx);
        __syncthreads();
        const uint64_t base = rep ? red[0] >> 32 << 32 : red[0];
        const int bits = bit_length<uint64_t>(red[1] - base);
        int cur = 0;
        for (int shift = rep ? 32 : 0; shift < bits; shift += 8) {
            for (int i = threadIdx.x; i < 256; i += kSlowThreads) hist[i] = 0;
            __syncthreads();
            for (int64_t e = threadIdx.x; e < cnt; e += kSlowThreads)
                atomicAdd(&hist[(uint32_t)((get(cur, e) - base) >> shift) & 255u], 1u);
            __syncthreads();
            digit_excl_scan<kSlowThreads, 256>(hist, tmp);
            for (int i = threadIdx.x; i < 256; i += kSlowThreads) run[i] = hist[i];
            __syncthreads();
            for (int64_t cs = 0; cs < cnt; cs += CH) {
                uint64_t w[kSlowItems];
                uint32_t d[kSlowItems], rk[kSlowItems];
#pragma unroll
                for (int i = 0; i < kSlowItems; ++i) {
                    const int64_t e = cs + striped_slot<kSlowThreads, kSlowItems>(i);
                    d[i] = 255u;  // past the end: after every real word of digit 255
                    if (e < cnt) {
                        w[i] = get(cur, e);
                        d[i] = (uint32_t)((w[i] - base) >> shift) & 255u;
                    }
                }
                Rank::rank(rsm, d, rk);
#pragma unroll
                for (int i = 0; i < kSlowItems; ++i)
                    if (cs + striped_slot<kSlowThreads, kSlowItems>(i) < cnt) put(1 - cur, run[d[i]] + rk[i], w[i]);
                __syncthreads();
                for (int i = threadIdx.x; i < 256; i += kSlowThreads) run[i] += rsm.digit_tot[i];
                __syncthreads();
            }
            cur = 1 - cur;
        }
        const PairSink<DT> sink{ok, ov, a.vals_in, a.last};
        for (int64_t e = threadIdx.x; e < cnt; e += kSlowThreads) {
            const uint64_t w = get(cur, e);
            if (rep) {
                ok[e] = KeyTraits<DT>::inv((uint32_t)(w >> 32));
                ov[e] = (uint32_t)w;
            } else {
                sink.one(e, w);
            }
        }
        __syncthreads();
    }
}

static void pair_args(const Ctx &c, PairArgs &a) {
    a = {};
    a.words = a.words_rw = (uint64_t *)c.ly.reg_keys;  // the regions of keys and payloads, as one array of words
    a.vals_in = c.vals_in;
    a.vsize = c.ly.vsize;
    a.voff = c.ly.voff;
    a.vphi = (const uint32_t *)c.ly.vphi;
    a.cap = c.pl.cap;
    a.P = c.pl.P;
    a.last = (uint32_t)(c.pl.n - 1);
    a.out_keys = (uint32_t *)c.keys_out;
    a.out_vals = c.vals_out;
    a.retry_flag = c.ly.retry_flag;
    a.retry_list = c.ly.retry_list;
    a.slow_list = c.ly.slow_list;
    a.st = c.ly.status;
    a.few_above = c.both_routes ? repeats_above(c.pl) : 0xffffffffu;
    a.reg_keys = (uint32_t *)c.ly.reg_keys;
    a.reg_vals = c.ly.reg_vals;
    a.slow_above = (int64_t)8 * 1024 * kPairItems32;
}

template <int DT, int SIZE> static cudaError_t launch_count(Exec &x) {
    auto kern = pair_count_kernel<DT, SIZE>;
    return launch_calls<PairArgs>(x, kern, kern, CountShape<SIZE>::T, CountShape<SIZE>::template Sort<uint64_t>::smem_bytes(),
                                  [](const Ctx &c, PairArgs &a) {
        const int64_t mean = c.pl.n / c.pl.P;
        if (count_sort_size(mean, 8) != SIZE) return 0u;
        pair_args(c, a);
        a.G = count_sort_ctas<SIZE>(c.pl.P, mean);
        return (uint32_t)(c.pl.P * a.G);
    });
}

template <int DT> static cudaError_t launch_t(Exec &x) {
    cudaError_t e = launch_count<DT, kCountSmall>(x);
    if (e == cudaSuccess) e = launch_count<DT, kCountMedium>(x);
    if (e == cudaSuccess) e = launch_count<DT, kCountLarge>(x);
    auto all = [](uint32_t blocks) {
        return [=](const Ctx &c, PairArgs &a) {
            pair_args(c, a);
            return blocks;
        };
    };
    auto listed = pair_listed_kernel<DT>;
    if (e == cudaSuccess)
        e = launch_calls<PairArgs>(x, listed, listed, 1024, SegSort<uint64_t, false, 8, kBucketItems64>::smem_bytes(), all(16 * 8));
    if (e == cudaSuccess && x.calls[0].both_routes) e = launch_repeats_cluster(x);
    auto slow = pair_slow_kernel<DT>;
    if (e == cudaSuccess) e = launch_calls<PairArgs>(x, slow, slow, kSlowThreads, 0, all(64));
    return e;
}

cudaError_t launch_pair_words(Exec &x) {
    switch (x.calls[0].pl.dtype) {
    case BSPS_U32: return launch_t<BSPS_U32>(x);
    case BSPS_I32: return launch_t<BSPS_I32>(x);
    case BSPS_F32: return launch_t<BSPS_F32>(x);
    default: return cudaErrorInvalidValue;
    }
}

} // namespace bsps
