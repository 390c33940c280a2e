// bucket.cuh -- final sort of every bucket (Fig. 2 step 12 / Fig. 3 step 14):
// the keys a bucket received, in input order, are sorted stably and written
// to the bucket's place in the output, in up to three tiers:
//   1. keys only: the streamed counting sort of countsort.cuh (unstable ranks,
//      which equal keys cannot reveal), one CTA or several per sub-bucket; with
//      payloads: sub-buckets of one key value are copied as they stand;
//   2. the other sub-buckets with payloads, or what tier 1 gives back: the
//      stable cluster sort of segsort.cuh over a list;
//   3. sub-buckets larger than a cluster's shared memory: an out-of-core
//      radix sort in global memory.
#pragma once

#include "many.cuh"
#include "segsort.cuh"
#include "countsort.cuh"

namespace bsps {

template <typename K> struct BucketArgs {
    const K *reg_keys;        // phi of the routed keys, region v at v*cap
    const uint32_t *reg_vals;
    const uint32_t *vsize;
    const uint64_t *voff;
    int64_t cap;
    K *out_keys;
    uint32_t *out_vals;
    uint32_t *slow_list;
    DevStatus *st;
    const K *vphi;            // sub-bucket splitters (bounds of every sub-bucket)
    int64_t P;
    uint32_t *retry_flag;     // tier 1 gave the sub-bucket back
    uint32_t *retry_list;
    const uint32_t *only;     // tier 2 over a list (nullable: every sub-bucket)
    const int32_t *only_count;
    int64_t slow_above;       // a larger sub-bucket, sorted in several parts, counts as out of core
    int one_value_done;       // sub-buckets of one key value are already in the output
    int G;                    // tier 1: CTAs per sub-bucket
    int only_repeats;         // pairs queued on both routes: this one runs if the sample's keys repeat
    uint32_t few_above;       // ... more often than this
    K *reg_keys_rw;           // tier 3 sorts between the regions and the output
    uint32_t *reg_vals_rw;
};

// The listed and the out-of-core tier work through every call of a batch.
template <bool MANY, typename A, typename F> __device__ __forceinline__ void each_call(const Many<A> &m, F f) {
    if constexpr (MANY) {
        for (int i = 0; i < m.count; ++i) f(m.all[i]);
    } else {
        f(m.one);
    }
}

template <int DT, bool PAIRS, int CL, int ITEMS, bool MANY>
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(1024, 1)
bucket_sort_kernel(const Many<BucketArgs<typename KeyTraits<DT>::T>> many) {
    using K = typename KeyTraits<DT>::T;
    using SS = SegSort<K, PAIRS, CL, ITEMS>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    typename SS::Smem &sm = *reinterpret_cast<typename SS::Smem *>(smem_raw);
    K *buf = reinterpret_cast<K *>(smem_raw + ((sizeof(typename SS::Smem) + 15) & ~size_t(15)));
    uint32_t *slots = reinterpret_cast<uint32_t *>(buf + SS::CAP);

    // the listed sub-buckets (of a batch's calls: rarely any)
    if constexpr (MANY) {
        bool any = false;
        for (int i = threadIdx.x; i < many.count; i += blockDim.x) any |= *many.all[i].only_count != 0;
        if (!__syncthreads_or(any)) return;  // (every CTA of the grid alike)
    }
    each_call<MANY>(many, [&](const BucketArgs<K> &a) {
    if constexpr (PAIRS)
        if (a.only_repeats && a.st->repeats <= a.few_above) return;
    const int64_t nitems = *a.only_count, clusters = gridDim.x / CL;
    for (int64_t it = blockIdx.x / CL; it < nitems; it += clusters) {
        const int64_t v = a.only[it];
        const int64_t cnt = imin64(a.vsize[v], a.cap);
        if (cnt == 0) continue;
        const uint64_t off = a.voff[v];
        const K *src = a.reg_keys + v * a.cap;
        const uint32_t *vsrc = a.reg_vals + v * a.cap;
        K *out_k = a.out_keys + off;
        uint32_t *out_v = a.out_vals + off;
        auto emit = [&](uint32_t pos, K key, uint32_t slot) {
            out_k[pos] = KeyTraits<DT>::inv(key);
            if constexpr (PAIRS) out_v[pos] = vsrc[slot];
        };
        const bool done = SS::run(sm, buf, slots, cnt, [&](int64_t e) { return src[e]; }, emit);
        if (!done && blockIdx.x % CL == 0 && threadIdx.x == 0) {
            atomicAdd(&a.st->slow_buckets, 1);
            a.slow_list[atomicAdd(&a.st->slow_count, 1)] = (uint32_t)v;
        }
        // the next sub-bucket reuses every CTA's shared memory
        cg::this_cluster().sync();
    }
    });
}

// With payloads, before the cluster sort: a sub-bucket between two splitters
// of equal phi holds one key value, and routing kept its keys in input order,
// which is their sorted order under the position tie-break (Sec. 5.1.1); it is
// copied out as it stands.  Every other non-empty sub-bucket goes on the list
// the cluster sort then works through.
constexpr int kCopyThreads = 512;
template <int DT, bool PAIRS>
__global__ void __launch_bounds__(kCopyThreads) bucket_copy_kernel(const BucketArgs<typename KeyTraits<DT>::T> a,
                                                                  uint32_t *list, int32_t *list_count) {
    using K = typename KeyTraits<DT>::T;
    for (int64_t v = blockIdx.x; v < a.P; v += gridDim.x) {
        const int64_t cnt = imin64(a.vsize[v], a.cap);
        if (cnt == 0) continue;
        if (v > 0 && v < a.P - 1 && a.vphi[v - 1] == a.vphi[v]) {
            if (a.one_value_done) continue;  // the segment copy wrote it
            const K x = KeyTraits<DT>::inv(a.vphi[v]);
            K *out_k = a.out_keys + a.voff[v];
            uint32_t *out_v = a.out_vals + a.voff[v];
            const uint32_t *vsrc = a.reg_vals + v * a.cap;
#pragma unroll 8
            for (int64_t e = threadIdx.x; e < cnt; e += kCopyThreads) {
                out_k[e] = x;
                if constexpr (PAIRS) out_v[e] = vsrc[e];
            }
        } else if (threadIdx.x == 0) {
            list[atomicAdd(list_count, 1)] = (uint32_t)v;
        }
    }
}

// Tier 1 (keys only): G CTAs per sub-bucket, the streamed counting sort of
// countsort.cuh; its bounds are the two splitters around it (for the end
// buckets its smallest or largest key).
template <int DT, int SIZE, bool MANY>
__global__ void __launch_bounds__(CountShape<SIZE>::T, CountShape<SIZE>::kPerSm)
bucket_count_kernel(const Many<BucketArgs<typename KeyTraits<DT>::T>> many) {
    using K = typename KeyTraits<DT>::T;
    using CS = typename CountShape<SIZE>::template Sort<K>;
    const Pick<MANY, BucketArgs<K>> pk(many);
    const BucketArgs<K> &a = pk.a;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int G = a.G;
    const int64_t v = pk.block / G;
    const int g = (int)(pk.block % G);
    const int64_t cnt = imin64(a.vsize[v], a.cap);
    if (cnt == 0) return;
    auto same = [](K k) { return k; };
    auto inv = [](K k) { return KeyTraits<DT>::inv(k); };
    const KeySource<K, CountShape<SIZE>::T, decltype(same)> src{a.reg_keys + v * a.cap, same};
    K lo, hi;
    if (v == 0 || v == a.P - 1) CS::bounds(smem_raw, src, (int)cnt, lo, hi);  // no splitter on one side
    if (v > 0) lo = a.vphi[v - 1];
    if (v < a.P - 1) hi = a.vphi[v];
    K *out_k = a.out_keys + a.voff[v];
    bool done = true;
    if (lo == hi) {  // one key value: nothing to read
        const K x = KeyTraits<DT>::inv(lo);
        const int64_t share = (cnt + G - 1) / G, e0 = g * share, e1 = imin64(cnt, e0 + share);
#pragma unroll 4
        for (int64_t e = e0 + threadIdx.x; e < e1; e += blockDim.x) out_k[e] = x;
    } else {
        done = CS::run(smem_raw, src, (int)cnt, lo, hi, KeySink<K, decltype(inv)>{out_k, inv}, g, G);
        // larger than a cluster's shared memory: sorted out of core, part by part
        if (done && cnt > a.slow_above && g == 0 && threadIdx.x == 0) atomicAdd(&a.st->slow_buckets, 1);
    }
    if (!done && threadIdx.x == 0 && atomicExch(&a.retry_flag[v], 1u) == 0u)
        a.retry_list[atomicAdd(&a.st->retry_count, 1)] = (uint32_t)v;
}

// ---------------------------------------------------------------------------
// Out-of-core path: one CTA sorts one oversized sub-bucket by LSD passes
// between its region and its output range, chunk by chunk, stably.
// ---------------------------------------------------------------------------
template <int DT, bool PAIRS, bool MANY>
__global__ void __launch_bounds__(kSlowThreads) bucket_slow_kernel(const Many<BucketArgs<typename KeyTraits<DT>::T>> many) {
    using K = typename KeyTraits<DT>::T;
    using Rank = BlockRank<kSlowThreads, kSlowItems, 8>;
    constexpr int CH = kSlowThreads * kSlowItems;
    __shared__ typename Rank::Smem rsm;
    __shared__ uint32_t hist[256], run[256], tmp[40];
    __shared__ K red[2];
    if constexpr (MANY) {
        bool any = false;
        for (int i = threadIdx.x; i < many.count; i += blockDim.x) any |= many.all[i].st->slow_count != 0;
        if (!__syncthreads_or(any)) return;
    }
    each_call<MANY>(many, [&](const BucketArgs<K> &a) {
    const int nslow = a.st->slow_count;
    for (int idx = blockIdx.x; idx < nslow; idx += gridDim.x) {
        const int64_t v = a.slow_list[idx];
        const int64_t cnt = imin64(a.vsize[v], a.cap);
        const uint64_t off = a.voff[v];
        K *bufk[2] = {a.reg_keys_rw + v * a.cap, reinterpret_cast<K *>(a.out_keys) + off};
        uint32_t *bufv[2] = {PAIRS ? a.reg_vals_rw + v * a.cap : nullptr, PAIRS ? a.out_vals + off : nullptr};
        // key range
        K mn = all_ones<K>(), mx = 0;
        for (int64_t e = threadIdx.x; e < cnt; e += kSlowThreads) {
            const K x = bufk[0][e];
            mn = x < mn ? x : mn;
            mx = x > mx ? x : mx;
        }
        if (threadIdx.x == 0) { red[0] = all_ones<K>(); red[1] = 0; }
        __syncthreads();
        if constexpr (sizeof(K) == 8) {
            atomicMin((unsigned long long *)&red[0], (unsigned long long)mn);
            atomicMax((unsigned long long *)&red[1], (unsigned long long)mx);
        } else {
            atomicMin((unsigned *)&red[0], (unsigned)mn);
            atomicMax((unsigned *)&red[1], (unsigned)mx);
        }
        __syncthreads();
        const K base = red[0];
        const int bits = bit_length<K>(red[1] - base);
        __syncthreads();
        int cur = 0;
        for (int shift = 0; shift < bits; shift += 8) {
            const K *sk = bufk[cur];
            K *dk = bufk[1 - cur];
            for (int i = threadIdx.x; i < 256; i += kSlowThreads) { hist[i] = 0; }
            __syncthreads();
            for (int64_t e = threadIdx.x; e < cnt; e += kSlowThreads)
                atomicAdd(&hist[(uint32_t)((sk[e] - base) >> shift) & 255u], 1u);
            __syncthreads();
            digit_excl_scan<kSlowThreads, 256>(hist, tmp);
            for (int i = threadIdx.x; i < 256; i += kSlowThreads) run[i] = hist[i];
            __syncthreads();
            for (int64_t cs = 0; cs < cnt; cs += CH) {
                K kk[kSlowItems];
                uint32_t vv[kSlowItems], d[kSlowItems], rk[kSlowItems];
#pragma unroll
                for (int i = 0; i < kSlowItems; ++i) {
                    const int64_t e = cs + striped_slot<kSlowThreads, kSlowItems>(i);
                    if (e < cnt) {
                        kk[i] = sk[e];
                        if constexpr (PAIRS) vv[i] = bufv[cur][e];
                        d[i] = (uint32_t)((kk[i] - base) >> shift) & 255u;
                    } else {
                        d[i] = 255u;
                    }
                }
                Rank::rank(rsm, d, rk);
#pragma unroll
                for (int i = 0; i < kSlowItems; ++i) {
                    const int64_t e = cs + striped_slot<kSlowThreads, kSlowItems>(i);
                    if (e < cnt) {
                        const uint32_t pos = run[d[i]] + rk[i];
                        dk[pos] = kk[i];
                        if constexpr (PAIRS) bufv[1 - cur][pos] = vv[i];
                    }
                }
                __syncthreads();
                for (int i = threadIdx.x; i < 256; i += kSlowThreads) run[i] += rsm.digit_tot[i];
                __syncthreads();
            }
            cur = 1 - cur;
        }
        // final placement in the output, back to key bits
        for (int64_t e = threadIdx.x; e < cnt; e += kSlowThreads) {
            const K x = bufk[cur][e];
            if constexpr (PAIRS) {
                if (cur == 0) a.out_vals[off + e] = bufv[0][e];
            }
            a.out_keys[off + e] = KeyTraits<DT>::inv(x);
        }
        __syncthreads();
    }
    });
}

static int sm_count() {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms > 0 ? sms : 1;
}

template <int DT> static void bucket_args(const Ctx &c, BucketArgs<typename KeyTraits<DT>::T> &a) {
    using K = typename KeyTraits<DT>::T;
    a = {};
    a.reg_keys = (const K *)c.ly.reg_keys;
    a.reg_vals = c.ly.reg_vals;
    a.vsize = c.ly.vsize;
    a.voff = c.ly.voff;
    a.cap = c.pl.cap;
    a.out_keys = (K *)c.keys_out;
    a.out_vals = c.vals_out;
    a.slow_list = c.ly.slow_list;
    a.st = c.ly.status;
    a.vphi = (const K *)c.ly.vphi;
    a.P = c.pl.P;
    a.retry_flag = c.ly.retry_flag;
    a.retry_list = c.ly.retry_list;
    a.only = c.ly.retry_list;
    a.only_count = &c.ly.status->retry_count;
    a.slow_above = (int64_t)8 * 1024 * (sizeof(K) == 8 ? kBucketItems64 : kBucketItems32);
    a.one_value_done = c.pl.seg_route;
    a.only_repeats = c.both_routes;
    a.few_above = repeats_above(c.pl);
    a.reg_keys_rw = (K *)c.ly.reg_keys;
    a.reg_vals_rw = c.ly.reg_vals;
}

// The cluster sort over the listed sub-buckets and the out-of-core sort: as
// many clusters as run at once (one CTA per SM), at least 16, for all calls.
// (Their kernels read a batch's arguments from the table, so the grid is given
// whole, by the first call.)
template <typename A, typename K1, typename KN>
static cudaError_t launch_listed(Exec &x, K1 single, KN all, unsigned grid, unsigned threads, size_t smem,
                                 void (*fill)(const Ctx &, A &)) {
    bool first = true;
    return launch_calls<A>(x, single, all, threads, smem, [&](const Ctx &c, A &a) {
        fill(c, a);
        const unsigned g = first ? grid : 0u;
        first = false;
        return x.many ? (g ? g : kNoBlocks) : g;
    });
}

template <int DT, bool PAIRS, int CL, int ITEMS> static cudaError_t launch_cluster(Exec &x) {
    using K = typename KeyTraits<DT>::T;
    using SS = SegSort<K, PAIRS, CL, ITEMS>;
    const int64_t clusters = imax64(16, sm_count() / CL);
    const int64_t most = x.many ? clusters : imin64(x.calls[0].pl.P, clusters);
    return launch_listed<BucketArgs<K>>(x, bucket_sort_kernel<DT, PAIRS, CL, ITEMS, false>,
                                        bucket_sort_kernel<DT, PAIRS, CL, ITEMS, !PAIRS>, (unsigned)(most * CL), 1024,
                                        SS::smem_bytes(), bucket_args<DT>);
}

template <int DT, bool PAIRS> static cudaError_t launch_slow(Exec &x) {
    return launch_listed<BucketArgs<typename KeyTraits<DT>::T>>(x, bucket_slow_kernel<DT, PAIRS, false>,
                                                                bucket_slow_kernel<DT, PAIRS, !PAIRS>, 64, kSlowThreads, 0,
                                                                bucket_args<DT>);
}

template <int DT, int SIZE> static cudaError_t launch_count(Exec &x) {
    using K = typename KeyTraits<DT>::T;
    using CS = typename CountShape<SIZE>::template Sort<K>;
    int64_t all = 0;
    for (int i = 0; i < x.count; ++i) all += x.calls[i].pl.P;
    return launch_calls<BucketArgs<K>>(x, bucket_count_kernel<DT, SIZE, false>, bucket_count_kernel<DT, SIZE, true>,
                                       CountShape<SIZE>::T, CS::smem_bytes(), [=](const Ctx &c, BucketArgs<K> &a) {
        const int64_t mean = c.pl.n / c.pl.P;
        if (count_sort_size(mean, sizeof(K)) != SIZE) return 0u;
        bucket_args<DT>(c, a);
        a.G = count_sort_ctas<SIZE>(all, mean);
        return (uint32_t)(c.pl.P * a.G);
    });
}

template <int DT> cudaError_t launch_bucket_keys_t(Exec &x) {
    using K = typename KeyTraits<DT>::T;
    cudaError_t e = launch_count<DT, kCountSmall>(x);
    if (e == cudaSuccess) e = launch_count<DT, kCountMedium>(x);
    if (e == cudaSuccess) e = launch_count<DT, kCountLarge>(x);
    // what tier 1 gave back
    if (e == cudaSuccess) e = launch_cluster<DT, false, 8, (sizeof(K) == 8 ? kBucketItems64 : kBucketItems32)>(x);
    if (e == cudaSuccess) e = launch_slow<DT, false>(x);
    return e;
}

} // namespace bsps
