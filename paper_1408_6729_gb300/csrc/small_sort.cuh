// small_sort.cuh -- whole sorts on chip: one CTA runs the method for one input of at
// most kSmallKeys keys (random sampling, the tie-break by position), for a
// single small call and for the small instances of a batch.
//
// The multi-kernel path would spend ten launches on such an input and leave
// the GPU idle through most of them: a call of 3000 int32 keys takes 28 us here
// (bound by one CTA's chain of phases, about 12 us of them the sample's sort)
// and took 205 us in 35 launches; 4096 instances of 2^8 to 2^14 keys take 567 us
// and took 1869 by bitonic networks.  Past 2^14 keys one CTA is the bottleneck
// and the multi-kernel path's many are not.
//
// Keys without payloads: the keys are sorted whole by the counting sort of
// countsort.cuh (equal keys need no order among them).  The sample's records
// (Fig. 3 step 4) are drawn and sorted in the space the keys leave, the
// records of rank i * s are the splitters (Fig. 2 step 6), and the keys are
// counted per bucket against them (Fig. 2 step 9, Fig. 1 step 9).
//
// With payloads the keys are sorted as words phi << 32 | position (the total
// order of Sec. 5.1.1), which places the payloads stably, and the rest is read
// off that order: the sample's draws are counted per position, their running
// sum along the sorted keys is the rank in the sorted sample, a splitter is
// the key where it reaches i * s, and a bucket's size is the distance between
// two of them.
//
// Three shapes by size keep several inputs on an SM: 256 threads up to 4096
// keys, 512 up to 8192, else 1024.
#pragma once

#include "small.cuh"

#include "countsort.cuh"

namespace bsps {

template <int SIZE> struct SmallShape {
    static constexpr int T = CountShape<SIZE>::T;
    static constexpr int kKeys = small_keys(SIZE);
    static constexpr int kPerSm = SIZE == kCountSmall ? 4 : SIZE == kCountMedium ? 2 : 1;
    // every key is stored as a 64-bit word; the bins' words take the sample
    // weights once the keys are in place
    static constexpr int kStage = (kKeys + 8) * 8;
    using Sort = CountSort<uint64_t, T, kKeys, kStage>;
    struct Extra {
        uint32_t start[kSmallBuckets + 1];  // sorted position of every bucket's first key
        uint32_t tmp[40];
    };
    static constexpr size_t kDraws = (Sort::smem_bytes() + 15) & ~size_t(15);
    static constexpr size_t kExtra = kDraws + (size_t)kKeys * 2 + 16;
    static constexpr size_t smem() { return ((kExtra + 15) & ~size_t(15)) + sizeof(Extra); }
    static_assert(kPerSm * (smem() + 1024) <= 228 * 1024, "resident CTAs");
};

// The status block of a single call.
template <int T> __device__ void small_status(uint32_t most, uint32_t *tmp, int64_t cap, DevStatus *st) {
    most = __reduce_max_sync(0xffffffffu, most);
    if ((threadIdx.x & 31) == 0) tmp[threadIdx.x >> 5] = most;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < T / 32; ++w) most = max(most, tmp[w]);
        DevStatus s = {};
        s.max_bucket = s.max_vbucket = most;
        if ((int64_t)most > cap) {
            s.overflow = 1;
            s.error = BSPS_ERR_BUCKET_OVERFLOW;
        }
        *st = s;
    }
}

// ---- keys without payloads ----
template <int SIZE> struct SmallKeysShape {
    static constexpr int T = CountShape<SIZE>::T;
    static constexpr int kKeys = small_keys(SIZE);
    static constexpr int kPerSm = SIZE == kCountSmall ? 6 : SIZE == kCountMedium ? 3 : 1;
    using Sort = CountSort<uint32_t, T, kKeys, (kKeys + 8) * 4>;
    using Records = BlockSort<uint64_t, T>;
    struct Extra {
        uint64_t split[kSmallBuckets];
        uint32_t hist[kSmallBuckets];
        uint32_t tmp[40];
    };
    static constexpr size_t kExtra = (Sort::smem_bytes() + 15) & ~size_t(15);
    static constexpr size_t smem() { return kExtra + sizeof(Extra); }
    // the records and their sort take the place of the keys' sort
    static constexpr size_t kRecords = (sizeof(typename Records::Smem) + 15) & ~size_t(15);
    static constexpr int64_t kSample = (int64_t)((kExtra - kRecords) / 8);
    static_assert(kPerSm * (smem() + 1024) <= 228 * 1024, "resident CTAs");
};

template <int DT, int SIZE>
__global__ void __launch_bounds__(SmallKeysShape<SIZE>::T, SmallKeysShape<SIZE>::kPerSm)
small_keys_kernel(const uint32_t *__restrict__ keys_in, uint32_t *keys_out, const SmallJob *__restrict__ jobs,
                  const __grid_constant__ SmallList list, bool batch, int64_t *bucket_sizes, DevStatus *st) {
    using Sh = SmallKeysShape<SIZE>;
    using CS = typename Sh::Sort;
    constexpr int T = Sh::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    typename Sh::Extra &ex = *reinterpret_cast<typename Sh::Extra *>(smem_raw + Sh::kExtra);
    const int tid = threadIdx.x, lane = tid & 31;
    const SmallJob J = jobs ? jobs[blockIdx.x] : list.job[blockIdx.x];
    if (batch && st && blockIdx.x == 0 && tid == 0) *st = DevStatus{};
    const int n = J.n, p = J.p;
    const uint32_t *in = keys_in + J.off;
    auto phi = [](uint32_t k) { return KeyTraits<DT>::phi(k); };
    auto inv = [](uint32_t k) { return KeyTraits<DT>::inv(k); };
    using Few = BlockSort<uint32_t, T>;
    if (n <= Few::M) {
        // one key to a thread (a batch of one instance of 447 keys takes 18 us
        // when they are counted)
        uint32_t *piv = reinterpret_cast<uint32_t *>(smem_raw);
        int m = 1;
        while (m < n) m <<= 1;
        Few::sort_pivots(piv, tid < n ? phi(in[tid]) : 0xffffffffu, m);
        if (tid < n) keys_out[J.off + tid] = inv(piv[tid]);
    } else {
        const KeySource<uint32_t, T, decltype(phi)> src{in, phi};
        uint32_t lo, hi;
        CS::bounds(smem_raw, src, n, lo, hi);
        CS::run(smem_raw, src, n, lo, hi, KeySink<uint32_t, decltype(inv)>{keys_out + J.off, inv}, 0, 1);
    }
    uint32_t most = (uint32_t)n;
    if (p > 1) {
        __syncthreads();
        uint64_t *rec = reinterpret_cast<uint64_t *>(smem_raw + Sh::kRecords);
        for (int b = tid; b < p; b += T) ex.hist[b] = 0;
        for (int blk = tid; blk * 4 < J.S; blk += T) {
            uint64_t c[4] = {(uint64_t)blk, 0, 0, 0};
            philox4x64_10(c, J.seed, 0);
#pragma unroll
            for (int w = 0; w < 4; ++w)
                if (blk * 4 + w < J.S && n > 0) {
                    const uint32_t g = (uint32_t)__umul64hi(c[w], (uint64_t)n);
                    rec[blk * 4 + w] = (uint64_t)phi(in[g]) << 32 | g;
                }
        }
        __syncthreads();
        Sh::Records::run(*reinterpret_cast<typename Sh::Records::Smem *>(smem_raw), rec, n > 0 ? J.S : 0);
        for (int i = tid; i < p - 1; i += T) ex.split[i] = rec[(int64_t)(i + 1) * J.s - 1];
        __syncthreads();
        for (int e0 = 0; e0 < n; e0 += T) {
            const int e = e0 + tid;
            const bool ok = e < n;
            uint32_t b = 0xffffffffu;
            if (ok) {
                const uint64_t key = (uint64_t)phi(in[e]) << 32 | (uint32_t)e;
                uint32_t a = 0, z = (uint32_t)p - 1;  // splitters at or below the key
                while (a < z) {
                    const uint32_t mid = (a + z) >> 1;
                    if (ex.split[mid] <= key) a = mid + 1;
                    else z = mid;
                }
                b = a;
            }
            // few buckets: a warp's keys of lane 0's bucket are counted at once
            const uint32_t b0 = __shfl_sync(0xffffffffu, b, 0);
            const uint32_t same = __ballot_sync(0xffffffffu, b == b0);
            if (ok && b != b0) atomicAdd(&ex.hist[b], 1u);
            if (lane == 0 && ok) atomicAdd(&ex.hist[b], (uint32_t)__popc(same));
        }
        __syncthreads();
        most = 0;
        for (int b = tid; b < p; b += T) most = max(most, ex.hist[b]);
    }
    if (bucket_sizes)
        for (int b = tid; b < p; b += T) bucket_sizes[J.bbase + b] = p > 1 ? ex.hist[b] : (uint32_t)n;
    if (!batch) small_status<T>(most, ex.tmp, J.cap, st);
}

// ---- keys with payloads ----
// The keys of an input as words phi << 32 | position.
template <int DT, int T> struct SmallSource {
    const uint32_t *__restrict__ keys;
    template <typename F> __device__ void each(int n, F f) const {
        auto word = [](uint32_t k, int e) { return (uint64_t)KeyTraits<DT>::phi(k) << 32 | (uint32_t)e; };
        int e = threadIdx.x;
        for (; e + 3 * T < n; e += 4 * T) {
            uint32_t k[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) k[j] = keys[e + j * T];
#pragma unroll
            for (int j = 0; j < 4; ++j) f(word(k[j], e + j * T));
        }
        for (; e < n; e += T) f(word(keys[e], e));
    }
};

// Sorted words out: the key, its payload, and the draws of its position.
template <int DT> struct SmallSink {
    uint32_t *keys;
    const uint32_t *vals_in;
    uint32_t *vals_out;
    const uint16_t *draws;  // by position
    uint16_t *weight;       // by sorted position
    static constexpr bool kApart = false;
    __device__ int pad(uint32_t p) const { return (int)(((uintptr_t)(keys + p) >> 2) & 3); }
    __device__ void one(int64_t p, uint64_t k) const {
        const uint32_t at = (uint32_t)k;
        keys[p] = KeyTraits<DT>::inv((uint32_t)(k >> 32));
        weight[p] = draws[at];
        vals_out[p] = vals_in[at];
    }
    template <typename Key> __device__ void eight(int64_t p, Key key) const {
#pragma unroll
        for (int j = 0; j < 8; j += 4) {
            const uint64_t a = key(j), b = key(j + 1), c = key(j + 2), d = key(j + 3);
            *reinterpret_cast<uint4 *>(keys + p + j) =
                make_uint4(KeyTraits<DT>::inv((uint32_t)(a >> 32)), KeyTraits<DT>::inv((uint32_t)(b >> 32)),
                           KeyTraits<DT>::inv((uint32_t)(c >> 32)), KeyTraits<DT>::inv((uint32_t)(d >> 32)));
            weight[p + j] = draws[(uint32_t)a];
            weight[p + j + 1] = draws[(uint32_t)b];
            weight[p + j + 2] = draws[(uint32_t)c];
            weight[p + j + 3] = draws[(uint32_t)d];
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) vals_out[p + j] = vals_in[(uint32_t)key(j)];
    }
};

template <int DT, int SIZE>
__global__ void __launch_bounds__(SmallShape<SIZE>::T, SmallShape<SIZE>::kPerSm)
small_pairs_kernel(const uint32_t *__restrict__ keys_in, const uint32_t *__restrict__ vals_in, uint32_t *keys_out,
                   uint32_t *vals_out, const SmallJob J, int64_t *bucket_sizes, DevStatus *st) {
    using Sh = SmallShape<SIZE>;
    using CS = typename Sh::Sort;
    constexpr int T = Sh::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    uint16_t *draws = reinterpret_cast<uint16_t *>(smem_raw + Sh::kDraws);
    typename Sh::Extra &ex = *reinterpret_cast<typename Sh::Extra *>(smem_raw + ((Sh::kExtra + 15) & ~size_t(15)));
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = J.n, p = J.p;
    // ---- draws per position of the random sample (Fig. 3 step 4) ----
    for (int e = tid; e < (n + 1) / 2; e += T) reinterpret_cast<uint32_t *>(draws)[e] = 0u;
    for (int b = tid; b <= p; b += T) ex.start[b] = b == 0 ? 0u : (uint32_t)n;
    __syncthreads();
    if (p > 1) {
        for (int blk = tid; blk * 4 < J.S; blk += T) {
            uint64_t c[4] = {(uint64_t)blk, 0, 0, 0};
            philox4x64_10(c, J.seed, 0);
#pragma unroll
            for (int w = 0; w < 4; ++w)
                if (blk * 4 + w < J.S) {
                    const uint32_t g = (uint32_t)__umul64hi(c[w], (uint64_t)n);
                    atomicAdd(reinterpret_cast<uint32_t *>(draws) + (g >> 1), (g & 1u) ? 0x10000u : 1u);
                }
        }
    }
    // ---- the keys in order (ties by position), and their positions' draws ----
    uint16_t *weight = reinterpret_cast<uint16_t *>(CS::bins(smem_raw));
    const SmallSource<DT, T> src{keys_in};
    uint64_t lo, hi;
    CS::bounds(smem_raw, src, n, lo, hi);
    CS::run(smem_raw, src, n, lo, hi,
            SmallSink<DT>{keys_out, vals_in, vals_out, draws, weight}, 0, 1);
    __syncthreads();
    // ---- splitters of rank i * s in the sample (Fig. 2 step 6): where the
    //      running sum of the draws reaches it ----
    if (p > 1) {
        const int per = (n + T - 1) / T, r0 = min(n, tid * per), r1 = min(n, r0 + per);
        uint32_t local = 0;
        for (int r = r0; r < r1; ++r) local += weight[r];
        uint32_t wtot;
        const uint32_t wex = warp_excl_scan(local, &wtot);
        if (lane == 31) ex.tmp[warp] = wtot;
        __syncthreads();
        uint32_t run = wex;
        for (int w = 0; w < warp; ++w) run += ex.tmp[w];
        if (local) {
            uint32_t i = run / (uint32_t)J.s + 1u;  // the next splitter's index
            for (int r = r0; r < r1; ++r) {
                run += weight[r];
                for (; i < (uint32_t)p && run >= i * (uint32_t)J.s; ++i) ex.start[i] = (uint32_t)r;
            }
        }
        __syncthreads();
    }
    uint32_t most = 0;
    for (int b = tid; b < p; b += T) {
        const uint32_t c = ex.start[b + 1] - ex.start[b];
        if (bucket_sizes) bucket_sizes[b] = c;
        most = max(most, c);
    }
    small_status<T>(most, ex.tmp, J.cap, st);
}

// ---- host side ----
template <int DT, int SIZE>
static cudaError_t launch_keys_t(const void *in, void *out, const SmallJob *jobs, int njobs, const SmallList &list, bool batch,
                                 int64_t *bsz, DevStatus *st, cudaStream_t stream) {
    using Sh = SmallKeysShape<SIZE>;
    auto kern = small_keys_kernel<DT, SIZE>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sh::smem());
    if (e != cudaSuccess) return e;
    kern<<<njobs, Sh::T, Sh::smem(), stream>>>((const uint32_t *)in, (uint32_t *)out, jobs, list, batch, bsz, st);
    return cudaGetLastError();
}

template <int DT, int SIZE>
static cudaError_t launch_pairs_t(const Ctx &c, const SmallJob &J) {
    using Sh = SmallShape<SIZE>;
    auto kern = small_pairs_kernel<DT, SIZE>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sh::smem());
    if (e != cudaSuccess) return e;
    kern<<<1, Sh::T, Sh::smem(), c.stream>>>((const uint32_t *)c.keys_in, c.vals_in, (uint32_t *)c.keys_out, c.vals_out, J,
                                             c.bucket_sizes, c.ly.status);
    return cudaGetLastError();
}

template <int DT>
cudaError_t launch_small_keys_t(int size, const void *in, void *out, const SmallJob *jobs, int njobs, const SmallList &list,
                                bool batch, int64_t *bsz, DevStatus *st, cudaStream_t stream) {
    switch (size) {
    case kCountSmall: return launch_keys_t<DT, kCountSmall>(in, out, jobs, njobs, list, batch, bsz, st, stream);
    case kCountMedium: return launch_keys_t<DT, kCountMedium>(in, out, jobs, njobs, list, batch, bsz, st, stream);
    default: return launch_keys_t<DT, kCountLarge>(in, out, jobs, njobs, list, batch, bsz, st, stream);
    }
}

template <int DT> cudaError_t launch_small_pairs_t(const Ctx &c, const SmallJob &J) {
    switch (small_size(J.n, 0)) {
    case kCountSmall: return launch_pairs_t<DT, kCountSmall>(c, J);
    case kCountMedium: return launch_pairs_t<DT, kCountMedium>(c, J);
    default: return launch_pairs_t<DT, kCountLarge>(c, J);
    }
}

} // namespace bsps
