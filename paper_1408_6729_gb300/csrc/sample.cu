// sample.cu -- oversampling, splitter selection (Fig. 1 steps
// 3-4 and 6-7, Fig. 3 steps 3-9) and the optional diagnostics.
#include <algorithm>

#include "classify.cuh"
#include "many.cuh"
#include "mlp.cuh"
#include "segsort.cuh"
#include "segsort_keys.cuh"
#include "countsort.cuh"

namespace bsps {

// ---------------------------------------------------------------------------
// Random oversampling (Fig. 3 step 4): s*p-1 positions drawn i.i.d. from the
// Philox4x64-10 stream; the record of draw j is (phi(key[g_j]), g_j).
// ---------------------------------------------------------------------------
template <typename K> struct SampleArgs {
    const K *keys;
    int64_t n, S;
    uint64_t seed;
    K *sphi;
    uint32_t *stag;
    DevStatus *st;          // cleared here, before anything of the call uses them
    uint32_t *cursor, *retry_flag;
    int64_t P;
    uint32_t *state;        // the look-back route's, where both routes of pairs are queued
    int64_t state_words;
};
template <int DT, bool MANY>
__global__ void __launch_bounds__(256) sample_random_kernel(const Many<SampleArgs<typename KeyTraits<DT>::T>> many) {
    const Pick<MANY, SampleArgs<typename KeyTraits<DT>::T>> pk(many);
    const auto &a = pk.a;
    const int64_t blk = (int64_t)pk.block * blockDim.x + threadIdx.x;
    if (blk == 0) *a.st = DevStatus{};
    for (int64_t v = blk; v < a.P; v += (int64_t)pk.blocks * blockDim.x) {
        a.cursor[v] = 0;
        a.retry_flag[v] = 0;
    }
    for (int64_t w = blk; w < a.state_words; w += (int64_t)pk.blocks * blockDim.x) a.state[w] = 0;
    const int64_t j0 = blk * 4;
    if (j0 >= a.S) return;
    uint64_t c[4] = {(uint64_t)blk, 0, 0, 0};
    philox4x64_10(c, a.seed, 0);
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        const int64_t j = j0 + w;
        if (j < a.S) {
            const uint64_t g = __umul64hi(c[w], (uint64_t)a.n);
            a.sphi[j] = KeyTraits<DT>::phi(a.keys[g]);
            a.stag[j] = (uint32_t)g;
        }
    }
}

// ---------------------------------------------------------------------------
// Regular oversampling (Fig. 1 steps 3-4): one cluster of CL CTAs sorts the
// block of virtual processor k stably and emits the records at sorted
// positions j*x - 1, j = 1..s.  Positions at or past the block's key count are
// pads (Lemma 5.1's padding), which follow every key in tag order.  For the
// merge final step (Fig. 1 step 12) the sorted block itself is written too
// (`runs`, with its payloads), at the block's place.
// ---------------------------------------------------------------------------
template <int DT, int CL, int ITEMS>
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(kSortThreads, 1)
run_sample_kernel(const typename KeyTraits<DT>::T *__restrict__ keys, int64_t n, int64_t m,
                  int64_t M, int64_t s, int64_t x, typename KeyTraits<DT>::T *sphi, uint32_t *stag,
                  uint32_t *too_big, const uint32_t *only, typename KeyTraits<DT>::T *runs,
                  const uint32_t *__restrict__ vals, uint32_t *runs_val) {
    using K = typename KeyTraits<DT>::T;
    using SS = SegSort<K, true, CL, ITEMS>;
    if (only && only[blockIdx.x / CL] == 0) return;  // only the blocks the keys-only sort gave back
    extern __shared__ __align__(16) unsigned char smem_raw[];
    typename SS::Smem &sm = *reinterpret_cast<typename SS::Smem *>(smem_raw);
    K *buf = reinterpret_cast<K *>(smem_raw + ((sizeof(typename SS::Smem) + 15) & ~size_t(15)));
    uint32_t *slots = reinterpret_cast<uint32_t *>(buf + SS::CAP);

    const int64_t k = blockIdx.x / CL;
    const int64_t lo = k * m;
    const int64_t len = lo < n ? imin64(m, n - lo) : 0;
    if (blockIdx.x % CL == 0) {  // pads: sorted positions len..M-1, in tag order
        for (int64_t j = 1 + threadIdx.x; j <= s; j += kSortThreads) {
            const int64_t pos = j * x - 1;
            if (pos >= len) {
                sphi[k * s + (j - 1)] = all_ones<K>();
                stag[k * s + (j - 1)] = (uint32_t)(n + k * M + pos);
            }
        }
    }
    if (len == 0) return;
    auto load = [&](int64_t e) { return KeyTraits<DT>::phi(keys[lo + e]); };
    auto emit = [&](uint32_t pos, K key, uint32_t slot) {
        if (runs) {  // the sorted block is kept for the merge final step
            runs[lo + pos] = key;
            if (runs_val) runs_val[lo + pos] = vals[lo + slot];
        }
        if ((pos + 1) % x == 0) {
            const int64_t j = (pos + 1) / x;
            sphi[k * s + (j - 1)] = key;
            stag[k * s + (j - 1)] = (uint32_t)(lo + slot);
        }
    };
    if (!SS::run(sm, buf, slots, len, load, emit) && threadIdx.x == 0 && blockIdx.x % CL == 0)
        atomicExch(too_big, 1u);
}

// The same sample from a faster sort: for 32-bit keys, (phi << 32 | position
// in the block) is unique, so the keys-only cluster sort of segsort_keys.cuh
// orders the block exactly as the stable sort does.  A block it gives back
// is flagged and sorted by run_sample_kernel.
constexpr int kRunKeysItems = 20;  // 512 threads x 20 = 10240 keys per CTA (room for uneven owners)
template <int DT, int CL>
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(512, 1)
run_sample_keys_kernel(const typename KeyTraits<DT>::T *__restrict__ keys, int64_t n, int64_t m, int64_t M,
                       int64_t s, int64_t x, typename KeyTraits<DT>::T *sphi, uint32_t *stag, uint32_t *retry,
                       typename KeyTraits<DT>::T *runs, const uint32_t *__restrict__ vals, uint32_t *runs_val) {
    using K = typename KeyTraits<DT>::T;
    static_assert(sizeof(K) == 4, "32-bit keys and 32-bit positions in one word");
    using SS = SegSortKeys<uint64_t, CL, kRunKeysItems>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int64_t k = blockIdx.x / CL;
    const int64_t lo = k * m;
    const int64_t len = lo < n ? imin64(m, n - lo) : 0;
    if (blockIdx.x % CL == 0) {  // pads: sorted positions len..M-1, in tag order
        for (int64_t j = 1 + threadIdx.x; j <= s; j += blockDim.x) {
            const int64_t pos = j * x - 1;
            if (pos >= len) {
                sphi[k * s + (j - 1)] = all_ones<K>();
                stag[k * s + (j - 1)] = (uint32_t)(n + k * M + pos);
            }
        }
    }
    if (len == 0) return;
    {
        // 64 evenly spaced keys of the block: many repeats mean many equal
        // keys, whose order by position the counting finish cannot resolve;
        // such a block goes to the stable sort at once (every CTA of the
        // cluster reads the same keys and decides alike)
        __shared__ uint32_t probe[64];
        __shared__ int repeats;
        if (threadIdx.x < 64) probe[threadIdx.x] = (uint32_t)KeyTraits<DT>::phi(keys[lo + threadIdx.x * len / 64]);
        if (threadIdx.x == 0) repeats = 0;
        __syncthreads();
        if (threadIdx.x < 64) {
            bool seen = false;
            for (int j = 0; j < (int)threadIdx.x; ++j) seen |= probe[j] == probe[threadIdx.x];
            if (seen) atomicAdd(&repeats, 1);
        }
        __syncthreads();
        if (len >= 64 && repeats > 8) {
            if (threadIdx.x == 0) retry[k] = 1u;
            return;
        }
    }
    auto loadf = [&](uint64_t (&kk)[kRunKeysItems], int64_t e0, int cnt) {
#pragma unroll
        for (int i = 0; i < kRunKeysItems; ++i) {
            const int e = SS::lidx(i);
            if (e < cnt) kk[i] = (uint64_t)KeyTraits<DT>::phi(keys[lo + e0 + e]) << 32 | (uint32_t)(e0 + e);
        }
    };
    const uint32_t xx = (uint32_t)x;
    auto emit = [&](uint32_t pos, uint64_t key) {
        if (runs) {  // the sorted block is kept for the merge final step
            runs[lo + pos] = (K)(key >> 32);
            if (runs_val) runs_val[lo + pos] = vals[lo + (uint32_t)key];
        }
        if ((pos + 1) % xx == 0) {
            const int64_t j = (pos + 1) / xx;
            sphi[k * s + (j - 1)] = (K)(key >> 32);
            stag[k * s + (j - 1)] = (uint32_t)(lo + (uint32_t)key);
        }
    };
    // a split bin of one key value (many equal keys) is ordered by position
    // only, which the counting finish cannot resolve: leave such blocks to the
    // stable sort at once
    auto one_value = [](uint64_t mn, uint64_t mx) { return (mn >> 32) == (mx >> 32); };
    if (!SS::run_load(smem_raw, len, 0ull, ~0ull, loadf, emit, one_value) && threadIdx.x == 0)
        atomicExch(&retry[k], 1u);
}

// ---------------------------------------------------------------------------
// The same sample from the counting sort, when the sorted blocks of keys
// without payloads are kept: a
// block's 32-bit keys (their phi, as they load) are sorted by the streamed
// counting sort of countsort.cuh -- the bucket sort's own -- into
// the sorted block; run_sample_tags_kernel then reads the keys at the sampled
// ranks and finds their tags (input positions).  Equal keys leave
// the counting sort in no particular order, which neither the sorted block
// (keys only) nor the tags (recovered in input order) can reveal.  A block
// the counting sort gives back, or with many repeated keys, is flagged for the
// few-values sampler and the stable block sort.
// ---------------------------------------------------------------------------
template <int DT> struct PhiOf {
    __device__ uint32_t operator()(uint32_t u) const { return (uint32_t)KeyTraits<DT>::phi(u); }
};

template <int DT, int SIZE>
__global__ void __launch_bounds__(CountShape<SIZE>::T, CountShape<SIZE>::kPerSm)
run_sample_count_kernel(const uint32_t *__restrict__ keys, int64_t n, int64_t m, int64_t M, int64_t s, int64_t x,
                        uint32_t *sphi, uint32_t *stag, uint32_t *retry, uint32_t *runs, int G) {
    // (sphi, stag: the pads' records only; the keys' records come from run_sample_tags_kernel)
    using CS = typename CountShape<SIZE>::template Sort<uint32_t>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int64_t k = blockIdx.x / G;
    const int g = (int)(blockIdx.x % G);
    const int64_t lo = k * m;
    const int64_t len = lo < n ? imin64(m, n - lo) : 0;
    if (g == 0) {  // pads: sorted positions len..M-1, in tag order
        for (int64_t j = imax64(1, (len + 1) / x) + threadIdx.x; j <= s; j += blockDim.x) {
            const int64_t pos = j * x - 1;
            if (pos >= len) {
                sphi[k * s + (j - 1)] = 0xffffffffu;
                stag[k * s + (j - 1)] = (uint32_t)(n + k * M + pos);
            }
        }
    }
    if (len == 0) return;
    {
        // many repeats among 64 evenly spaced keys: the few-values sampler
        // (every CTA of the block reads the same keys and decides alike)
        __shared__ uint32_t probe[64];
        __shared__ int repeats;
        if (threadIdx.x < 64) probe[threadIdx.x] = keys[lo + threadIdx.x * len / 64];
        if (threadIdx.x == 0) repeats = 0;
        __syncthreads();
        if (threadIdx.x < 64) {
            bool seen = false;
            for (int j = 0; j < (int)threadIdx.x; ++j) seen |= probe[j] == probe[threadIdx.x];
            if (seen) atomicAdd(&repeats, 1);
        }
        __syncthreads();
        if (len >= 64 && repeats > 8) {
            if (threadIdx.x == 0) retry[k] = 1u;
            return;
        }
    }
    uint32_t kmin, kmax;
    const KeySource<uint32_t, CountShape<SIZE>::T, PhiOf<DT>> src{keys + lo, PhiOf<DT>()};
    CS::bounds(smem_raw, src, (int)len, kmin, kmax);
    auto same = [](uint32_t v) { return v; };
    if (!CS::run(smem_raw, src, (int)len, kmin, kmax, KeySink<uint32_t, decltype(same)>{runs + lo, same}, g, G) &&
        threadIdx.x == 0)
        retry[k] = 1u;
}

// Tags of the sampled keys of a block sorted by run_sample_count_kernel: the
// sampled rank r = j*x - 1 holds key v, the o-th (o = r - first rank of v) of
// the block's keys equal to v in input order (Sec. 5.1.1), so its tag is the
// o-th smallest input position holding v.  One pass over the block's input
// serves every sampled key: a key that occurs once in the block is found
// through a shared-memory hash of those keys; the positions of a repeated one
// are gathered into a list (a second hash gives each such key its list) and
// the o-th smallest is picked.  A block whose sampled keys overflow the
// hash, or whose repeated keys occur too often (more than kTagRunMax times
// each, or too many positions in all), goes to the stable block sort.
constexpr int kTagThreads = 1024, kTagSlotBitsMax = 14, kTagDupBits = 9, kTagDupSlots = 1 << kTagDupBits,
              kTagListMax = 4096, kTagAhead = 8, kTagRunMax = 32;
// hash slots: a power of two at least four times the sampled keys of a block
static int tag_slot_bits(const Plan &p) {
    const int64_t js = p.m / p.x;
    int b = 10;
    while (b < kTagSlotBitsMax && ((int64_t)1 << b) < 4 * js) ++b;
    return b;
}
static size_t tag_smem(int bits) {
    return sizeof(unsigned long long) * (((size_t)1 << bits) + kTagDupSlots) + sizeof(uint32_t) * (kTagDupSlots * 3 + kTagListMax);
}

template <int DT>
__global__ void __launch_bounds__(kTagThreads, 1)
run_sample_tags_kernel(const uint32_t *__restrict__ keys, const uint32_t *__restrict__ runs, int64_t n, int64_t m,
                       int64_t s, int64_t x, int slot_bits, uint32_t *sphi, uint32_t *stag, uint32_t *retry) {
    extern __shared__ __align__(16) unsigned char tag_raw[];
    const int slots = 1 << slot_bits;
    unsigned long long *H = reinterpret_cast<unsigned long long *>(tag_raw);  // key << 32 | j, 0 = empty
    unsigned long long *D = H + slots;                                       // key << 32 | (d + 1): repeated keys
    uint32_t *dcount = reinterpret_cast<uint32_t *>(D + kTagDupSlots);       // occurrences of repeated key d
    uint32_t *dstart = dcount + kTagDupSlots;                                // its list's start
    uint32_t *dfill = dstart + kTagDupSlots;                                 // positions gathered so far
    uint32_t *list = dfill + kTagDupSlots;                                   // the positions
    __shared__ uint32_t ndist, nlist, bad;
    const int64_t k = blockIdx.x;
    if (retry[k]) return;  // the few-values sampler or the stable sort takes it
    const int64_t lo = k * m;
    const int64_t len = lo < n ? imin64(m, n - lo) : 0;
    if (len == 0) return;
    const int64_t js = len / x;  // sampled ranks j*x - 1 inside the block's keys
    if (js == 0) return;
    if (4 * js > slots) {
        if (threadIdx.x == 0) retry[k] = 1u;
        return;
    }
    const uint32_t *blk = runs + lo;
    auto hash = [](uint32_t v, int bits) { return (v * 0x9e3779b1u) >> (32 - bits); };
    for (int i = threadIdx.x; i < slots; i += kTagThreads) H[i] = 0ull;
    for (int i = threadIdx.x; i < kTagDupSlots; i += kTagThreads) {
        D[i] = 0ull;
        dfill[i] = 0;
    }
    if (threadIdx.x == 0) {
        ndist = 0;
        nlist = 0;
        bad = 0;
    }
    __syncthreads();
    // the sampled keys: once-occurring ones into H; repeated ones into D, with
    // their occurrence counts (the run of equal keys around r)
    for (int64_t j = 1 + threadIdx.x; j <= js; j += kTagThreads) {
        const int64_t r = j * x - 1;
        const uint32_t v = blk[r];
        sphi[k * s + (j - 1)] = v;
        if ((r == 0 || blk[r - 1] != v) && (r + 1 == len || blk[r + 1] != v)) {
            const unsigned long long e = (unsigned long long)v << 32 | (uint32_t)j;
            uint32_t h = hash(v, slot_bits);
            for (int probe = 0; probe < slots; ++probe, h = (h + 1) & (slots - 1))
                if (atomicCAS(&H[h], 0ull, e) == 0ull) break;
            continue;
        }
        uint32_t h = hash(v, kTagDupBits);
        for (int probe = 0; probe < kTagDupSlots; ++probe, h = (h + 1) & (kTagDupSlots - 1)) {
            const unsigned long long cur = D[h];
            if (cur != 0ull && (uint32_t)(cur >> 32) == v) break;  // another sampled rank of the same key
            if (cur == 0ull) {
                const uint32_t d = atomicAdd(&ndist, 1u);
                if (d >= kTagDupSlots / 2) {
                    bad = 1;
                    break;
                }
                const unsigned long long want = (unsigned long long)v << 32 | (d + 1);
                const unsigned long long old = atomicCAS(&D[h], 0ull, want);
                if (old == 0ull) {
                    int64_t a = 0, b = r;  // the run of v: [a, c)
                    while (a < b) {
                        const int64_t mid = (a + b) >> 1;
                        if (blk[mid] < v) a = mid + 1;
                        else b = mid;
                    }
                    int64_t lo2 = r, c = len;
                    while (lo2 < c) {
                        const int64_t mid = (lo2 + c) >> 1;
                        if (blk[mid] <= v) lo2 = mid + 1;
                        else c = mid;
                    }
                    const uint32_t cnt = (uint32_t)(c - a);
                    dcount[d] = cnt;
                    const uint32_t at = atomicAdd(&nlist, cnt);
                    if (cnt > (uint32_t)kTagRunMax || at + cnt > (uint32_t)kTagListMax) bad = 1;
                    dstart[d] = at;
                    break;
                }
                if ((uint32_t)(old >> 32) == v) break;
                // the slot went to another key: probe on (d stays unused)
            }
        }
    }
    __syncthreads();
    if (bad) {  // uniform
        if (threadIdx.x == 0) retry[k] = 1u;
        return;
    }
    const bool any_dup = ndist > 0;
    // one pass over the block's input, kTagAhead keys per thread in flight
    for (int64_t t0 = 0; t0 < len; t0 += (int64_t)kTagThreads * kTagAhead) {
        uint32_t u[kTagAhead];
#pragma unroll
        for (int q = 0; q < kTagAhead; ++q) {
            const int64_t t = t0 + q * kTagThreads + threadIdx.x;
            u[q] = t < len ? (uint32_t)KeyTraits<DT>::phi(keys[lo + t]) : 0u;
        }
#pragma unroll
        for (int q = 0; q < kTagAhead; ++q) {
            const int64_t t = t0 + q * kTagThreads + threadIdx.x;
            if (t >= len) continue;
            uint32_t h = hash(u[q], slot_bits);
            for (int probe = 0; probe < slots; ++probe, h = (h + 1) & (slots - 1)) {
                const unsigned long long e = H[h];
                if (e == 0ull) break;
                if ((uint32_t)(e >> 32) == u[q]) {
                    stag[k * s + ((uint32_t)e - 1)] = (uint32_t)(lo + t);
                    break;
                }
            }
            if (any_dup) {
                uint32_t g = hash(u[q], kTagDupBits);
                for (int probe = 0; probe < kTagDupSlots; ++probe, g = (g + 1) & (kTagDupSlots - 1)) {
                    const unsigned long long e = D[g];
                    if (e == 0ull) break;
                    if ((uint32_t)(e >> 32) == u[q]) {
                        const uint32_t d = (uint32_t)e - 1;
                        const uint32_t at = atomicAdd(&dfill[d], 1u);
                        if (at < dcount[d]) list[dstart[d] + at] = (uint32_t)t;
                        break;
                    }
                }
            }
        }
    }
    if (!any_dup) return;
    __syncthreads();
    // repeated keys: the o-th smallest of the gathered positions
    for (int64_t j = 1 + threadIdx.x; j <= js; j += kTagThreads) {
        const int64_t r = j * x - 1;
        const uint32_t v = blk[r];
        if ((r == 0 || blk[r - 1] != v) && (r + 1 == len || blk[r + 1] != v)) continue;
        uint32_t g = hash(v, kTagDupBits), d = 0;
        for (int probe = 0; probe < kTagDupSlots; ++probe, g = (g + 1) & (kTagDupSlots - 1)) {
            const unsigned long long e = D[g];
            if (e == 0ull) break;
            if ((uint32_t)(e >> 32) == v) {
                d = (uint32_t)e - 1;
                break;
            }
        }
        int64_t a = 0, b = r;  // the first rank of v
        while (a < b) {
            const int64_t mid = (a + b) >> 1;
            if (blk[mid] < v) a = mid + 1;
            else b = mid;
        }
        const uint32_t o = (uint32_t)(r - a), c = dcount[d], *L = list + dstart[d];
        uint32_t tag = 0;
        for (uint32_t i = 0; i < c; ++i) {  // the position with exactly o smaller ones
            uint32_t below = 0;
            for (uint32_t q = 0; q < c; ++q) below += L[q] < L[i];
            if (below == o) tag = L[i];
        }
        stag[k * s + (j - 1)] = (uint32_t)(lo + tag);
    }
}

// ---------------------------------------------------------------------------
// Blocks of few distinct keys (regular sampling, 32-bit keys): a block's
// sorted order by (phi, tag) is its distinct values in order, each repeated in
// position order.  One CTA finds the values with a shared-memory hash table;
// warp w of the CTA owns the w-th of 32 contiguous segments of the block and
// counts the values in it.  From the counts come the distinct values' sorted
// starts and, per warp, the keys of each value in earlier segments.  Every
// warp then walks its segment again in position order: the sorted rank of a
// key is the start of its value, plus that value's keys in earlier segments,
// plus its earlier occurrences in this segment (a running count and the lanes
// of the same value below it).  The records at ranks j*x - 1 are emitted
// without sorting.  When the sorted block is kept, its keys are written as
// runs of equal values in position order and every payload at its key's rank
// (a stable counting sort).  Blocks with more than kLowCardMax values keep their flag
// for the stable block sort.
//
// Bound by instructions and shared-memory latency, not bytes.  The table is
// read two slots at a time and at most a quarter full where counts of 16 bits
// do (blocks of at most kLowCardStashMax keys), so few keys probe twice; there
// the first pass also leaves, for each key, its slot and its place among the
// equal keys of its step (16 bits), and the second neither matches lanes nor
// reads the table.  2^28 Zipf pairs in blocks of 2^16: 3.45 ms when both passes
// matched and probed a table half full one slot at a time, 3.29 with the
// places kept, 2.86 with the pairs of slots.
constexpr int kLowCardThreads = 1024, kLowCardMax = 256;
constexpr int kLowCardWarps = kLowCardThreads / 32;
constexpr int64_t kLowCardStashMax = 65536;
template <bool STASH> struct LowCard {
    using Count = typename std::conditional<STASH, uint16_t, uint32_t>::type;
    static constexpr int kBits = STASH ? 10 : 9, NS = 1 << kBits;
    static constexpr size_t kCounts = sizeof(Count) * kLowCardWarps * NS;
    static size_t smem(int64_t m) { return kCounts + (STASH ? 2 * (size_t)m : 0); }
};
template <int DT, bool STASH>
__global__ void __launch_bounds__(kLowCardThreads, 1)
run_sample_lowcard_kernel(const typename KeyTraits<DT>::T *__restrict__ keys, int64_t n, int64_t m, int64_t s,
                          int64_t x, typename KeyTraits<DT>::T *sphi, uint32_t *stag, uint32_t *retry,
                          typename KeyTraits<DT>::T *runs, const uint32_t *__restrict__ vals_in,
                          uint32_t *runs_val) {
    using K = typename KeyTraits<DT>::T;
    using Count = typename LowCard<STASH>::Count;
    static_assert(sizeof(K) == 4, "32-bit keys");
    constexpr int T = kLowCardThreads, W = kLowCardWarps, NS = LowCard<STASH>::NS;
    extern __shared__ __align__(16) unsigned char low_smem[];
    Count *wcnt = reinterpret_cast<Count *>(low_smem);                         // [W][NS]: keys per slot in warp w's segment
    uint16_t *word16 = reinterpret_cast<uint16_t *>(low_smem + LowCard<STASH>::kCounts);  // per key, for the second pass
    __shared__ __align__(16) unsigned long long slot[NS];   // (1 << 32) | phi, 0 = empty
    __shared__ uint32_t start[NS];                          // sorted start of the slot's value
    __shared__ uint32_t vals[kLowCardMax], sid[kLowCardMax], rank_of[kLowCardMax], tot_sorted[kLowCardMax];
    __shared__ uint32_t val_of_rank[kLowCardMax];
    __shared__ uint32_t tmp[W + 1];
    __shared__ int ndistinct, overflow;
    const int64_t k = blockIdx.x;
    if (retry[k] == 0) return;  // sorted by the keys-only block sort
    const uint32_t xx = (uint32_t)x;
    const int64_t lo = k * m;
    const int64_t len64 = lo < n ? imin64(m, n - lo) : 0;  // < 2^32 (positions are 32 bits wide)
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int i = tid; i < NS; i += T) slot[i] = 0ull;
    for (int i = tid; i < (int)(LowCard<STASH>::kCounts / 16); i += T)
        reinterpret_cast<uint4 *>(low_smem)[i] = make_uint4(0u, 0u, 0u, 0u);
    if (tid == 0) {
        ndistinct = 0;
        overflow = 0;
    }
    __syncthreads();
    auto hash = [](uint32_t f) {  // murmur3's 32-bit finaliser, its top bits: the first of a pair of slots
        f ^= f >> 16;
        f *= 0x85ebca6bu;
        f ^= f >> 13;
        f *= 0xc2b2ae35u;
        f ^= f >> 16;
        return f >> (33 - LowCard<STASH>::kBits) << 1;
    };
    // slot holding f, inserted when absent; -1 when the table is full
    auto find = [&](uint32_t f, uint32_t h) -> int {
        const unsigned long long want = (1ull << 32) | f;
        for (int probe = 0; probe < NS; ++probe, h = (h + 1) & (NS - 1)) {
            unsigned long long cur = slot[h];
            if (cur == want) return (int)h;
            if (cur == 0ull) {
                cur = atomicCAS(&slot[h], 0ull, want);
                if (cur == 0ull) {
                    if (atomicAdd(&ndistinct, 1) >= kLowCardMax) overflow = 1;
                    return (int)h;
                }
                if (cur == want) return (int)h;
            }
        }
        return -1;
    };
    // warp w's segment of the block: [seg0, seg1), whole steps of 32 keys
    const uint32_t len = (uint32_t)len64, seg = ((len + W - 1) / W + 31) / 32 * 32;
    const uint32_t seg0 = min(len, warp * seg), seg1 = min(len, seg0 + seg);
    Count *mine = wcnt + warp * NS;
    // keys of kAhead steps of 32 are loaded before the first is used
    constexpr int kAhead = 8;
    const K *blk = keys + lo;
    // What a key needs in the second pass: its slot, the keys of its value in
    // lower lanes of its step, whether no higher lane has one.
    constexpr uint32_t kBelow = LowCard<STASH>::kBits, kLast = kBelow + 5;
    uint32_t word[kAhead];
    auto look_up = [&](uint32_t e0, bool count, auto full) {
        uint32_t f[kAhead];
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            const uint32_t e = e0 + u * 32 + lane;
            f[u] = decltype(full)::value || e < seg1 ? (uint32_t)KeyTraits<DT>::phi(blk[e]) : 0u;
        }
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            const bool ok = decltype(full)::value || e0 + u * 32 + lane < seg1;
            uint32_t peers = __match_any_sync(0xffffffffu, f[u]);
            if (!decltype(full)::value) peers &= __ballot_sync(0xffffffffu, ok);
            const uint32_t h = hash(f[u]);
            const ulonglong2 e = *reinterpret_cast<const ulonglong2 *>(&slot[h]);
            const unsigned long long want = (1ull << 32) | f[u];
            const bool one = e.x == want, two = e.y == want;
            word[u] = h + (two ? 1u : 0u);
            if (!(one || two) && ok) {
                const int at = find(f[u], h);
                if (at < 0) overflow = 1;
                word[u] = (uint32_t)max(at, 0);
            }
            const uint32_t below = (uint32_t)__popc(peers & lanemask_lt()), all = (uint32_t)__popc(peers);
            if (count && below == 0 && ok) {
                if constexpr (STASH)  // (a segment's count has 16 bits to spare: no carry)
                    atomicAdd(reinterpret_cast<uint32_t *>(mine) + (word[u] >> 1), all << (16 * (word[u] & 1u)));
                else
                    atomicAdd(&mine[word[u]], all);
            }
            word[u] |= below << kBelow | (below + 1 == all ? 1u : 0u) << kLast;
        }
    };
    // pass 1: distinct values, and their keys per segment
    auto first_pass = [&](uint32_t e0, auto full) {
        look_up(e0, true, full);
        if constexpr (STASH) {
#pragma unroll
            for (int u = 0; u < kAhead; ++u)
                if (decltype(full)::value || e0 + u * 32 + lane < seg1) word16[e0 + u * 32 + lane] = (uint16_t)word[u];
        }
    };
    for (uint32_t e0 = seg0; e0 < seg1; e0 += 32 * kAhead) {
        if (e0 + 32 * kAhead <= seg1) first_pass(e0, std::true_type{});
        else first_pass(e0, std::false_type{});
        if (__any_sync(0xffffffffu, *(volatile int *)&overflow)) break;  // (the warp as one)
    }
    __syncthreads();
    if (overflow || ndistinct > kLowCardMax) return;  // leave the block to the stable sort
    const int nd = ndistinct;
    // the distinct values, compacted in slot order (ballots over the slots)
    if (tid < NS) {
        const uint32_t b = __ballot_sync(0xffffffffu, slot[tid] != 0ull);
        if (lane == 0) tmp[warp] = (uint32_t)__popc(b);
    }
    __syncthreads();
    if (tid < NS) {
        const bool occ = slot[tid] != 0ull;
        uint32_t c = (uint32_t)__popc(__ballot_sync(0xffffffffu, occ) & lanemask_lt());
        for (int w = 0; w < warp; ++w) c += tmp[w];
        if (occ) {
            vals[c] = (uint32_t)slot[tid];
            sid[c] = (uint32_t)tid;
        }
    }
    __syncthreads();
    // value rank = number of smaller values; per value its total and, per
    // warp, its keys in earlier segments (in place of the counts)
    if (tid < nd) {
        uint32_t r = 0;
        const uint32_t v = vals[tid];
        for (int j = 0; j < nd; ++j) r += vals[j] < v;
        rank_of[tid] = r;
        const uint32_t h = sid[tid];
        uint32_t acc = 0;
        for (int w = 0; w < W; ++w) {
            const uint32_t b = wcnt[w * NS + h];
            wcnt[w * NS + h] = acc;
            acc += b;
        }
        tot_sorted[r] = acc;
    }
    __syncthreads();
    // first sorted position of every value: exclusive scan in rank order
    uint32_t ex = 0;
    if (tid < kLowCardMax) {
        uint32_t wt;
        ex = warp_excl_scan(tid < nd ? tot_sorted[tid] : 0u, &wt);
        if (lane == 31) tmp[warp] = wt;
    }
    __syncthreads();
    if (tid < nd) {
        for (int w = 0; w < warp; ++w) ex += tmp[w];
        tot_sorted[tid] = ex;
    }
    __syncthreads();
    if (tid < nd) {
        start[sid[tid]] = tot_sorted[rank_of[tid]];
        val_of_rank[rank_of[tid]] = vals[tid];
    }
    __syncthreads();
    if (runs) {
        // the sorted block's keys: value of rank r over [start_r, start_r+1),
        // written in position order.  Warp w writes positions [w*len/W,
        // (w+1)*len/W), 32 consecutive ones at a time; each lane finds the
        // rank of its first position and then walks forward.
        const int64_t p0 = (int64_t)warp * len / W, p1 = (int64_t)(warp + 1) * len / W;
        int r = 0;
        if (p0 + lane < p1) {
            int l = 0, h = nd - 1;  // the last rank starting at or before the position
            while (l < h) {
                const int mid = (l + h + 1) >> 1;
                if (tot_sorted[mid] <= (uint32_t)(p0 + lane)) l = mid;
                else h = mid - 1;
            }
            r = l;
        }
        for (int64_t t = p0 + lane; t < p1; t += 32) {
            while (r + 1 < nd && tot_sorted[r + 1] <= (uint32_t)t) ++r;
            runs[lo + t] = (K)val_of_rank[r];
        }
    }
    // the rank of each value's first key of this segment
    for (int h = lane; h < NS; h += 32) mine[h] += (Count)start[h];
    __syncwarp();
    // pass 2: in position order, sorted rank = first rank + earlier here
    // j = g / x when x divides g: a rounded float quotient is exact below 2^21
    const float inv_x = 1.0f / (float)xx;
    const bool few = s < (int64_t)1 << 21;
    const uint32_t *val_blk = vals_in + lo;
    uint32_t *val_run = runs_val + lo;
    K *sample_phi = sphi + k * s - 1;
    uint32_t *sample_tag = stag + k * s - 1;
    auto second_pass = [&](uint32_t e0, auto full) {
        if constexpr (STASH) {
#pragma unroll
            for (int u = 0; u < kAhead; ++u) {
                const uint32_t e = e0 + u * 32 + lane;
                word[u] = decltype(full)::value || e < seg1 ? word16[e] : 0u;
            }
        } else {
            look_up(e0, false, full);
        }
        uint32_t va[kAhead];  // the payloads of the kAhead steps, loaded before the first is stored
        if (runs_val) {
#pragma unroll
            for (int u = 0; u < kAhead; ++u) {
                const uint32_t e = e0 + u * 32 + lane;
                va[u] = decltype(full)::value || e < seg1 ? val_blk[e] : 0u;
            }
        }
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            const uint32_t e = e0 + u * 32 + lane;
            const uint32_t h = word[u] & (NS - 1), g = mine[h] + (word[u] >> kBelow & 31u) + 1;  // rank, from one
            __syncwarp();
            if (decltype(full)::value || e < seg1) {
                if (word[u] >> kLast & 1u) mine[h] = (Count)g;
                if (runs_val) val_run[g - 1] = va[u];  // payloads at their ranks
                const uint32_t j = few ? __float2uint_rn((float)g * inv_x) : g / xx;
                if (j * xx == g) {
                    sample_phi[j] = (K)(uint32_t)slot[h];
                    sample_tag[j] = (uint32_t)(lo + e);
                }
            }
            __syncwarp();
        }
    };
    for (uint32_t e0 = seg0; e0 < seg1; e0 += 32 * kAhead) {
        if (e0 + 32 * kAhead <= seg1) second_pass(e0, std::true_type{});
        else second_pass(e0, std::false_type{});
    }
    if (tid == 0) retry[k] = 0;  // done
}

// ---------------------------------------------------------------------------
// Splitter selection (Fig. 1 step 6): splitter i of the p buckets is the
// sample record of 1-indexed rank i*Q (Q = q regular, s random).  Each bucket
// is refined into B sub-buckets by the records of rank floor(j*Q/B); for
// j = i*B these are the paper's splitters, so the buckets are unchanged.
// "Broadcast" (Fig. 1 step 7) is the copy into every CTA's shared memory.
// ---------------------------------------------------------------------------
template <typename K> struct SplitterArgs {
    const K *phi;
    const uint32_t *tag;
    int64_t P, Q, B;
    K *vphi;
    uint32_t *vtag;
    LutParams<K> *lutp;
    uint16_t *lut;
    int lut_bits;
    uint32_t probes;        // neighbours in the sample compared, counted in *repeats
    int64_t S;
    uint32_t *repeats;
};
template <typename K, bool MANY>
__global__ void __launch_bounds__(256) splitter_kernel(const Many<SplitterArgs<K>> many) {
    const Pick<MANY, SplitterArgs<K>> pk(many);
    const K *phi = pk.a.phi;
    const uint32_t *tag = pk.a.tag;
    const int64_t P = pk.a.P, Q = pk.a.Q, B = pk.a.B;
    K *vphi = pk.a.vphi;
    uint32_t *vtag = pk.a.vtag;
    LutParams<K> *lutp = pk.a.lutp;
    uint16_t *lut = pk.a.lut;
    const int lut_bits = pk.a.lut_bits;
    auto rank = [&](int64_t j) { return (j * Q) / B - 1; };  // sorted index of splitter j, 1 <= j < P
    LutParams<K> lp;
    lp.base = P > 1 ? phi[rank(1)] : K(0);
    lp.span = P > 1 ? phi[rank(P - 1)] - lp.base : K(0);
    const int bl = bit_length<K>(lp.span);
    lp.shift = bl > lut_bits ? (uint32_t)(bl - lut_bits) : 0u;
    lp.nsplit = (uint32_t)(P - 1);
    const int64_t t = (int64_t)pk.block * blockDim.x + threadIdx.x;
    if (t == 0) *lutp = lp;
    if (t < P - 1) {
        const int64_t r = rank(t + 1);
        vphi[t] = phi[r];
        vtag[t] = tag[r];
    } else if (t == P - 1) {  // above every key, for comparisons without a bounds check
        vphi[t] = all_ones<K>();
        vtag[t] = 0xffffffffu;
    }
    if (pk.a.probes > 0) {
        bool same = false;
        if (t < pk.a.probes) {
            const int64_t r = t * (pk.a.S - 1) / pk.a.probes;
            same = phi[r] == phi[r + 1];
        }
        const uint32_t m = __ballot_sync(0xffffffffu, same);
        if (m && (threadIdx.x & 31) == 0) atomicAdd(pk.a.repeats, (uint32_t)__popc(m));
    }
    // the radix index, from the sorted sample itself
    if (t <= (1 << lut_bits))
        lut[t] = (uint16_t)lut_cell((uint32_t)t, lp, [&](uint32_t i) { return phi[rank((int64_t)i + 1)]; });
}

// ---------------------------------------------------------------------------
// Diagnostics: records in the paper's tag form, per-key buckets, pad counts.
// ---------------------------------------------------------------------------
template <typename K>
__device__ __forceinline__ bsps_record to_record(K phi, uint32_t tag, int64_t n, int64_t m, int64_t M,
                                                 bool regular) {
    bsps_record r;
    if ((int64_t)tag >= n) {
        r.phi = ~0ull;
        r.tag = (uint64_t)tag - (uint64_t)n;
        r.pad = 1;
    } else {
        r.phi = (uint64_t)phi;
        r.tag = regular ? (uint64_t)(tag / m) * M + tag % m : tag;
        r.pad = 0;
    }
    r.reserved = 0;
    return r;
}

template <typename K>
__global__ void sample_records_kernel(RecordBuffers<K> b, int fin, int64_t S,
                                      int64_t n, int64_t m, int64_t M, bool regular, bsps_record *out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < S) out[i] = to_record(b.phi[fin][i], b.tag[fin][i], n, m, M, regular);
}

template <typename K>
__global__ void splitter_records_kernel(const K *vphi, const uint32_t *vtag, int64_t p, int64_t B,
                                        int64_t n, int64_t m, int64_t M, bool regular,
                                        bsps_record *out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x + 1;
    if (i < p) out[i - 1] = to_record(vphi[i * B - 1], vtag[i * B - 1], n, m, M, regular);
}

// Per-key buckets of the keys (diagnostics).  With the learned classifier
// every key goes through the same classify_learned (network, index over its
// output, search and check) the routing kernels use, so its result can be
// compared key by key.
template <int DT, bool LEARNED>
__global__ void __launch_bounds__(256) bucket_of_kernel(const typename KeyTraits<DT>::T *keys, int64_t n, int64_t B,
                                 const typename KeyTraits<DT>::T *vphi, const uint32_t *vtag,
                                 const uint16_t *lut,
                                 const LutParams<typename KeyTraits<DT>::T> *lutp, const MlpTables *mlp_tables,
                                 const uint16_t *ylut, int64_t P, uint32_t tag_floor, int32_t *out) {
    __shared__ __align__(16) unsigned char mt_raw[LEARNED ? sizeof(MlpTables) : 16];
    const MlpTables *mt = reinterpret_cast<const MlpTables *>(mt_raw);
    if constexpr (LEARNED) {
        const uint32_t *src = reinterpret_cast<const uint32_t *>(mlp_tables);
        uint32_t *dst = reinterpret_cast<uint32_t *>(mt_raw);
        for (int q = threadIdx.x; q < (int)(sizeof(MlpTables) / 4); q += blockDim.x) dst[q] = src[q];
        __syncthreads();
    }
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= n) return;
    uint32_t v;
    if constexpr (LEARNED) {
        uint32_t steps;
        bool mis;
        v = classify_learned<DT>(keys[g], max((uint32_t)g, tag_floor), *mt, ylut, (uint32_t)(P - 1), vphi, vtag,
                                 steps, mis);
    } else {
        const LutParams<typename KeyTraits<DT>::T> lp = *lutp;
        v = classify_key(KeyTraits<DT>::phi(keys[g]), max((uint32_t)g, tag_floor), lp, lut, vphi, vtag);
    }
    out[g] = (int32_t)(v / B);
}

template <typename K>
__global__ void pad_sizes_kernel(int64_t n, int64_t R, int64_t m, int64_t M, int64_t B, const K *vphi,
                                 const uint32_t *vtag, const uint16_t *lut, const LutParams<K> *lutp,
                                 int dup_off, unsigned long long *out) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= R * M) return;
    const int64_t k = t / M, j = t % M;
    const int64_t len = k * m < n ? min(m, n - k * m) : 0;
    if (j < len) return;
    const LutParams<K> lp = *lutp;
    // without tags a pad equals the pad splitters and follows them all
    const uint32_t tag = dup_off ? 0xffffffffu : (uint32_t)(n + k * M + j);
    const uint32_t v = classify_key(all_ones<K>(), tag, lp, lut, vphi, vtag);
    atomicAdd(&out[v / B], 1ull);
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
template <int DT> static RecordBuffers<typename KeyTraits<DT>::T> record_buffers(const Ctx &c) {
    using K = typename KeyTraits<DT>::T;
    RecordBuffers<K> b;
    b.phi[0] = (K *)c.ly.sphi[0];
    b.phi[1] = (K *)c.ly.sphi[1];
    b.tag[0] = c.ly.stag[0];
    b.tag[1] = c.ly.stag[1];
    return b;
}

template <int DT, int CL, int ITEMS> static cudaError_t launch_run_sample(const Ctx &c, const uint32_t *only) {
    using K = typename KeyTraits<DT>::T;
    using SS = SegSort<K, true, CL, ITEMS>;
    const size_t smem = SS::smem_bytes();
    auto kern = run_sample_kernel<DT, CL, ITEMS>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const Plan &p = c.pl;
    kern<<<(unsigned)(p.R * CL), kSortThreads, smem, c.stream>>>(
        (const K *)c.keys_in, p.n, p.m, p.M, p.s, p.x, (K *)c.ly.sphi[0], c.ly.stag[0],
        (uint32_t *)&c.ly.status->run_too_big, only, p.keep_runs ? (K *)c.ly.runs : nullptr, c.vals_in,
        p.keep_runs && p.pairs ? c.ly.runs_val : nullptr);
    return cudaGetLastError();
}

template <int DT, int CL> static cudaError_t launch_run_sample_keys(const Ctx &c) {
    using K = typename KeyTraits<DT>::T;
    using SS = SegSortKeys<uint64_t, CL, kRunKeysItems>;
    const size_t smem = SS::smem_bytes();
    auto kern = run_sample_keys_kernel<DT, CL>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const Plan &p = c.pl;
    e = cudaMemsetAsync(c.ly.run_retry, 0, (size_t)p.R * 4, c.stream);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)(p.R * CL), 512, smem, c.stream>>>(
        (const K *)c.keys_in, p.n, p.m, p.M, p.s, p.x, (K *)c.ly.sphi[0], c.ly.stag[0], c.ly.run_retry,
        p.keep_runs ? (K *)c.ly.runs : nullptr, c.vals_in, p.keep_runs && p.pairs ? c.ly.runs_val : nullptr);
    return cudaGetLastError();
}

// the kept blocks are sorted by the counting sort: keys without payloads (it
// moves keys only)
bool counting_block_sort(const Ctx &c) {
    const Plan &p = c.pl;
    return p.keep_runs && !p.pairs && p.key_bytes == 4 && run_keys_cluster(p) != 0;
}

template <int DT, int SIZE> static cudaError_t launch_run_sample_count(const Ctx &c) {
    using CS = typename CountShape<SIZE>::template Sort<uint32_t>;
    auto kern = run_sample_count_kernel<DT, SIZE>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CS::smem_bytes());
    if (e != cudaSuccess) return e;
    const Plan &p = c.pl;
    e = cudaMemsetAsync(c.ly.run_retry, 0, (size_t)p.R * 4, c.stream);
    if (e != cudaSuccess) return e;
    const int G = count_sort_ctas<SIZE>(p.R, p.m);
    kern<<<(unsigned)(p.R * G), CountShape<SIZE>::T, CS::smem_bytes(), c.stream>>>(
        (const uint32_t *)c.keys_in, p.n, p.m, p.M, p.s, p.x, (uint32_t *)c.ly.sphi[0], c.ly.stag[0], c.ly.run_retry,
        (uint32_t *)c.ly.runs, G);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int bits = tag_slot_bits(p);
    e = cudaFuncSetAttribute(run_sample_tags_kernel<DT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)tag_smem(kTagSlotBitsMax));
    if (e != cudaSuccess) return e;
    run_sample_tags_kernel<DT><<<(unsigned)p.R, kTagThreads, tag_smem(bits), c.stream>>>(
        (const uint32_t *)c.keys_in, (const uint32_t *)c.ly.runs, p.n, p.m, p.s, p.x, bits,
        (uint32_t *)c.ly.sphi[0], c.ly.stag[0], c.ly.run_retry);
    return cudaGetLastError();
}

// cluster size of the keys-only block sort (0: not used)
int run_keys_cluster(const Plan &p) {
    if (p.sampling != BSPS_REGULAR || p.key_bytes != 4 || p.m >= ((int64_t)1 << 32)) return 0;
    for (int cl = 1; cl <= 8; cl *= 2)
        if (p.m <= (int64_t)cl * 512 * kRunKeysItems) return cl;
    return 0;
}

template <int DT> static cudaError_t launch_sample_t(const Ctx &c) {
    using K = typename KeyTraits<DT>::T;
    const Plan &p = c.pl;
    const uint32_t *only = nullptr;
    if constexpr (sizeof(K) == 4) {
        cudaError_t e = cudaSuccess;
        if (counting_block_sort(c)) {
            switch (count_sort_size(p.m, 4)) {
            case kCountSmall: e = launch_run_sample_count<DT, kCountSmall>(c); break;
            case kCountMedium: e = launch_run_sample_count<DT, kCountMedium>(c); break;
            default: e = launch_run_sample_count<DT, kCountLarge>(c); break;
            }
            only = c.ly.run_retry;
        } else {
            switch (run_keys_cluster(p)) {
            case 0: break;
            case 1: e = launch_run_sample_keys<DT, 1>(c); only = c.ly.run_retry; break;
            case 2: e = launch_run_sample_keys<DT, 2>(c); only = c.ly.run_retry; break;
            case 4: e = launch_run_sample_keys<DT, 4>(c); only = c.ly.run_retry; break;
            default: e = launch_run_sample_keys<DT, 8>(c); only = c.ly.run_retry; break;
            }
        }
        if (e != cudaSuccess) return e;
        if (only) {  // blocks of few distinct keys, before the stable sort
            const bool stash = p.m <= kLowCardStashMax;
            auto kern = stash ? run_sample_lowcard_kernel<DT, true> : run_sample_lowcard_kernel<DT, false>;
            const DynSmem smem = stash ? DynSmem(LowCard<true>::smem(p.m), LowCard<true>::smem(kLowCardStashMax))
                                       : DynSmem(LowCard<false>::smem(p.m));
            e = smem.allow(kern);
            if (e != cudaSuccess) return e;
            kern<<<(unsigned)p.R, kLowCardThreads, smem.bytes, c.stream>>>(
                (const K *)c.keys_in, p.n, p.m, p.s, p.x, (K *)c.ly.sphi[0], c.ly.stag[0], c.ly.run_retry,
                p.keep_runs ? (K *)c.ly.runs : nullptr, c.vals_in, p.keep_runs && p.pairs ? c.ly.runs_val : nullptr);
            e = cudaGetLastError();
            if (e != cudaSuccess) return e;
        }
    }
    constexpr int IT = sizeof(K) == 8 ? kRunItems64 : kRunItems32;
    switch (p.run_cl) {
    case 1: return launch_run_sample<DT, 1, IT>(c, only);
    case 2: return launch_run_sample<DT, 2, IT>(c, only);
    case 4: return launch_run_sample<DT, 4, IT>(c, only);
    case 8: return launch_run_sample<DT, 8, IT>(c, only);
    default: return cudaErrorInvalidValue;
    }
}

template <int DT> static cudaError_t launch_sample_random_t(Exec &x) {
    using K = typename KeyTraits<DT>::T;
    return launch_calls<SampleArgs<K>>(x, sample_random_kernel<DT, false>, sample_random_kernel<DT, true>, 256, 0,
                                       [](const Ctx &c, SampleArgs<K> &a) {
        const Plan &p = c.pl;
        a = {(const K *)c.keys_in, p.n, p.sample_size, p.seed, (K *)c.ly.sphi[0], c.ly.stag[0], c.ly.status, c.ly.cursor,
             c.ly.retry_flag, p.P, c.ly.state, c.both_routes ? p.tiles * p.P : 0};
        return (uint32_t)imax64(1, (p.sample_size + 1023) / 1024);
    });
}

cudaError_t launch_sample_random(Exec &x) {
    switch (x.calls[0].pl.dtype) {
    case BSPS_U32: return launch_sample_random_t<BSPS_U32>(x);
    case BSPS_I32: return launch_sample_random_t<BSPS_I32>(x);
    case BSPS_F32: return launch_sample_random_t<BSPS_F32>(x);
    default: return launch_sample_random_t<BSPS_F64>(x);
    }
}

cudaError_t launch_sample(const Ctx &c) {
    switch (c.pl.dtype) {
    case BSPS_U32: return launch_sample_t<BSPS_U32>(c);
    case BSPS_I32: return launch_sample_t<BSPS_I32>(c);
    case BSPS_F32: return launch_sample_t<BSPS_F32>(c);
    default: return launch_sample_t<BSPS_F64>(c);
    }
}

template <typename K> static RecordBuffers<K> buffers_of(const Ctx &c) {
    RecordBuffers<K> b;
    b.phi[0] = (K *)c.ly.sphi[0];
    b.phi[1] = (K *)c.ly.sphi[1];
    b.tag[0] = c.ly.stag[0];
    b.tag[1] = c.ly.stag[1];
    return b;
}

template <typename K> static cudaError_t launch_splitters_t(Exec &x) {
    return launch_calls<SplitterArgs<K>>(x, splitter_kernel<K, false>, splitter_kernel<K, true>, 256, 0,
                                         [](const Ctx &c, SplitterArgs<K> &a) {
        const Plan &p = c.pl;
        const RecordBuffers<K> b = buffers_of<K>(c);
        const int fin = sample_final(p);
        a = {b.phi[fin], b.tag[fin], p.P, p.Q, p.B, (K *)c.ly.vphi, c.ly.vtag, (LutParams<K> *)c.ly.lutp, c.ly.lut, p.lut_bits,
             c.both_routes ? repeat_probes(p) : 0u, p.sample_size, &c.ly.status->repeats};
        static_assert(kRepeatProbes <= kLutCells, "a thread for each probe");
        return (uint32_t)((imax64(p.P, (1 << p.lut_bits) + 1) + 255) / 256);
    });
}

cudaError_t launch_splitters(Exec &x) {
    return x.calls[0].pl.key_bytes == 8 ? launch_splitters_t<uint64_t>(x) : launch_splitters_t<uint32_t>(x);
}

template <int DT> static cudaError_t launch_debug_t(const Ctx &c) {
    using K = typename KeyTraits<DT>::T;
    const Plan &p = c.pl;
    const bool regular = p.sampling == BSPS_REGULAR;
    RecordBuffers<K> b = record_buffers<DT>(c);
    if (c.dbg.sample && p.sample_size > 0)
        sample_records_kernel<K><<<(unsigned)((p.sample_size + 255) / 256), 256, 0, c.stream>>>(
            b, sample_final(p), p.sample_size, p.n, p.m, p.M, regular, c.dbg.sample);
    if (c.dbg.splitters && p.p > 1)
        splitter_records_kernel<K><<<(unsigned)((p.p + 255) / 256), 256, 0, c.stream>>>(
            (const K *)c.ly.vphi, c.ly.vtag, p.p, p.B, p.n, p.m, p.M, regular, c.dbg.splitters);
    if (c.dbg.bucket_of && p.n > 0) {
        auto kern = p.classify == BSPS_LEARNED ? bucket_of_kernel<DT, true> : bucket_of_kernel<DT, false>;
        kern<<<(unsigned)((p.n + 255) / 256), 256, 0, c.stream>>>(
            (const K *)c.keys_in, p.n, p.B, (const K *)c.ly.vphi, c.ly.vtag, c.ly.lut,
            (const LutParams<K> *)c.ly.lutp, c.ly.mlp_tables, c.ly.ylut, p.P,
            p.dup_off ? (uint32_t)(p.n - 1) : 0u, c.dbg.bucket_of);
    }
    if (c.dbg.pad_sizes) {
        cudaError_t e = cudaMemsetAsync(c.dbg.pad_sizes, 0, sizeof(int64_t) * p.p, c.stream);
        if (e != cudaSuccess) return e;
        if (regular && p.R * p.M > p.n)
            pad_sizes_kernel<K><<<(unsigned)((p.R * p.M + 255) / 256), 256, 0, c.stream>>>(
                p.n, p.R, p.m, p.M, p.B, (const K *)c.ly.vphi, c.ly.vtag, c.ly.lut,
                (const LutParams<K> *)c.ly.lutp, p.dup_off, (unsigned long long *)c.dbg.pad_sizes);
    }
    return cudaGetLastError();
}

cudaError_t launch_debug(const Ctx &c) {
    switch (c.pl.dtype) {
    case BSPS_U32: return launch_debug_t<BSPS_U32>(c);
    case BSPS_I32: return launch_debug_t<BSPS_I32>(c);
    case BSPS_F32: return launch_debug_t<BSPS_F32>(c);
    default: return launch_debug_t<BSPS_F64>(c);
    }
}

} // namespace bsps
