// sample_sort.cu -- the sort of the sample's records (Fig. 1 step 5).
#include <algorithm>

#include "classify.cuh"
#include "countsort.cuh"
#include "many.cuh"

namespace bsps {

// ---------------------------------------------------------------------------
// Sample sort (Fig. 1 step 5): the records (phi, tag) in order.  A sample of at
// most kOneSample records is sorted by one CTA.  A larger one is itself sample
// sorted, which no distribution of the keys unbalances: one CTA sorts
// candidates, one drawn from each of equal stretches of the sample (a plain
// stride would meet the same rank of every block of a regular sample), every
// few of them is a pivot (and where several pivots share a key value, so are
// that value's first and last possible record: a bin then holds no part of it
// beside other values, whose tags and phi would spread it unevenly), the
// records are counted and scattered into the
// pivots' bins, and every bin is sorted on chip by the counting sort of
// countsort.cuh over words phi << 32 | tag.  Four
// launches for any sample (an LSD radix sort over the record's bytes, which
// this replaces, took 24 to 36 of them): 6.4M records 0.29 ms, before 0.34;
// 16.8M of Zipf keys 0.81, before 0.90; 16K records 0.04, before 0.13 (one CTA
// up to kOneSample records, where the bins would not fill the GPU).
// ---------------------------------------------------------------------------
constexpr int64_t kOneSample = 8192;
constexpr int kPivotBinsMax = 4096;
constexpr int kPivotCells = 4096;  // cells of the index over the pivots
constexpr int kPivotThreads = 512;
constexpr int kOneThreads = 1024;

// Bins of a sample of S records (a power of two; half of them between chosen
// pivots, about 512 to 1024 records each up to 2^21 records, half for the ends
// of repeated values), and the candidates the pivots are chosen from.
static int pivot_bins(int64_t S) {
    int b = 64;
    while (b < kPivotBinsMax / 2 && (int64_t)b * 1024 < S) b *= 2;
    return 2 * b;
}
static int pivot_candidates(int bins) { return std::min(bins * 2, (int)kOneSample / 2); }

// The sample sort's scratch (Layout::pivots): bin counts, starts, cursors and
// a ticket, the pivots, their index.
template <typename P> struct PivotScratch {
    uint32_t *count, *start, *cursor, *ticket;
    P *phi;
    uint32_t *tag;
    LutParams<P> *lutp;
    uint16_t *lut;
    __host__ __device__ static size_t bytes(int bins) {
        return (size_t)bins * 4 * 4 + 64 + (size_t)bins * sizeof(P) + 64 + (kPivotCells + 2) * 2;
    }
    PivotScratch() = default;
    __host__ __device__ PivotScratch(void *at, int bins) {
        unsigned char *b = (unsigned char *)at;
        phi = (P *)b;                 b += (size_t)bins * sizeof(P);
        lutp = (LutParams<P> *)b;     b += 64;
        count = (uint32_t *)b;        b += (size_t)bins * 4;
        cursor = (uint32_t *)b;       b += (size_t)bins * 4;
        ticket = (uint32_t *)b;       b += 16;
        start = (uint32_t *)b;        b += (size_t)(bins + 4) * 4;
        tag = (uint32_t *)b;          b += (size_t)bins * 4;
        lut = (uint16_t *)b;
    }
};

size_t sample_scratch_bytes(const Plan &p) {
    if (p.sample_size <= kOneSample) return 1;
    const int bins = pivot_bins(p.sample_size);
    return p.key_bytes == 8 ? PivotScratch<uint64_t>::bytes(bins) : PivotScratch<uint32_t>::bytes(bins);
}
int sample_sort_kernels(const Plan &p) { return p.sample_size == 0 ? 0 : p.sample_size <= kOneSample ? 1 : 4; }
int sample_final(const Plan &p) { return p.sample_size <= kOneSample ? 1 : 0; }

template <typename P> using OneSort = BlockSort<typename RecordSink<P>::K, kOneThreads>;
template <typename P> static size_t one_smem(int n) {
    return ((sizeof(typename OneSort<P>::Smem) + 15) & ~size_t(15)) + (size_t)n * sizeof(typename RecordSink<P>::K);
}
template <typename P> static size_t pivots_smem(int bins) { return one_smem<P>(pivot_candidates(bins)) + (size_t)bins * sizeof(P); }
static_assert(OneSort<uint32_t>::kMost >= kOneSample && OneSort<uint64_t>::kMost >= kOneSample, "records one CTA sorts");

template <typename P> struct SortArgs {
    RecordBuffers<P> b;
    int64_t S;
    int cand, bins;
    PivotScratch<P> sc;
};
template <typename P, bool MANY>
__global__ void __launch_bounds__(kOneThreads, 1) sample_one_kernel(const Many<SortArgs<P>> many) {
    const Pick<MANY, SortArgs<P>> pk(many);
    const P *phi = pk.a.b.phi[0];
    const uint32_t *tag = pk.a.b.tag[0];
    P *out_phi = pk.a.b.phi[1];
    uint32_t *out_tag = pk.a.b.tag[1];
    const int S = (int)pk.a.S;
    using K = typename RecordSink<P>::K;
    using Smem = typename OneSort<P>::Smem;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    K *a = reinterpret_cast<K *>(smem_raw + ((sizeof(Smem) + 15) & ~size_t(15)));
    for (int i = threadIdx.x; i < S; i += kOneThreads) a[i] = (K)phi[i] << 32 | tag[i];
    __syncthreads();
    OneSort<P>::run(*reinterpret_cast<Smem *>(smem_raw), a, S);
    for (int i = threadIdx.x; i < S; i += kOneThreads) {
        out_phi[i] = (P)(a[i] >> 32);
        out_tag[i] = (uint32_t)a[i];
    }
}

template <typename P, bool MANY>
__global__ void __launch_bounds__(kOneThreads, 1) sample_pivots_kernel(const Many<SortArgs<P>> many) {
    const Pick<MANY, SortArgs<P>> pk(many);
    const P *phi = pk.a.b.phi[0];
    const uint32_t *tag = pk.a.b.tag[0];
    const int64_t S = pk.a.S;
    const int cand = pk.a.cand, bins = pk.a.bins;
    const PivotScratch<P> &sc = pk.a.sc;
    using K = typename RecordSink<P>::K;
    using Smem = typename OneSort<P>::Smem;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    K *a = reinterpret_cast<K *>(smem_raw + ((sizeof(Smem) + 15) & ~size_t(15)));
    P *piv_phi = reinterpret_cast<P *>(a + cand);  // bins entries
    const uint32_t stretch = (uint32_t)(S / cand);
    for (int i = threadIdx.x; i < bins; i += kOneThreads) sc.count[i] = 0;
    if (threadIdx.x == 0) *sc.ticket = 0;
#pragma unroll
    for (int j = 0; j < (int)(kOneSample / kOneThreads); ++j) {
        const int i = j * kOneThreads + threadIdx.x;
        if (i < cand) {
            // a place in stretch i: the top bits of a multiplicative hash
            const int64_t r = (int64_t)i * stretch + __umulhi((uint32_t)i * 0x9e3779b1u, stretch);
            a[i] = (K)phi[r] << 32 | tag[r];
        }
    }
    __syncthreads();
    OneSort<P>::run(*reinterpret_cast<Smem *>(smem_raw), a, cand);
    // chosen pivot i: candidate of 1-indexed rank (i + 1) * step.  A value that
    // two neighbouring pivots share gets two more, before its first and past
    // its last record.
    const int chosen = bins / 2 - 1, step = cand / (bins / 2);
    auto phi_of = [&](int i) { return (P)(a[(i + 1) * step - 1] >> 32); };
    __shared__ uint32_t tmp[40];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int PER = kPivotBinsMax / 2 / kOneThreads;
    uint32_t extra[PER], loc = 0;  // 1: before, 2: after
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const int i = threadIdx.x * PER + j;
        extra[j] = 0;
        if (i < chosen) {
            const bool as_prev = i > 0 && phi_of(i - 1) == phi_of(i), as_next = i + 1 < chosen && phi_of(i + 1) == phi_of(i);
            if (as_next && !as_prev) extra[j] = 1;
            if (as_prev && !as_next && phi_of(i) != all_ones<P>()) extra[j] = 2;
            loc += 1 + (extra[j] != 0);
        }
    }
    uint32_t tot;
    const uint32_t ex = warp_excl_scan(loc, &tot);
    if (lane == 31) tmp[warp] = tot;
    __syncthreads();
    uint32_t at = ex, all = 0;
    for (int w = 0; w < kOneThreads / 32; ++w) {
        at += w < warp ? tmp[w] : 0u;
        all += tmp[w];
    }
    for (int i = (int)all + threadIdx.x; i < bins; i += kOneThreads) {  // the rest: past every record
        piv_phi[i] = all_ones<P>();
        sc.phi[i] = all_ones<P>();
        sc.tag[i] = 0xffffffffu;
    }
    auto put = [&](P f, uint32_t t) {
        piv_phi[at] = f;
        sc.phi[at] = f;
        sc.tag[at] = t;
        ++at;
    };
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const int i = threadIdx.x * PER + j;
        if (i < chosen) {
            if (extra[j] == 1) put(phi_of(i), 0u);
            put(phi_of(i), (uint32_t)a[(i + 1) * step - 1]);
            if (extra[j] == 2) put(phi_of(i) + 1, 0u);
        }
    }
    __syncthreads();
    // the index over the pivots, as over the splitters
    LutParams<P> lp;
    lp.base = piv_phi[0];
    lp.span = piv_phi[all - 1] - lp.base;  // (all >= 31 pivots)
    const int bl = bit_length<P>(lp.span);
    lp.shift = bl > 12 ? (uint32_t)(bl - 12) : 0u;
    lp.nsplit = all;
    static_assert(kPivotCells == 1 << 12, "cells of the index");
    if (threadIdx.x == 0) *sc.lutp = lp;
    for (int c = threadIdx.x; c <= kPivotCells; c += kOneThreads)
        sc.lut[c] = (uint16_t)lut_cell((uint32_t)c, lp, [&](uint32_t i) { return piv_phi[i]; });
}

// Records of a CTA's tiles per bin; the last CTA to finish turns the totals
// into the bins' starts.
template <typename P> constexpr size_t pivot_smem(int bins) {
    return 64 + (size_t)bins * (sizeof(P) + 4) + (kPivotCells + 8) * 2;  // (tags, read on ties, stay in global memory)
}
template <typename P> struct PivotSmem {
    LutParams<P> *lp;
    P *phi;
    uint32_t *cnt;
    uint16_t *lut;
    __device__ PivotSmem(unsigned char *b, int bins) {
        lp = (LutParams<P> *)b;   b += 64;
        phi = (P *)b;             b += (size_t)bins * sizeof(P);
        cnt = (uint32_t *)b;      b += (size_t)bins * 4;
        lut = (uint16_t *)b;
    }
    __device__ void load(const PivotScratch<P> &sc, int bins) {
        for (int i = threadIdx.x; i < bins; i += kPivotThreads) {
            phi[i] = sc.phi[i];
            cnt[i] = 0;
        }
        for (int i = threadIdx.x; i <= kPivotCells; i += kPivotThreads) lut[i] = sc.lut[i];
        if (threadIdx.x == 0) *lp = *sc.lutp;
        __syncthreads();
    }
};

template <typename P, bool MANY>
__global__ void __launch_bounds__(kPivotThreads) sample_hist_kernel(const Many<SortArgs<P>> many) {
    const Pick<MANY, SortArgs<P>> pk(many);
    const P *phi = pk.a.b.phi[0];
    const uint32_t *tag = pk.a.b.tag[0];
    const int64_t S = pk.a.S;
    const int bins = pk.a.bins;
    const PivotScratch<P> &sc = pk.a.sc;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    PivotSmem<P> sm(smem_raw, bins);
    __shared__ uint32_t tmp[40];
    __shared__ bool last;
    sm.load(sc, bins);
    const LutParams<P> lp = *sm.lp;
    const int64_t step = (int64_t)pk.blocks * kPivotThreads;
    for (int64_t r = (int64_t)pk.block * kPivotThreads + threadIdx.x; r < S; r += 4 * step) {
        P f[4];
        uint32_t t[4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (r + j * step < S) {
                f[j] = phi[r + j * step];
                t[j] = tag[r + j * step];
            }
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (r + j * step < S) atomicAdd(&sm.cnt[classify_key(f[j], t[j], lp, sm.lut, sm.phi, sc.tag)], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < bins; i += kPivotThreads)
        if (sm.cnt[i]) atomicAdd(&sc.count[i], sm.cnt[i]);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(sc.ticket, 1u) == pk.blocks - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    for (int i = threadIdx.x; i < bins; i += kPivotThreads) {
        sm.cnt[i] = ld_volatile(&sc.count[i]);
        sc.cursor[i] = 0;
    }
    __syncthreads();
    const uint32_t tot = block_excl_scan_smem<kPivotThreads>(sm.cnt, bins, tmp);
    for (int i = threadIdx.x; i < bins; i += kPivotThreads) sc.start[i] = sm.cnt[i];
    if (threadIdx.x == 0) sc.start[bins] = tot;
}

// Records of a tile, grouped by bin in shared memory, each bin's run written
// contiguously at its bin's start plus a reserved offset.
template <typename P, int ITEMS> constexpr size_t pivot_scatter_smem(int bins) {
    return pivot_smem<P>(bins) + (size_t)bins * 4 + (size_t)kPivotThreads * ITEMS * (sizeof(P) + 4 + 2) + 64;
}
template <typename P, int ITEMS, bool MANY>
__global__ void __launch_bounds__(kPivotThreads) sample_scatter_kernel(const Many<SortArgs<P>> many) {
    const Pick<MANY, SortArgs<P>> pk(many);
    const RecordBuffers<P> &b = pk.a.b;
    const int64_t S = pk.a.S;
    const int bins = pk.a.bins;
    const PivotScratch<P> &sc = pk.a.sc;
    constexpr int TILE = kPivotThreads * ITEMS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    PivotSmem<P> sm(smem_raw, bins);
    unsigned char *at8 = smem_raw + ((pivot_smem<P>(bins) + 15) & ~size_t(15));
    P *st_f = (P *)at8;
    uint32_t *st_t = (uint32_t *)(st_f + TILE), *dlt = st_t + TILE;
    uint16_t *st_b = (uint16_t *)(dlt + bins);
    __shared__ uint32_t tmp[40];
    sm.load(sc, bins);
    const LutParams<P> lp = *sm.lp;
    const int tid = threadIdx.x;
    for (int64_t t0 = (int64_t)pk.block * TILE; t0 < S; t0 += (int64_t)pk.blocks * TILE) {
        const int nh = (int)imin64(TILE, S - t0);
        P f[ITEMS];
        uint32_t t[ITEMS], br[ITEMS];
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            const int s = i * kPivotThreads + tid;
            if (s < nh) {
                f[i] = b.phi[0][t0 + s];
                t[i] = b.tag[0][t0 + s];
            }
        }
#pragma unroll
        for (int i = 0; i < ITEMS; ++i)
            if (i * kPivotThreads + tid < nh) {
                const uint32_t bin = classify_key(f[i], t[i], lp, sm.lut, sm.phi, sc.tag);
                br[i] = bin << 16 | atomicAdd(&sm.cnt[bin], 1u);
            }
        __syncthreads();
        for (int i = tid; i < bins; i += kPivotThreads) {
            const uint32_t c = sm.cnt[i];
            dlt[i] = c ? sc.start[i] + atomicAdd(&sc.cursor[i], c) : 0u;
        }
        __syncthreads();
        block_excl_scan_smem<kPivotThreads>(sm.cnt, bins, tmp);
        for (int i = tid; i < bins; i += kPivotThreads) dlt[i] -= sm.cnt[i];  // output slot of tile position s: dlt + s
#pragma unroll
        for (int i = 0; i < ITEMS; ++i)
            if (i * kPivotThreads + tid < nh) {
                const uint32_t bin = br[i] >> 16, pos = sm.cnt[bin] + (br[i] & 0xffffu);
                st_f[pos] = f[i];
                st_t[pos] = t[i];
                st_b[pos] = (uint16_t)bin;
            }
        __syncthreads();
        for (int s = tid; s < nh; s += kPivotThreads) {
            const uint32_t o = dlt[st_b[s]] + (uint32_t)s;
            b.phi[1][o] = st_f[s];
            b.tag[1][o] = st_t[s];
        }
        for (int i = tid; i < bins; i += kPivotThreads) sm.cnt[i] = 0;
        __syncthreads();
    }
}

// A bin's records in order by stable radix passes over the bytes in which they
// differ (none: a copy), from buffer 1 to buffer 0 and back, by T threads.
template <typename P, int T> struct RadixBin {
    static constexpr int ITEMS = 8, CH = T * ITEMS;
    using Rank = BlockRank<T, ITEMS, 8>;
    struct Smem {
        typename Rank::Smem rank;
        uint32_t run[256], tmp[40], any[3], all[3];  // any, all: of the tags and the halves of the phi
    };
    __device__ static void run(Smem &sm, const RecordBuffers<P> &b, int64_t at, int n) {
        const int tid = threadIdx.x;
        if (tid < 3) {
            sm.any[tid] = 0u;
            sm.all[tid] = 0xffffffffu;
        }
        __syncthreads();
        uint32_t any[3] = {}, all[3] = {~0u, ~0u, ~0u};
#pragma unroll 8
        for (int i = tid; i < n; i += T) {
            const P f = b.phi[1][at + i];
            const uint32_t w[3] = {b.tag[1][at + i], (uint32_t)f, (uint32_t)((uint64_t)f >> 32)};
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                any[k] |= w[k];
                all[k] &= w[k];
            }
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const uint32_t x = __reduce_or_sync(0xffffffffu, any[k]), y = __reduce_and_sync(0xffffffffu, all[k]);
            if ((tid & 31) == 0) {
                atomicOr(&sm.any[k], x);
                atomicAnd(&sm.all[k], y);
            }
        }
        __syncthreads();
        int cur = 1;
        for (int pass = 0; pass < 4 + (int)sizeof(P); ++pass) {
            const int shift = pass * 8 % 32;
            if (((sm.any[pass / 4] ^ sm.all[pass / 4]) >> shift & 255u) == 0) continue;
            const P *sf = b.phi[cur] + at;
            const uint32_t *st = b.tag[cur] + at;
            P *df = b.phi[1 - cur] + at;
            uint32_t *dt = b.tag[1 - cur] + at;
            auto digit = [&](P f, uint32_t t) {
                return (pass < 4 ? t >> shift : (uint32_t)(f >> (pass * 8 - 32))) & 255u;
            };
            for (int i = tid; i < 256; i += T) sm.run[i] = 0;
            __syncthreads();
#pragma unroll 4
            for (int i = tid; i < n; i += T) atomicAdd(&sm.run[pass < 4 ? digit(0, st[i]) : digit(sf[i], 0u)], 1u);
            __syncthreads();
            digit_excl_scan<T, 256>(sm.run, sm.tmp);
            for (int c = 0; c < n; c += CH) {
                P f[ITEMS];
                uint32_t t[ITEMS], d[ITEMS], rk[ITEMS];
#pragma unroll
                for (int i = 0; i < ITEMS; ++i) {
                    const int e = c + striped_slot<T, ITEMS>(i);
                    if (e < n) {
                        f[i] = sf[e];
                        t[i] = st[e];
                    }
                }
#pragma unroll
                for (int i = 0; i < ITEMS; ++i)  // past the end: after every record of digit 255
                    d[i] = c + striped_slot<T, ITEMS>(i) < n ? digit(f[i], t[i]) : 255u;
                Rank::rank(sm.rank, d, rk);
#pragma unroll
                for (int i = 0; i < ITEMS; ++i)
                    if (c + striped_slot<T, ITEMS>(i) < n) {
                        const uint32_t o = sm.run[d[i]] + rk[i];
                        df[o] = f[i];
                        dt[o] = t[i];
                    }
                __syncthreads();
                for (int i = tid; i < 256; i += T) sm.run[i] += sm.rank.digit_tot[i];
                __syncthreads();
            }
            cur = 1 - cur;
        }
        if (cur == 1) {
#pragma unroll 8
            for (int i = tid; i < n; i += T) {
                b.phi[0][at + i] = b.phi[1][at + i];
                b.tag[0][at + i] = b.tag[1][at + i];
            }
        }
    }
};

// Bins too large for the counting sort (radix_bins), one per CTA.
constexpr int kRadixThreads = 512;
template <typename P, bool MANY>
__global__ void __launch_bounds__(kRadixThreads, 2) sample_radix_kernel(const Many<SortArgs<P>> many) {
    const Pick<MANY, SortArgs<P>> pk(many);
    __shared__ typename RadixBin<P, kRadixThreads>::Smem sm;
    const uint32_t at = pk.a.sc.start[pk.block];
    const int n = (int)(pk.a.sc.start[pk.block + 1] - at);
    if (n > 0) RadixBin<P, kRadixThreads>::run(sm, pk.a.b, at, n);
}

// One bin per CTA, from buffer 1 into its place in buffer 0.  A bin of one
// record (a sample of many more draws than keys) is copied; what the counting
// sort gives back is sorted by radix passes.
template <typename P, int SIZE, bool MANY>
__global__ void __launch_bounds__(CountShape<SIZE>::T, CountShape<SIZE>::kPerSm)
sample_bins_kernel(const Many<SortArgs<P>> many) {
    const Pick<MANY, SortArgs<P>> pk(many);
    const RecordBuffers<P> &b = pk.a.b;
    const PivotScratch<P> &sc = pk.a.sc;
    using K = typename RecordSink<P>::K;
    using CS = typename CountShape<SIZE>::template Sort<K>;
    constexpr int T = CountShape<SIZE>::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const uint32_t at = sc.start[pk.block];
    const int n = (int)(sc.start[pk.block + 1] - at);
    if (n == 0) return;
    const RecordSource<P, T> src{b.phi[1] + at, b.tag[1] + at};
    K lo, hi;
    CS::bounds(smem_raw, src, n, lo, hi);
    if (lo != hi && CS::run(smem_raw, src, n, lo, hi, RecordSink<P>{b.phi[0], b.tag[0], (int64_t)at}, 0, 1)) return;
    __syncthreads();
    using Radix = RadixBin<P, T>;
    static_assert(sizeof(typename Radix::Smem) <= CS::smem_bytes(), "in the counting sort's place");
    Radix::run(*reinterpret_cast<typename Radix::Smem *>(smem_raw), b, at, n);
}

static int sm_count() {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return std::max(sms, 1);
}

template <typename K> static RecordBuffers<K> buffers_of(const Ctx &c) {
    RecordBuffers<K> b;
    b.phi[0] = (K *)c.ly.sphi[0];
    b.phi[1] = (K *)c.ly.sphi[1];
    b.tag[0] = c.ly.stag[0];
    b.tag[1] = c.ly.stag[1];
    return b;
}

template <typename K> static void sort_args(const Ctx &c, SortArgs<K> &a) {
    a.b = buffers_of<K>(c);
    a.S = c.pl.sample_size;
    a.bins = pivot_bins(a.S);
    a.cand = pivot_candidates(a.bins);
    a.sc = PivotScratch<K>(c.ly.pivots, a.bins);
}

// The shape that sorts a bin (its mean is 2 S / bins records; the stages hold
// 3832, 8696 and 18,680 of them, and two CTAs of 512 threads on an SM beat one of
// 1024 while a bin fits: 8.4M records 344 us and 383), and the tiles of the scatter: 2K records until there are enough
// of 4K to fill the GPU.
static int bins_shape(int64_t S, int key_bytes) {
    if (key_bytes == 8) return kCountRecord;
    const int64_t half = S / pivot_bins(S);
    return half <= 700 ? kCountSmall : half <= 3000 ? kCountMedium : kCountLarge;
}
// Bins past this mean take radix passes: the counting sort reads a bin again for
// every part of it (a stage holds 5112 records of doubles, 18,680 of 4-byte keys).
static bool radix_bins(int64_t S, int key_bytes) {
    return 2 * S / pivot_bins(S) > (key_bytes == 8 ? 12288 : 65536);
}
static int scatter_items(int64_t S) { return S < (1 << 20) ? 4 : 8; }

template <typename K, int SIZE> static cudaError_t launch_sample_bins(Exec &x) {
    using CS = typename CountShape<SIZE>::template Sort<typename RecordSink<K>::K>;
    return launch_calls<SortArgs<K>>(x, sample_bins_kernel<K, SIZE, false>, sample_bins_kernel<K, SIZE, true>,
                                     CountShape<SIZE>::T, CS::smem_bytes(), [](const Ctx &c, SortArgs<K> &a) {
        if (c.pl.sample_size <= kOneSample || bins_shape(c.pl.sample_size, sizeof(K)) != SIZE ||
            radix_bins(c.pl.sample_size, sizeof(K)))
            return 0u;
        sort_args(c, a);
        return (uint32_t)a.bins;
    });
}

template <typename K, int ITEMS> static cudaError_t launch_sample_scatter(Exec &x, int bins) {
    const int64_t wave = 2 * sm_count();
    const DynSmem smem(pivot_scatter_smem<K, ITEMS>(bins), pivot_scatter_smem<K, ITEMS>(kPivotBinsMax));
    return launch_calls<SortArgs<K>>(x, sample_scatter_kernel<K, ITEMS, false>, sample_scatter_kernel<K, ITEMS, true>,
                                     kPivotThreads, smem, [=](const Ctx &c, SortArgs<K> &a) {
        const int64_t S = c.pl.sample_size, tile = (int64_t)kPivotThreads * ITEMS;
        if (S <= kOneSample || scatter_items(S) != ITEMS) return 0u;
        sort_args(c, a);
        return (uint32_t)imin64((S + tile - 1) / tile, wave);
    });
}

template <typename K> static cudaError_t launch_sample_sort_t(Exec &x) {
    // shared memory: for the largest sample among the calls
    int64_t one = 0, most = 0;
    for (int i = 0; i < x.count; ++i) {
        const int64_t S = x.calls[i].pl.sample_size;
        if (S <= kOneSample) one = imax64(one, S);
        else most = imax64(most, S);
    }
    cudaError_t e = cudaSuccess;
    if (one > 0)
        e = launch_calls<SortArgs<K>>(x, sample_one_kernel<K, false>, sample_one_kernel<K, true>, kOneThreads,
                                      DynSmem(one_smem<K>((int)one), one_smem<K>((int)kOneSample)), [](const Ctx &c, SortArgs<K> &a) {
            if (c.pl.sample_size == 0 || c.pl.sample_size > kOneSample) return 0u;
            a.b = buffers_of<K>(c);
            a.S = c.pl.sample_size;
            return 1u;
        });
    if (e != cudaSuccess || most == 0) return e;
    const int bins = pivot_bins(most);
    e = launch_calls<SortArgs<K>>(x, sample_pivots_kernel<K, false>, sample_pivots_kernel<K, true>, kOneThreads,
                                  DynSmem(pivots_smem<K>(bins), pivots_smem<K>(kPivotBinsMax)),
                                  [](const Ctx &c, SortArgs<K> &a) {
        if (c.pl.sample_size <= kOneSample) return 0u;
        sort_args(c, a);
        return 1u;
    });
    if (e != cudaSuccess) return e;
    const int64_t wave = 2 * sm_count();
    e = launch_calls<SortArgs<K>>(x, sample_hist_kernel<K, false>, sample_hist_kernel<K, true>, kPivotThreads,
                                  DynSmem(pivot_smem<K>(bins), pivot_smem<K>(kPivotBinsMax)), [=](const Ctx &c, SortArgs<K> &a) {
        if (c.pl.sample_size <= kOneSample) return 0u;
        sort_args(c, a);
        return (uint32_t)imin64(wave, (a.S + 4 * kPivotThreads - 1) / (4 * kPivotThreads));
    });
    if (e == cudaSuccess) e = launch_sample_scatter<K, 4>(x, bins);
    if (e == cudaSuccess) e = launch_sample_scatter<K, 8>(x, bins);
    if (e == cudaSuccess)
        e = launch_calls<SortArgs<K>>(x, sample_radix_kernel<K, false>, sample_radix_kernel<K, true>, kRadixThreads, 0,
                                      [](const Ctx &c, SortArgs<K> &a) {
            if (c.pl.sample_size <= kOneSample || !radix_bins(c.pl.sample_size, sizeof(K))) return 0u;
            sort_args(c, a);
            return (uint32_t)a.bins;
        });
    if (e != cudaSuccess) return e;
    if constexpr (sizeof(K) == 8) {
        return launch_sample_bins<K, kCountRecord>(x);
    } else {
        e = launch_sample_bins<K, kCountSmall>(x);
        if (e == cudaSuccess) e = launch_sample_bins<K, kCountMedium>(x);
        if (e == cudaSuccess) e = launch_sample_bins<K, kCountLarge>(x);
        return e;
    }
}

cudaError_t launch_sample_sort(Exec &x) {
    return x.calls[0].pl.key_bytes == 8 ? launch_sample_sort_t<uint64_t>(x) : launch_sample_sort_t<uint32_t>(x);
}

} // namespace bsps
