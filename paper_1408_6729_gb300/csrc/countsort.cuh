// countsort.cuh -- keys-only sort of one segment by one CTA (or by several that
// share its output): the bucket sort of Fig. 2 step 12 and the block sort of
// Fig. 1 step 3 where no payload moves.  Equal keys cannot be told apart, so no
// rank needs to be stable.
//
// The segment's keys lie in [lo, hi].  It stays in global memory (L2 after the
// first pass) and is streamed, so its size is not bounded by shared memory:
//   1. every key is counted in one of up to NBMAX bins, (key - lo) >> shift,
//      with one shared-memory reduction (bins b and b + nb/2 are the halves of
//      one word);
//   2. a scan turns the counts into the bins' first positions.  The positions
//      are cut into parts that the stage holds, at multiples of 256 bins;
//   3. per part, the keys are read again and each key of the part is stored at
//      its bin's next position of a shared-memory stage (one atomic);
//   4. the stage is now sorted up to the order inside each bin.  A bin of at
//      most kEdge keys is finished in registers: a warp takes 256 consecutive
//      positions, eight to a lane, sorts them by a network inside the lanes and
//      across their borders (odd-even transposition rounds where a bin needs
//      more) and writes the middle 224 with 16-byte stores; every bin touching
//      those lies inside the 256.  Longer bins (skewed or repeated keys) are
//      listed by the scan (or, past the list's room, found again by their
//      cursors) and sorted in the stage first: not at all when all
//      their keys are equal, else by a warp or, above kWarpBin keys, by the CTA.
// Per key that is two shared-memory atomics and one shared store, and no
// exchange between CTAs.
//
// A narrow stage holds only the low half of key - lo (16 bits of 32, 32 of 64),
// so twice the keys: a 65,536-key bucket of 32-bit keys is one part, read twice
// instead of three times.  The rest follows from the position: key - lo is cut
// into units of 2^(half - 1) values, every unit is a range of bins, and the
// scan records the position where it starts.  A window of at most two units is
// put in order and rebuilt from the half words alone.  It is taken when the
// units are few and long (ranges up to 2^23 values at 65,536 keys).
//
// Where 256 bins hold more than half of what the stage takes (keys that crowd
// in a small part of the range: a narrow component of a mixture, floats around
// zero, a value with thousands of copies), they are sorted by themselves
// afterwards, from the keys of the segment that lie in their range, with bins
// as fine as that needs; a run of one-value bins that is larger than the stage
// is written from its counts.
//
// Several CTAs (G of them) may take one segment: each counts all of it and
// takes every G-th part.  Every decision is a function of the segment alone,
// so the CTAs agree without talking to each other.
//
// Bound by instruction issue (about 93 warp instructions per 32 keys, the
// integer ones at half rate) and by the latency of the phases.  2^28 uniform
// int32 keys in 65,536-key sub-buckets: 1.26 ms (1.70 TB/s of keys read and
// written); the cluster split, exchange and count it replaced took 2.38.  With
// a wide stage in two parts 1.26 against 1.22, with edge checks in every window
// 1.23.  2^28 skewed doubles in 4096 sub-buckets: 2.6 ms, before the crowded
// ranges were sorted here 3.8 and 0.84 for one bucket out of core.
#pragma once

#include <type_traits>

#include "radix.cuh"

namespace bsps {

// A wide record: 64-bit phi and 32-bit tag in one comparable word.
using u128 = unsigned __int128;

template <typename K> __device__ __forceinline__ K shfl_up_one(K v) {
    if constexpr (sizeof(K) == 16) {
        const uint64_t a = __shfl_up_sync(0xffffffffu, (uint64_t)(v >> 64), 1), b = __shfl_up_sync(0xffffffffu, (uint64_t)v, 1);
        return (u128)a << 64 | b;
    } else {
        return __shfl_up_sync(0xffffffffu, v, 1);
    }
}
template <typename K> __device__ __forceinline__ K shfl_down_one(K v) {
    if constexpr (sizeof(K) == 16) {
        const uint64_t a = __shfl_down_sync(0xffffffffu, (uint64_t)(v >> 64), 1), b = __shfl_down_sync(0xffffffffu, (uint64_t)v, 1);
        return (u128)a << 64 | b;
    } else {
        return __shfl_down_sync(0xffffffffu, v, 1);
    }
}
template <typename K> __device__ __forceinline__ K shfl_xor_any(K v, int o) {
    if constexpr (sizeof(K) == 16) {
        const uint64_t a = __shfl_xor_sync(0xffffffffu, (uint64_t)(v >> 64), o), b = __shfl_xor_sync(0xffffffffu, (uint64_t)v, o);
        return (u128)a << 64 | b;
    } else {
        return __shfl_xor_sync(0xffffffffu, v, o);
    }
}
template <typename K> __device__ __forceinline__ K shfl_any(K v, int lane) {
    if constexpr (sizeof(K) == 16) {
        const uint64_t a = __shfl_sync(0xffffffffu, (uint64_t)(v >> 64), lane), b = __shfl_sync(0xffffffffu, (uint64_t)v, lane);
        return (u128)a << 64 | b;
    } else {
        return __shfl_sync(0xffffffffu, v, lane);
    }
}
template <typename K> __device__ __forceinline__ int word_bits(K v) {
    if constexpr (sizeof(K) == 16) return (v >> 64) ? 64 + bit_length<uint64_t>((uint64_t)(v >> 64)) : bit_length<uint64_t>((uint64_t)v);
    else return bit_length<K>(v);
}

// Ascending bitonic network over a[0..len), whose runs of h0 keys are sorted,
// by `size` threads, this one being `rank`; every comparator puts the larger
// key higher, so positions past len act as keys above all others and are never
// touched.
template <typename E, typename Sync>
__device__ void bitonic(E *a, int len, int rank, int size, Sync sync, int h0 = 1) {
    int n2 = 1;
    while (n2 < len) n2 <<= 1;
    auto step = [&](int i, int l) {
        if (l < len) {
            const E x = a[i], y = a[l];
            if (x > y) {
                a[i] = y;
                a[l] = x;
            }
        }
    };
    for (int h = h0; h < n2; h <<= 1) {  // runs of h sorted: merge pairs of them
        for (int t = rank; t < (n2 >> 1); t += size) {
            const int b = (t & ~(h - 1)) * 2, o = t & (h - 1);
            step(b + o, b + 2 * h - 1 - o);
        }
        sync();
        for (int j = h >> 1; j > 0; j >>= 1) {
            for (int t = rank; t < (n2 >> 1); t += size) {
                const int i = 2 * t - (t & (j - 1));
                step(i, i + j);
            }
            sync();
        }
    }
}

// One warp's sort of a[0..len), len <= 32 * R, in registers: R runs of 32, one
// key to a lane, then pairs of runs merged (a merge's first step pairs mirrored
// places).
template <typename E, int R> __device__ __forceinline__ void warp_sort_regs(E *a, uint32_t len) {
    const uint32_t lane = threadIdx.x & 31;
    E x[R];
#pragma unroll
    for (int r = 0; r < R; ++r) x[r] = r * 32 + lane < len ? a[r * 32 + lane] : all_ones<E>();
    auto lanes = [&](E &v, int o, int bit) {  // v against the key o lanes away, the lower lane taking the smaller
        const E y = shfl_xor_any(v, o);
        v = (lane & bit) == 0 ? (y < v ? y : v) : (y > v ? y : v);
    };
#pragma unroll
    for (int h = 1; h < 32; h <<= 1) {
        if (R == 1 && (uint32_t)h >= len) break;
#pragma unroll
        for (int j = h; j > 0; j >>= 1)
#pragma unroll
            for (int r = 0; r < R; ++r) lanes(x[r], j == h ? 2 * h - 1 : j, j);
    }
#pragma unroll
    for (int h = 1; h < R; h <<= 1) {
#pragma unroll
        for (int g = 0; g < R; g += 2 * h)
#pragma unroll
            for (int q = 0; q < h; ++q) {
                E &u = x[g + q], &v = x[g + 2 * h - 1 - q];
                const E uu = shfl_xor_any(u, 31), vv = shfl_xor_any(v, 31);
                u = vv < u ? vv : u;
                v = uu > v ? uu : v;
            }
#pragma unroll
        for (int j = h >> 1; j > 0; j >>= 1)
#pragma unroll
            for (int r = 0; r < R; ++r)
                if ((r & j) == 0) {
                    const E u = x[r], v = x[r + j];
                    x[r] = u < v ? u : v;
                    x[r + j] = u < v ? v : u;
                }
#pragma unroll
        for (int j = 16; j > 0; j >>= 1)
#pragma unroll
            for (int r = 0; r < R; ++r) lanes(x[r], j, j);
    }
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (r * 32 + lane < len) a[r * 32 + lane] = x[r];
}
// ... of more than 32 keys: runs of 256 in registers, those merged where they
// lie (128-bit words, which would fill the registers, all where they lie).
template <typename E> __device__ __noinline__ void warp_sort_more(E *a, uint32_t len) {
    const int lane = (int)(threadIdx.x & 31);
    if constexpr (sizeof(E) <= 8) {
        if (len <= 64) {
            warp_sort_regs<E, 2>(a, len);
        } else if (len <= 128) {
            warp_sort_regs<E, 4>(a, len);
        } else {
            for (uint32_t r = 0; r < len; r += 256) warp_sort_regs<E, 8>(a + r, len - r < 256 ? len - r : 256);
            __syncwarp();
            if (len > 256) bitonic(a, (int)len, lane, 32, [] { __syncwarp(); }, 256);
        }
    } else {
        bitonic(a, (int)len, lane, 32, [] { __syncwarp(); });
    }
}
// One warp's sort of a[0..len): nothing when all keys are equal.
template <typename E> __device__ __forceinline__ void warp_sort(E *a, uint32_t len) {
    const uint32_t lane = threadIdx.x & 31;
    bool differ = false;
    const E first = a[0];
    for (uint32_t e = lane; e < len; e += 32) differ |= a[e] != first;
    if (!__any_sync(0xffffffffu, differ)) return;
    if (len <= 32) warp_sort_regs<E, 1>(a, len);
    else warp_sort_more(a, len);
}

// The key that more than half of 32 spread over a[0..len) are equal to, if three
// tries find it (every warp that asks finds the same).
template <typename E> __device__ __forceinline__ bool common_key(const E *a, uint32_t len, E &v) {
    const E s = a[(threadIdx.x & 31) * len / 32];
    for (int i = 0; i < 3; ++i) {
        const uint32_t m = __ballot_sync(0xffffffffu, s == a[(i * 13 + 3) * len / 32]);
        v = a[(i * 13 + 3) * len / 32];
        if (__popc(m) > 16) return true;
    }
    return false;
}

// One warp's sort of a[0..len) where at most 32 keys differ from one that most
// are equal to (a value with many copies, and what shares its bin): they are
// taken out, put in order, and written to the ends.  False, and nothing
// changed, elsewhere.
template <typename E> __device__ __noinline__ bool warp_sort_mostly_one(E *a, uint32_t len) {
    const uint32_t lane = threadIdx.x & 31;
    E v, other = all_ones<E>();
    if (!common_key(a, len, v)) return false;
    uint32_t n = 0, at = 0;  // lane i < n holds the i-th other key and its place
    for (uint32_t e0 = 0; e0 < len; e0 += 128) {
        E x[4];
        bool d[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t e = e0 + j * 32 + lane;
            x[j] = e < len ? a[e] : v;
            d[j] = x[j] != v;
        }
        if (!__any_sync(0xffffffffu, d[0] | d[1] | d[2] | d[3])) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j)
            for (uint32_t m = __ballot_sync(0xffffffffu, d[j]); m; m &= m - 1) {
                const int l = __ffs(m) - 1;
                const E y = shfl_any(x[j], l);
                if (n == 32) return false;
                if (lane == n) {
                    other = y;
                    at = e0 + j * 32 + l;
                }
                ++n;
            }
    }
    if (lane < n) a[at] = v;
    __syncwarp();
#pragma unroll
    for (int h = 1; h < 32; h <<= 1) {
        if ((uint32_t)h >= n) break;
#pragma unroll
        for (int j = h; j > 0; j >>= 1) {
            const E y = shfl_xor_any(other, j == h ? 2 * h - 1 : j);
            other = (lane & j) == 0 ? (y < other ? y : other) : (y > other ? y : other);
        }
    }
    const uint32_t below = (uint32_t)__popc(__ballot_sync(0xffffffffu, lane < n && other < v));
    if (lane < n) a[lane < below ? lane : len - n + lane] = other;
    __syncwarp();
    return true;
}

// A whole CTA's sort of a[0..n) in shared memory, in time that hardly depends on
// the keys: M of them, one drawn from each of M stretches, are put in order one
// to a thread (shuffles up to 32 apart), every key finds its place among them --
// equal to one, which needs no more order, or between two -- and a warp
// finishes each gap.  (A bin of 5000 copies of a value and a few other keys:
// 2^22 keys, nine in ten of them copies, 1.56 ms when the gap above a pivot held
// the pivot's copies, too, and 0.41 by the cluster sort.)
template <typename E, int T> struct BlockSort {
    static constexpr int M = T < 512 ? T : 512, ITEMS = T == 1024 ? 8 : 16, kMost = T * ITEMS;
    struct Smem {
        E piv[M];
        uint32_t cnt[M + 4];
        uint32_t tmp[40];
    };
    // the keys of threads < m (a power of two, at most M) in ascending order at
    // piv[0..m); what the threads past them hold ends past those
    __device__ static void sort_pivots(E *piv, E x, int m = M) {
        const int t = threadIdx.x;
        for (int h = 1; h < m; h <<= 1) {
            for (int j = h; j > 0; j >>= 1) {
                // the first step of a merge pairs mirrored positions
                const int o = j == h ? 2 * h - 1 : j;
                E y;
                if (o < 32) {
                    y = shfl_xor_any(x, o);
                } else {
                    if (t < M) piv[t] = x;
                    __syncthreads();
                    y = t < M ? piv[t ^ o] : x;
                    __syncthreads();
                }
                const bool low = (t & (j == h ? h : j)) == 0;
                x = low ? (y < x ? y : x) : (y > x ? y : x);
            }
        }
        if (t < M) piv[t] = x;
        __syncthreads();
    }

    // As warp_sort_mostly_one, by the CTA, with at most M other keys.
    __device__ __noinline__ static bool mostly_one(Smem &sm, E *a, int n) {
        const int t = threadIdx.x;
        E v;
        if (!common_key(a, (uint32_t)n, v)) return false;  // (every warp alike)
        if (t == 0) sm.cnt[M] = 0;
        __syncthreads();
        for (int e = t; e < n; e += T)
            if (a[e] != v) {
                const uint32_t k = atomicAdd(&sm.cnt[M], 1u);
                if (k < (uint32_t)M) {
                    sm.piv[k] = a[e];
                    sm.cnt[k] = (uint32_t)e;
                }
            }
        __syncthreads();
        const int c = (int)min(sm.cnt[M], (uint32_t)M + 1);
        const E x = t < min(c, M) ? sm.piv[t] : all_ones<E>();
        const uint32_t at = t < min(c, M) ? sm.cnt[t] : 0u;
        __syncthreads();
        if (c > M) return false;
        if (c == 0) return true;
        if (t < c) a[at] = v;
        sort_pivots(sm.piv, x);
        const int below = __syncthreads_count(t < c && sm.piv[t] < v);
        if (t < c) a[t < below ? t : n - c + t] = sm.piv[t];
        __syncthreads();
        return true;
    }

    __device__ __noinline__ static void run(Smem &sm, E *a, int n) {
        const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
        if (n <= M) {
            sort_pivots(sm.piv, t < n ? a[t] : all_ones<E>());
            if (t < n) a[t] = sm.piv[t];
            __syncthreads();
            return;
        }
        if (n > kMost) {
            bitonic(a, n, t, T, [] { __syncthreads(); });
            return;
        }
        const uint32_t stretch = (uint32_t)n / M;
        E x = all_ones<E>();
        if (t < M) x = a[(uint32_t)t * stretch + __umulhi((uint32_t)t * 0x9e3779b1u, stretch)];
        for (int i = t; i < M + 4; i += T) sm.cnt[i] = 0;
        sort_pivots(sm.piv, x);
        // bin b, the keys with b pivots (of the first M - 1) at or below them:
        // copies of the last of those (count in the low half), then the others
        E k[ITEMS];
        uint32_t br[ITEMS];  // bin << 16 | copy << 15 | place among its kind
        static_assert(kMost <= 0x7fff + 1, "places of 15 bits");
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            if (i * T >= n) break;  // (the code of the rest is not even fetched: few keys, one CTA)
            const int e = i * T + t;
            if (e < n) {
                k[i] = a[e];
                uint32_t b = 0;
#pragma unroll
                for (int w = M / 2; w > 0; w >>= 1)
                    if (!(k[i] < sm.piv[b + w - 1])) b += w;
                const bool copy = b > 0 && !(sm.piv[b - 1] < k[i]);
                const uint32_t old = atomicAdd(&sm.cnt[b], copy ? 1u : 0x10000u);
                br[i] = b << 16 | (copy ? 0x8000u | (old & 0xffffu) : old >> 16);
            }
        }
        __syncthreads();
        // each bin's first place and its copies
        const uint32_t c = t < M ? sm.cnt[t] : 0u;
        uint32_t tot;
        uint32_t first = warp_excl_scan((c & 0xffffu) + (c >> 16), &tot);
        if (lane == 31) sm.tmp[warp] = tot;
        __syncthreads();
        uint32_t all;
        const uint32_t before = warp_excl_scan(lane < T / 32 ? sm.tmp[lane] : 0u, &all);
        first += __shfl_sync(0xffffffffu, before, warp);
        if (t < M) sm.cnt[t] = first | c << 16;
        if (t == 0) sm.cnt[M] = (uint32_t)n;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            if (i * T >= n) break;
            if (i * T + t < n) {
                const uint32_t w = sm.cnt[br[i] >> 16];
                a[(w & 0xffffu) + ((br[i] & 0x8000u) ? 0u : w >> 16) + (br[i] & 0x7fffu)] = k[i];
            }
        }
        __syncthreads();
        // the gaps: two keys by one thread, more by a warp
        if (t < M) {
            const uint32_t at = (sm.cnt[t] & 0xffffu) + (sm.cnt[t] >> 16), end = sm.cnt[t + 1] & 0xffffu;
            if (end - at == 2) {
                const E u = a[at], v = a[at + 1];
                if (v < u) {
                    a[at] = v;
                    a[at + 1] = u;
                }
            }
        }
        for (int b = warp; b < M; b += T / 32) {
            const uint32_t at = (sm.cnt[b] & 0xffffu) + (sm.cnt[b] >> 16), len = (sm.cnt[b + 1] & 0xffffu) - at;
            if (len <= 2) continue;
            if (len <= 32) warp_sort_regs<E, 1>(a + at, len);
            else warp_sort_more(a + at, len);
        }
        __syncthreads();
    }
};

// Where a segment's keys come from: each(n, f) calls f(key) for all n of them,
// shared out over the T threads of a CTA.
template <typename K, int T, typename Xf> struct KeySource {
    const K *__restrict__ src;
    Xf xf;  // a loaded word to the key sorted
    template <typename F> __device__ void each(int n, F f) const {
        constexpr int V = 16 / (int)sizeof(K);
        const int tid = threadIdx.x;
        if (((uintptr_t)src & 15) == 0) {
            const uint4 *s4 = reinterpret_cast<const uint4 *>(src);
            const int nq = n / V;
            auto take = [&](const uint4 &w) {
                if constexpr (sizeof(K) == 4) {
                    f(xf(w.x)); f(xf(w.y)); f(xf(w.z)); f(xf(w.w));
                } else {
                    f(xf((uint64_t)w.y << 32 | w.x)); f(xf((uint64_t)w.w << 32 | w.z));
                }
            };
            int q = tid;
            for (; q + 3 * T < nq; q += 4 * T) {
                uint4 w[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) w[j] = s4[q + j * T];
#pragma unroll
                for (int j = 0; j < 4; ++j) take(w[j]);
            }
            for (; q < nq; q += T) take(s4[q]);
            const int e = nq * V + tid;
            if (e < n) f(xf(src[e]));
        } else {
            int e = tid;
            for (; e + 3 * T < n; e += 4 * T) {
                K w[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) w[j] = src[e + j * T];
#pragma unroll
                for (int j = 0; j < 4; ++j) f(xf(w[j]));
            }
            for (; e < n; e += T) f(xf(src[e]));
        }
    }
};

// Records (phi, tag) of two arrays as single words.
template <typename P, int T> struct RecordSource {
    using K = typename std::conditional<sizeof(P) == 8, u128, uint64_t>::type;
    const P *__restrict__ phi;
    const uint32_t *__restrict__ tag;
    template <typename F> __device__ void each(int n, F f) const {
        int e = threadIdx.x;
        for (; e + 3 * T < n; e += 4 * T) {
            P a[4];
            uint32_t b[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                a[j] = phi[e + j * T];
                b[j] = tag[e + j * T];
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) f((K)a[j] << 32 | b[j]);
        }
        for (; e < n; e += T) f((K)phi[e] << 32 | tag[e]);
    }
};

// Where the sorted keys go: pad(p) is position p's offset from 16-byte
// alignment, eight() stores the keys of eight positions from an aligned one.
template <typename K, typename Inv> struct KeySink {
    K *out;
    Inv inv;  // a sorted key to the word stored
    static constexpr int V = 16 / (int)sizeof(K);
    // 8-byte keys are emitted in a function of its own: inlined into the sort
    // it spills there (2^26 uniform doubles in 4096 sub-buckets 766 us, 738)
    static constexpr bool kApart = sizeof(K) == 8;
    __device__ int pad(uint32_t p) const { return (int)(((uintptr_t)(out + p) / sizeof(K)) & (V - 1)); }
    __device__ void one(int64_t p, K k) const { out[p] = inv(k); }
    template <typename Key> __device__ void eight(int64_t p, Key key) const {
#pragma unroll
        for (int j = 0; j < 8 / V; ++j) {
            uint4 w;
            if constexpr (sizeof(K) == 4) {
                w = make_uint4(inv(key(j * 4)), inv(key(j * 4 + 1)), inv(key(j * 4 + 2)), inv(key(j * 4 + 3)));
            } else {
                const uint64_t a = inv(key(j * 2)), b = inv(key(j * 2 + 1));
                w = make_uint4((uint32_t)a, (uint32_t)(a >> 32), (uint32_t)b, (uint32_t)(b >> 32));
            }
            *reinterpret_cast<uint4 *>(out + p + j * V) = w;
        }
    }
};

// Records back into two arrays (16-byte aligned).
template <typename P> struct RecordSink {
    using K = typename std::conditional<sizeof(P) == 8, u128, uint64_t>::type;
    P *phi;
    uint32_t *tag;
    int64_t at;  // array index of position 0
    static constexpr bool kApart = false;
    __device__ int pad(uint32_t p) const { return (int)((at + p) & 3); }
    __device__ void one(int64_t p, K k) const {
        phi[at + p] = (P)(k >> 32);
        tag[at + p] = (uint32_t)k;
    }
    template <typename Key> __device__ void eight(int64_t p, Key key) const {
#pragma unroll
        for (int j = 0; j < 8; j += 4) {
            const K a = key(j), b = key(j + 1), c = key(j + 2), d = key(j + 3);
            if constexpr (sizeof(P) == 4) {
                *reinterpret_cast<uint4 *>(phi + at + p + j) =
                    make_uint4((uint32_t)(a >> 32), (uint32_t)(b >> 32), (uint32_t)(c >> 32), (uint32_t)(d >> 32));
            } else {
                phi[at + p + j] = (P)(a >> 32);
                phi[at + p + j + 1] = (P)(b >> 32);
                phi[at + p + j + 2] = (P)(c >> 32);
                phi[at + p + j + 3] = (P)(d >> 32);
            }
            *reinterpret_cast<uint4 *>(tag + at + p + j) = make_uint4((uint32_t)a, (uint32_t)b, (uint32_t)c, (uint32_t)d);
        }
    }
};

template <typename K, int T, int NBMAX, int STAGE> struct CountSort {
    using S = typename std::conditional<sizeof(K) >= 8, uint32_t, uint16_t>::type;  // word of a narrow stage
    static constexpr int UB = sizeof(K) >= 8 ? 31 : 15;  // bits of a unit
    static constexpr int W = T / 32;
    static constexpr int V = 16 / (int)sizeof(K);    // keys per 16-byte access
    static constexpr int kSegBins = 256;             // bins per scan step of a warp
    static constexpr int kSegs = NBMAX / kSegBins;
    static constexpr int kWin = 256, kEdge = 16, kStep = kWin - 2 * kEdge;
    static constexpr int kPer = kWin / 32;           // keys of a window per lane
    static constexpr int kLongMax = NBMAX / 16;      // listed long bins
    static constexpr int kWarpBin = 256;             // long bins up to this size are sorted by one warp,
    static constexpr int kWarpMany = T < 1024 ? kWarpBin : 1024;  // up to this where there are many, and nearly
    static constexpr int kWarpMost = 8192;           // one value up to this
    static constexpr int kPartsMax = 32;
    static constexpr int kUnits = 256;               // units of a narrow stage
    static constexpr int kTodo = 16;                 // crowded ranges waiting
    static constexpr uint32_t kUseWide = STAGE / sizeof(K) - 8, kUseNarrow = STAGE / sizeof(S) - 8;
    static_assert(NBMAX % 512 == 0 && kSegs <= 128 && NBMAX <= 65536, "the segments are scanned by one warp, four to a lane");
    static_assert(kUseNarrow / (kWarpBin + 1) < kLongMax, "a part's bins for the CTA fit the list");
    static_assert(kUseWide < 65528 && STAGE % 16 == 0, "16-bit positions inside a part");

    struct Smem {
        uint32_t seg[kSegs + 1];              // first position of every segment of 256 bins
        uint32_t pseg[kPartsMax + 1];         // first segment of every part
        uint32_t unit[kUnits + 2];            // first position of every unit (narrow stage)
        uint32_t longs[kLongMax];             // bin | length << 16
        uint32_t nlong, nbig, nparts, bad, half, heavy;  // heavy: bit p, part p is one crowded run of 256 bins
        uint32_t ntodo, todo_at[kTodo], todo_n[kTodo];
        alignas(16) K todo_lo[kTodo], todo_hi[kTodo];  // ranges still to sort: bounds, first position, keys
        alignas(16) unsigned char sort[sizeof(typename BlockSort<K, T>::Smem)];  // of a long bin by the whole CTA
    };
    static constexpr size_t kHead = (sizeof(Smem) + 15) & ~size_t(15);
    static constexpr size_t smem_bytes() { return kHead + (size_t)NBMAX * 2 + STAGE; }
    // the bins' words (NBMAX of 16 bits): free for the sink's use while the
    // only part of a segment is written
    __device__ static uint32_t *bins(unsigned char *smem) { return reinterpret_cast<uint32_t *>(smem + kHead); }

    // The slot that bin b's cursor stands at, given its word.
    __device__ static uint32_t slot_of(uint32_t b, uint32_t word, uint32_t wmask, uint32_t half) {
        return b > wmask ? (word >> 16) + half : word & 0xffffu;
    }

    // The long bins inside bins [b0, b0 + bn), each unsorted in the len slots
    // that end at its cursor (the first bin's start at slot pad).  A warp sorts a
    // bin of up to kWarpBin keys, up to kWarpMany where there are bins for half
    // of the warps, and up to kWarpMost of nearly one value; the CTA takes the
    // others one after the other.
    template <typename E>
    __device__ __noinline__ static void sort_long(Smem &sm, E *stage, uint32_t b0, uint32_t bn, uint32_t pad,
                                                   const uint32_t *cnt, uint32_t wmask, uint32_t half) {
        auto end_of = [=](uint32_t b) { return slot_of(b, cnt[b & wmask], wmask, half); };
        const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
        uint32_t nl = sm.nlong;
        if (tid == 0) sm.nbig = 0;
        __syncthreads();
        if (nl <= (uint32_t)kLongMax) {
            for (uint32_t i = warp; i < nl; i += W) {
                const uint32_t b = sm.longs[i] & 0xffffu, len = sm.longs[i] >> 16;
                if (b - b0 >= bn) continue;
                E *a = stage + (end_of(b) - len);
                if (len <= (uint32_t)kWarpBin) {
                    warp_sort(a, len);
                } else if (len <= (uint32_t)kWarpMost && warp_sort_mostly_one(a, len)) {
                    if (lane == 0) sm.longs[i] = 0;  // done
                } else if (lane == 0) {
                    atomicAdd(&sm.nbig, 1u);
                }
            }
        } else {
            // more than the list holds (values of a few dozen copies each, say):
            // every bin is looked at, and the list takes the larger ones
            for (uint32_t c = warp * 32; c < bn; c += T) {
                const uint32_t b = b0 + c + lane, end = end_of(b), len = end - (c + lane > 0 ? end_of(b - 1) : pad);
                for (uint32_t m = __ballot_sync(0xffffffffu, len > (uint32_t)kEdge); m; m &= m - 1) {
                    const int l = __ffs(m) - 1;
                    const uint32_t n = __shfl_sync(0xffffffffu, len, l), at = __shfl_sync(0xffffffffu, end, l) - n;
                    if (n <= (uint32_t)kWarpBin) warp_sort(stage + at, n);
                    else if (n > (uint32_t)kWarpMost || !warp_sort_mostly_one(stage + at, n)) {
                        if (lane == 0) sm.longs[atomicAdd(&sm.nbig, 1u)] = (b0 + c + l) | n << 16;
                    }
                }
            }
        }
        __syncthreads();
        const uint32_t nbig = sm.nbig;
        if (nbig == 0) return;
        if (nl > (uint32_t)kLongMax) nl = nbig;
        uint32_t warps_take = kWarpBin;
        if (kWarpMany > kWarpBin && nbig >= (uint32_t)W / 2) {
            warps_take = kWarpMany;
            for (uint32_t i = warp; i < nl; i += W) {
                const uint32_t b = sm.longs[i] & 0xffffu, len = sm.longs[i] >> 16;
                if (b - b0 < bn && len > (uint32_t)kWarpBin && len <= warps_take) warp_sort(stage + (end_of(b) - len), len);
            }
        }
        for (uint32_t i = 0; i < nl; i += 32) {  // (every warp reads the same entries, 32 at a time)
            const uint32_t mine = i + lane < nl ? sm.longs[i + lane] : 0u;
            const bool big = (mine & 0xffffu) - b0 < bn && mine >> 16 > warps_take;
            for (uint32_t m = __ballot_sync(0xffffffffu, big); m; m &= m - 1) {
                const uint32_t w = __shfl_sync(0xffffffffu, mine, __ffs(m) - 1), len = w >> 16;
                E *a = stage + (end_of(w & 0xffffu) - len);
                using BS = BlockSort<E, T>;
                typename BS::Smem &bs = *reinterpret_cast<typename BS::Smem *>(sm.sort);
                if (!BS::mostly_one(bs, a, (int)len)) BS::run(bs, a, (int)len);
            }
        }
    }

    template <typename E> __device__ static void order(E &a, E &b) {
        const E x = a, y = b;
        a = x < y ? x : y;
        b = x < y ? y : x;
    }

    // A window in order: the eight words of every lane (19 comparators), then a
    // bin across the border of two lanes -- my upper four words and the next
    // lane's lower four merge, each lane computing its own side -- then odd-even
    // transposition rounds until nothing is out of order (rarely any).
    template <typename E> __device__ static void sort_window(E (&x)[kPer]) {
        const int lane = threadIdx.x & 31;
        order(x[0], x[2]); order(x[1], x[3]); order(x[4], x[6]); order(x[5], x[7]);
        order(x[0], x[4]); order(x[1], x[5]); order(x[2], x[6]); order(x[3], x[7]);
        order(x[0], x[1]); order(x[2], x[3]); order(x[4], x[5]); order(x[6], x[7]);
        order(x[2], x[4]); order(x[3], x[5]);
        order(x[1], x[4]); order(x[3], x[6]);
        order(x[1], x[2]); order(x[3], x[4]); order(x[5], x[6]);
        E nx[4], pv[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            nx[j] = shfl_down_one(x[j]);
            pv[j] = shfl_up_one(x[4 + j]);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (lane < 31) x[4 + j] = nx[3 - j] < x[4 + j] ? nx[3 - j] : x[4 + j];
            if (lane > 0) x[j] = pv[3 - j] > x[j] ? pv[3 - j] : x[j];
        }
        order(x[4], x[6]); order(x[5], x[7]); order(x[4], x[5]); order(x[6], x[7]);
        order(x[0], x[2]); order(x[1], x[3]); order(x[0], x[1]); order(x[2], x[3]);
        for (;;) {
            bool bad = false;
#pragma unroll
            for (int j = 0; j + 1 < kPer; ++j) bad |= x[j + 1] < x[j];
            const E nxt = shfl_down_one(x[0]);
            bad |= lane < 31 && nxt < x[kPer - 1];
            if (!__any_sync(0xffffffffu, bad)) break;
#pragma unroll
            for (int j = 0; j + 1 < kPer; j += 2) order(x[j], x[j + 1]);
            const E up = shfl_up_one(x[kPer - 1]), dn = shfl_down_one(x[0]);
#pragma unroll
            for (int j = 1; j + 1 < kPer; j += 2) order(x[j], x[j + 1]);
            if (lane > 0) x[0] = up > x[0] ? up : x[0];
            if (lane < 31) x[kPer - 1] = dn < x[kPer - 1] ? dn : x[kPer - 1];
        }
    }

    // Writes a lane's keys key(j) of slots at + j, position p0 being slot pad; at
    // the ends of a part only those inside [pad, end).
    template <typename Sink, typename Key>
    __device__ static void put(const Sink &sink, uint32_t p0, int at, bool inner, int pad, int end, Key key) {
        const int64_t p = (int64_t)p0 + at - pad;
        if (inner) {
            sink.eight(p, key);
        } else {
#pragma unroll
            for (int j = 0; j < kPer; ++j)
                if (at + j >= pad && at + j < end) sink.one(p + j, key(j));
        }
    }

    // A part of np keys at stage[pad..): its windows, written to positions p0 on
    // (position p0 + j and slot pad + j have the same 16-byte alignment).
    template <typename Sink>
    __device__ static void emit_wide(const K *stage, int pad, int np, uint32_t p0, const Sink &sink) {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, end = pad + np;
        for (int w0 = warp * kStep; w0 < end; w0 += W * kStep) {
            const int at = w0 - kEdge + lane * kPer;
            const bool inner = w0 - kEdge >= pad && w0 + kWin - kEdge <= end;  // the whole window
            K x[kPer];
            if (inner) {
#pragma unroll
                for (int j = 0; j < kPer / V; ++j) {
                    const uint4 w = *reinterpret_cast<const uint4 *>(stage + at + j * V);
                    if constexpr (sizeof(K) == 4) {
                        x[j * 4] = w.x; x[j * 4 + 1] = w.y; x[j * 4 + 2] = w.z; x[j * 4 + 3] = w.w;
                    } else if constexpr (sizeof(K) == 16) {
                        x[j] = (u128)((uint64_t)w.w << 32 | w.z) << 64 | ((uint64_t)w.y << 32 | w.x);
                    } else {
                        x[j * 2] = (uint64_t)w.y << 32 | w.x;
                        x[j * 2 + 1] = (uint64_t)w.w << 32 | w.z;
                    }
                }
            } else {
#pragma unroll
                for (int j = 0; j < kPer; ++j)
                    x[j] = at + j < pad ? K(0) : (at + j < end ? stage[at + j] : all_ones<K>());
            }
            sort_window(x);
            if (lane >= kEdge / kPer && lane < 32 - kEdge / kPer)
                put(sink, p0, at, inner, pad, end, [&](int j) { return x[j]; });
        }
    }

    // The same from a narrow stage (p0: the part's first position in the range,
    // whose first position is `from` in the sink).
    template <typename Sink>
    __device__ static void emit_narrow(const Smem &sm, const S *stage, int pad, int np, uint32_t p0, uint32_t from,
                                       uint32_t nunits, K lo, const Sink &sink) {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, end = pad + np;
        for (int w0 = warp * kStep; w0 < end; w0 += W * kStep) {
            const int at = w0 - kEdge + lane * kPer;
            // the unit of the window's first position: the last one starting at or before it
            const uint32_t first = p0 + (uint32_t)(max(w0 - kEdge, pad) - pad);
            const uint32_t last = p0 + (uint32_t)(min(w0 + kWin - kEdge, end) - 1 - pad);
            uint32_t u0 = 0;
            for (uint32_t b = 0; b < nunits; b += 32) {
                const uint32_t below = __ballot_sync(0xffffffffu, b + lane < nunits && sm.unit[b + lane] <= first);
                u0 += (uint32_t)__popc(below);
                if (below != 0xffffffffu) break;
            }
            --u0;
            const bool inner = w0 - kEdge >= pad && w0 + kWin - kEdge <= end;  // the whole window
            const bool two = sm.unit[u0 + 2] > last;  // at most two units: offsets from the first fit a half word
            // an offset from unit u0: half word minus u0 << UB, which flips its top bit when u0 is odd
            const uint32_t flip = two && (u0 & 1u) ? (sizeof(K) == 4 ? 0x80008000u : 0x80000000u) : 0u;
            uint32_t s[kPer];
            if (inner) {
                uint4 w = *reinterpret_cast<const uint4 *>(stage + at);
                w = make_uint4(w.x ^ flip, w.y ^ flip, w.z ^ flip, w.w ^ flip);
                if constexpr (sizeof(K) == 4) {
                    s[0] = w.x & 0xffffu; s[1] = w.x >> 16; s[2] = w.y & 0xffffu; s[3] = w.y >> 16;
                    s[4] = w.z & 0xffffu; s[5] = w.z >> 16; s[6] = w.w & 0xffffu; s[7] = w.w >> 16;
                } else {
                    const uint4 y = *reinterpret_cast<const uint4 *>(stage + at + 4);
                    s[0] = w.x; s[1] = w.y; s[2] = w.z; s[3] = w.w;
                    s[4] = y.x ^ flip; s[5] = y.y ^ flip; s[6] = y.z ^ flip; s[7] = y.w ^ flip;
                }
            } else {
#pragma unroll
                for (int j = 0; j < kPer; ++j)
                    s[j] = at + j < pad ? 0u : (at + j < end ? (uint32_t)(S)(stage[at + j] ^ (S)flip) : 0xffffffffu);
            }
            if (two) {
                sort_window(s);
                const K base = lo + ((K)u0 << UB);
                if (lane >= kEdge / kPer && lane < 32 - kEdge / kPer)
                    put(sink, from + p0, at, inner, pad, end, [&](int j) { return base + s[j]; });
            } else {
                K x[kPer];
#pragma unroll
                for (int j = 0; j < kPer; ++j) {
                    if (at + j < pad) x[j] = K(0);
                    else if (at + j >= end) x[j] = all_ones<K>();
                    else {
                        uint32_t u = u0;
                        while (sm.unit[u + 1] <= p0 + (uint32_t)(at + j - pad)) ++u;
                        x[j] = lo + (((K)u << UB) | (s[j] & ((1u << UB) - 1u)));
                    }
                }
                sort_window(x);
                if (lane >= kEdge / kPer && lane < 32 - kEdge / kPer)
                    put(sink, from + p0, at, inner, pad, end, [&](int j) { return x[j]; });
            }
        }
    }

    template <typename Sink>
    __device__ static __noinline__ void emit_wide_apart(const K *stage, int pad, int np, uint32_t p0, const Sink &sink) {
        emit_wide(stage, pad, np, p0, sink);
    }
    template <typename Sink>
    __device__ static __noinline__ void emit_narrow_apart(const Smem &sm, const S *stage, int pad, int np, uint32_t p0, uint32_t from,
                                                          uint32_t nunits, K lo, const Sink &sink) {
        emit_narrow(sm, stage, pad, np, p0, from, nunits, lo, sink);
    }

    // Smallest and largest key of the segment (n >= 1), for every thread.
    template <typename Source>
    __device__ static void bounds(unsigned char *smem, const Source &src, int n, K &lo, K &hi) {
        K *red = reinterpret_cast<K *>(smem);
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        K mn = all_ones<K>(), mx = K(0);
        src.each(n, [&](K k) {
            mn = k < mn ? k : mn;
            mx = k > mx ? k : mx;
        });
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const K a = shfl_xor_any(mn, o), b = shfl_xor_any(mx, o);
            mn = a < mn ? a : mn;
            mx = b > mx ? b : mx;
        }
        if (lane == 0) {
            red[warp] = mn;
            red[W + warp] = mx;
        }
        __syncthreads();
        lo = red[0];
        hi = red[W];
        for (int w = 1; w < W; ++w) {
            lo = red[w] < lo ? red[w] : lo;
            hi = red[W + w] > hi ? red[W + w] : hi;
        }
        __syncthreads();
    }

    // Sorts the n keys of src into positions [0, n) of sink, as CTA g of G.
    // Returns false, in every CTA of the segment alike, when it gives up: more
    // crowded ranges than the list holds, more parts than there may be, or more
    // than 65,535 keys in a bin.  What was written by then is rewritten by whoever takes over.
    template <typename Source, typename Sink>
    __device__ static bool run(unsigned char *smem, const Source &src, int n, K lo, K hi, const Sink &sink, int g, int G) {
        Smem &sm = *reinterpret_cast<Smem *>(smem);
        if (threadIdx.x == 0) sm.ntodo = 0;
        if (!run_range(smem, src, n, (uint32_t)n, lo, hi, 0u, sink, g, G)) return false;
        __syncthreads();
        return sm.ntodo == 0 || run_crowded(smem, src, n, sink, g, G);
    }

    // The keys of src in a range.
    template <typename Source> struct Within {
        const Source &src;
        K lo, span;
        template <typename F> __device__ void each(int n, F f) const {
            src.each(n, [&](K k) {
                if (k - lo <= span) f(k);
            });
        }
    };
    static_assert(2 * W * sizeof(K) <= offsetof(Smem, longs), "bounds() leaves the ranges to sort alone");

    // The crowded ranges, each a small part of the one it came from (so this ends).
    template <typename Source, typename Sink>
    __device__ static __noinline__ bool run_crowded(unsigned char *smem, const Source &src, int n, const Sink &sink, int g,
                                                    int G) {
        Smem &sm = *reinterpret_cast<Smem *>(smem);
        for (;;) {
            __syncthreads();
            const uint32_t t = sm.ntodo;
            if (t == 0) return true;
            const Within<Source> in{src, sm.todo_lo[t - 1], sm.todo_hi[t - 1] - sm.todo_lo[t - 1]};
            const uint32_t at = sm.todo_at[t - 1], keys = sm.todo_n[t - 1];
            __syncthreads();
            if (threadIdx.x == 0) sm.ntodo = t - 1;
            K lo, hi;  // of the keys themselves: what crowds may be far narrower than its bins
            bounds(smem, in, n, lo, hi);
            if (lo == hi) {  // copies of one value: no need to count them
                for (uint32_t e = g * T + threadIdx.x; e < keys; e += G * T) sink.one((int64_t)at + e, lo);
                continue;
            }
            if (!run_range(smem, in, n, keys, lo, hi, at, sink, g, G)) return false;
        }
    }

    // The n keys that src, which reads nsrc, gives, all in [lo, hi], into
    // positions [base, base + n) of sink.
    template <typename Source, typename Sink>
    __device__ static bool run_range(unsigned char *smem, const Source &src, int nsrc, uint32_t n, K lo, K hi, uint32_t base,
                                     const Sink &sink, int g, int G) {
        Smem &sm = *reinterpret_cast<Smem *>(smem);
        uint32_t *cnt = reinterpret_cast<uint32_t *>(smem + kHead);
        unsigned char *stage = smem + kHead + (size_t)NBMAX * 2;
        const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
        // bins: a power of two about the number of keys
        int nbl = 9;
        while ((1 << nbl) < NBMAX && (1u << nbl) < n) ++nbl;
        const K range = hi - lo;
        const int bits = word_bits<K>(range);
        const int shift = bits > nbl ? bits - nbl : 0;
        const uint32_t nb = 1u << nbl, nseg = nb / kSegBins, hseg = nseg / 2, wmask = nb / 2 - 1;
        // a narrow stage where a wide one would need more parts (or, of 64-bit
        // keys, wherever it can be: its windows sort half words)
        const K nu = (range >> UB) + 1;
        const bool narrow = sizeof(K) <= 8 && (sizeof(K) == 8 || n > kUseWide) && shift + 3 <= UB && nu <= (K)kUnits &&
                            (nu <= 2 || (uint64_t)nu * kWin <= (uint64_t)n);
        const uint32_t nunits = (uint32_t)nu;
        for (uint32_t q = tid; q < nb / 8; q += T) reinterpret_cast<uint4 *>(cnt)[q] = make_uint4(0u, 0u, 0u, 0u);
        if (tid == 0) {
            sm.nlong = 0;
            sm.bad = 0;
        }
        __syncthreads();
        // keys outside [lo, hi] (a region that overflowed, which is reported) stay in bounds
        auto bin_of = [&](K v) { return min((uint32_t)(v >> shift), nb - 1u); };
        src.each(nsrc, [&](K k) {
            const uint32_t b = bin_of(k - lo);
            atomicAdd(&cnt[b & wmask], b > wmask ? 0x10000u : 1u);
        });
        __syncthreads();
        // a warp takes 256 words: 256 bins in the low halves, 256 in the high ones
        auto load8 = [&](uint32_t s, uint32_t (&w)[8]) {
            const uint4 a = reinterpret_cast<const uint4 *>(cnt)[s * 64 + lane * 2];
            const uint4 b = reinterpret_cast<const uint4 *>(cnt)[s * 64 + lane * 2 + 1];
            w[0] = a.x; w[1] = a.y; w[2] = a.z; w[3] = a.w;
            w[4] = b.x; w[5] = b.y; w[6] = b.z; w[7] = b.w;
        };
        for (uint32_t s = warp; s < hseg; s += W) {
            uint32_t w[8], l = 0, h = 0;
            load8(s, w);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                l += w[j] & 0xffffu;
                h += w[j] >> 16;
            }
            l = __reduce_add_sync(0xffffffffu, l);
            h = __reduce_add_sync(0xffffffffu, h);
            if (lane == 0) {
                sm.seg[s] = l;
                sm.seg[hseg + s] = h;
            }
        }
        __syncthreads();
        if (warp == 0) {
            uint32_t v[4], loc = 0, mx = 0;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint32_t s = lane * 4 + j;
                v[j] = s < nseg ? sm.seg[s] : 0u;
                loc += v[j];
                mx = max(mx, v[j]);
            }
            mx = __reduce_max_sync(0xffffffffu, mx);
            uint32_t tot;
            uint32_t at = warp_excl_scan(loc, &tot);
            __syncwarp();
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint32_t s = lane * 4 + j;
                if (s < nseg) sm.seg[s] = at;
                at += v[j];
            }
            if (lane == 31) sm.seg[nseg] = tot;
            __syncwarp();
            // One part when the stage holds the segment.  Its positions are 16
            // bits wide, counted from the middle bin's in the upper half of
            // the bins.  Otherwise a part starts at the first segment at or
            // past a multiple of target, so it holds at most target + mx keys,
            // and its positions count from its start.  (A bin count past 16
            // bits shows in the total.)
            const uint32_t use = narrow ? kUseNarrow : kUseWide, mid = sm.seg[hseg];
            uint32_t np = 1, half = mid;
            const uint32_t most = min(use, 65528u);
            bool ok = tot == n;
            const bool split = n > use || G > 1 || mid > 65000u || n - mid > 65000u;
            const bool crowded = split && mx > most / 2;
            if (crowded) {
                // parts one after the other, a crowded run of bins by itself
                half = 0;
                if (lane == 0 && ok) {
                    const uint32_t fits = shift > 0 ? most / 2 : most;
                    uint32_t from = 0, heavy = 0;
                    np = 0;
                    auto part = [&](uint32_t first, bool is_heavy) {
                        if (np < (uint32_t)kPartsMax) {
                            sm.pseg[np] = first;
                            heavy |= (is_heavy ? 1u : 0u) << np;
                        }
                        ++np;
                    };
                    for (uint32_t s = 0; s < nseg; ++s) {
                        const uint32_t c = sm.seg[s + 1] - sm.seg[s];
                        if (c > fits) {
                            if (s > from) part(from, false);
                            part(s, true);
                            from = s + 1;
                        } else if (sm.seg[s + 1] - sm.seg[from] > most) {
                            part(from, false);
                            from = s;
                        }
                    }
                    if (from < nseg) part(from, false);
                    sm.heavy = heavy;
                    ok = np <= (uint32_t)kPartsMax;
                    if (ok) sm.pseg[np] = nseg;
                }
                np = __shfl_sync(0xffffffffu, np, 0);
                ok = __shfl_sync(0xffffffffu, (int)ok, 0) != 0;
            } else {
                if (split) {
                    np = (n + (most - mx) - 1) / (most - mx);
                    np = min(max(np, (uint32_t)G), max(np, nseg));
                    ok = ok && np <= (uint32_t)kPartsMax;
                    half = 0;
                }
                const uint32_t target = (n + np - 1) / np;
                if (ok && lane < (int)np) {  // part `lane` starts at the first segment at or past lane * target
                    const uint32_t want = lane * target;
                    uint32_t a = 0, b = nseg;
                    while (a < b) {
                        const uint32_t m = (a + b) >> 1;
                        if (sm.seg[m] < want) a = m + 1;
                        else b = m;
                    }
                    sm.pseg[lane] = a;
                }
                if (lane == 0) {
                    if (ok) sm.pseg[np] = nseg;
                    sm.heavy = 0;
                }
            }
            if (lane == 0) {
                sm.nparts = np;
                sm.half = half;
                sm.bad = !ok;
                sm.unit[nunits <= (uint32_t)kUnits ? nunits : 0] = 0xffffffffu;
                sm.unit[nunits <= (uint32_t)kUnits ? nunits + 1 : 0] = 0xffffffffu;
            }
        }
        __syncthreads();
        if (sm.bad) return false;
        const uint32_t nparts = sm.nparts, half = sm.half, heavy = sm.heavy;
        // counts -> each bin's first slot inside its part; units and long bins recorded
        for (uint32_t s = warp; s < hseg; s += W) {
            uint32_t w[8], out_w[8];
            load8(s, w);
#pragma unroll
            for (int j = 0; j < 8; ++j) out_w[j] = 0;
#pragma unroll
            for (int hi_half = 0; hi_half < 2; ++hi_half) {
                const uint32_t sg = s + hi_half * hseg;
                uint32_t t = 0, m = 0;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const uint32_t c = (w[j] >> (16 * hi_half)) & 0xffffu;
                    t += c;
                    m = max(m, c);
                }
                uint32_t tot;
                uint32_t p = warp_excl_scan(t, &tot) + sm.seg[sg];
                uint32_t ps = 0;  // the part of this segment: the last one starting at or before it
                for (uint32_t q = 1; q < nparts; ++q)
                    if (sm.pseg[q] <= sg) ps = q;
                const uint32_t bin0 = sg * kSegBins + lane * 8;
                if (narrow && (bin0 & ((1u << (UB - shift)) - 1u)) == 0u && (bin0 >> (UB - shift)) < nunits)
                    sm.unit[bin0 >> (UB - shift)] = p;
                if (heavy >> ps & 1u) {
                    // sorted by itself later; where bins are single values, written here
                    if (shift == 0)
                        for (int l = 0; l < 32; ++l) {
                            uint32_t q = __shfl_sync(0xffffffffu, p, l);
#pragma unroll
                            for (int j = 0; j < 8; ++j) {
                                const uint32_t c = __shfl_sync(0xffffffffu, (w[j] >> (16 * hi_half)) & 0xffffu, l);
                                for (uint32_t e = g * 32 + lane; e < c; e += G * 32)
                                    sink.one((int64_t)base + q + e, lo + (K)(sg * kSegBins + l * 8 + j));
                                q += c;
                            }
                        }
                    continue;
                }
                // relative to the part's start (or the middle) and the stage's pad
                const uint32_t pstart = sm.seg[sm.pseg[ps]];
                p += (uint32_t)sink.pad(base + pstart) - pstart - (hi_half ? half : 0u);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    out_w[j] |= p << (16 * hi_half);
                    p += (w[j] >> (16 * hi_half)) & 0xffffu;
                }
                if (shift > 0 && m > (uint32_t)kEdge) {
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const uint32_t c = (w[j] >> (16 * hi_half)) & 0xffffu;
                        if (c > (uint32_t)kEdge) {
                            const uint32_t at = atomicAdd(&sm.nlong, 1u);
                            if (at < (uint32_t)kLongMax) sm.longs[at] = (bin0 + j) | c << 16;
                        }
                    }
                }
            }
            reinterpret_cast<uint4 *>(cnt)[s * 64 + lane * 2] = make_uint4(out_w[0], out_w[1], out_w[2], out_w[3]);
            reinterpret_cast<uint4 *>(cnt)[s * 64 + lane * 2 + 1] = make_uint4(out_w[4], out_w[5], out_w[6], out_w[7]);
        }
        __syncthreads();
        auto next_slot = [&](uint32_t b) {
            return slot_of(b, atomicAdd(&cnt[b & wmask], b > wmask ? 0x10000u : 1u), wmask, half);
        };
        auto place = [&](uint32_t b, K v, K k) {
            const uint32_t at = next_slot(b);
            if (narrow) reinterpret_cast<S *>(stage)[at] = (S)v;
            else reinterpret_cast<K *>(stage)[at] = k;
        };
        for (uint32_t part = g; part < nparts; part += G) {
            const uint32_t s0 = sm.pseg[part], s1 = sm.pseg[part + 1];
            const uint32_t p0 = sm.seg[s0], np = sm.seg[s1] - p0;
            if (np == 0 || (heavy >> part & 1u)) continue;  // uniform
            const uint32_t b0 = s0 * kSegBins, bn = (s1 - s0) * kSegBins;
            if (nparts == 1) {
                if (narrow) {
                    src.each(nsrc, [&](K k) {
                        const K v = k - lo;
                        const uint32_t b = bin_of(v);
                        reinterpret_cast<S *>(stage)[next_slot(b)] = (S)v;
                    });
                } else {
                    src.each(nsrc, [&](K k) {
                        const uint32_t b = bin_of(k - lo);
                        reinterpret_cast<K *>(stage)[next_slot(b)] = k;
                    });
                }
            } else {
                src.each(nsrc, [&](K k) {
                    const K v = k - lo;
                    const uint32_t b = bin_of(v);
                    if (b - b0 < bn) place(b, v, k);
                });
            }
            __syncthreads();
            const int pad = sink.pad(base + p0);
            if (sm.nlong) {
                if (sizeof(K) <= 8 && narrow) sort_long(sm, reinterpret_cast<S *>(stage), b0, bn, (uint32_t)pad, cnt, wmask, half);
                else sort_long(sm, reinterpret_cast<K *>(stage), b0, bn, (uint32_t)pad, cnt, wmask, half);
                __syncthreads();
            }
            if constexpr (sizeof(K) <= 8) if (narrow) {
                const S *halves = reinterpret_cast<const S *>(stage);
                if constexpr (Sink::kApart) emit_narrow_apart(sm, halves, pad, (int)np, p0, base, nunits, lo, sink);
                else emit_narrow(sm, halves, pad, (int)np, p0, base, nunits, lo, sink);
            }
            if (!narrow) {
                const K *words = reinterpret_cast<const K *>(stage);
                if constexpr (Sink::kApart) emit_wide_apart(words, pad, (int)np, base + p0, sink);
                else emit_wide(words, pad, (int)np, base + p0, sink);
            }
            __syncthreads();  // the next part reuses the stage
        }
        if (heavy && shift > 0) {
            if (tid == 0)
                for (uint32_t part = 0; part < nparts; ++part)
                    if (heavy >> part & 1u) {
                        const uint32_t s = sm.pseg[part], t = sm.ntodo++;
                        if (t >= (uint32_t)kTodo) continue;
                        const K first = (K)(s * kSegBins) << shift, past = ((K)kSegBins << shift) - 1;
                        sm.todo_lo[t] = lo + first;
                        sm.todo_hi[t] = range - first < past ? hi : lo + first + past;
                        sm.todo_at[t] = base + sm.seg[s];
                        sm.todo_n[t] = sm.seg[s + 1] - sm.seg[s];
                    }
            __syncthreads();
            if (sm.ntodo > (uint32_t)kTodo) return false;
        }
        return true;
    }
};

// The shapes it runs in: one CTA of 1024 threads per SM, two of 512, or five
// of 256 (228 KB of shared memory per SM, 1 KB of it reserved per CTA); for the
// 128-bit words of wide records two of 256 with twice the registers.
enum { kCountSmall = 0, kCountMedium = 1, kCountLarge = 2, kCountRecord = 3 };
template <int SIZE> struct CountShape {
    static constexpr int T = SIZE == kCountLarge ? 1024 : SIZE == kCountMedium ? 512 : 256;
    static constexpr int kPerSm = SIZE == kCountLarge ? 1 : SIZE == kCountSmall ? 5 : 2;
    static constexpr int kBins = SIZE == kCountLarge ? 32768 : SIZE == kCountMedium ? 16384 : SIZE == kCountRecord ? 8192 : 4096;
    static constexpr int kStageBytes = SIZE == kCountLarge ? 149504 : SIZE == kCountMedium ? 69632 : SIZE == kCountRecord ? 81920 : 30720;
    template <typename K> using Sort = CountSort<K, T, kBins, kStageBytes>;
    static_assert(kPerSm * (Sort<uint64_t>::smem_bytes() + 1024) <= 228 * 1024, "resident CTAs");
};

// The shape for segments of about `keys` keys: the smallest whose stage holds
// one with room for uneven ones, because several small CTAs on an SM hide each
// other's phases and one part reads the segment least often.
inline int count_sort_size(int64_t keys, int key_bytes) {
    if (keys * key_bytes <= CountShape<kCountSmall>::kStageBytes * 3 / 4) return kCountSmall;
    if (keys * key_bytes <= CountShape<kCountMedium>::kStageBytes * 7 / 8) return kCountMedium;
    return kCountLarge;
}

// CTAs per segment: one when the segments fill the GPU, else as many as keep it
// full while each still places 1024 keys or more.
template <int SIZE> int count_sort_ctas(int64_t segments, int64_t keys) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t slots = (int64_t)(sms > 0 ? sms : 1) * CountShape<SIZE>::kPerSm;
    const int64_t g = segments > 0 ? slots / segments : 1;
    return (int)imax64(1, imin64(imin64(g, keys / 1024), 16));
}

} // namespace bsps
