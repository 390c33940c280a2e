// route_keys.cu -- classification and the routing permutation for keys
// without payloads (Fig. 1 steps 9-11; Fig. 2 steps 9-11), in one pass, and for
// 4-byte keys with payloads as words phi << 32 | input position.
//
// Without payloads the order of keys inside a bucket is free (equal keys
// cannot be told apart; the words of pairs carry their order with them), so the
// per-bucket prefix of Fig. 1 step 9 need not follow input order: every chunk of keys reserves its run in each bucket
// region with one atomic on that bucket's cursor.  A chunk is loaded into
// registers with 16-byte loads, each key is classified once (Fig. 2 step 9)
// and ranked inside the chunk with a shared-memory atomic, the chunk is
// grouped by bucket in shared memory, and every bucket's run is written
// contiguously into its region.  One CTA of 1024 threads per SM; chunks of
// 16K keys keep the reservations to about one per four keys.
//
// The kernel is bound by the shared-memory pipe (a random access costs a warp
// about 3.5 wavefronts) and by latency between barriers:
//  - Each step runs over all of a thread's keys before the next, so the loads
//    of one step overlap.
//  - The radix index says of a key's cell whether splitters share it: none (7
//    of 8 cells at 2^15 cells and 4096 splitters), and the cell names the
//    bucket; one or two, and as many comparisons decide; more, or a key equal
//    to a splitter, and that key searches, where it lies in the registers (2^26
//    keys of 256 Zipf values into 4096: 0.97 ms, and 2.38 when all keys of such
//    a thread searched in a loop that picked them out one by one; 2^26 normal
//    floats into 1024: 0.43 and 1.00).
//  - The grouped chunk keeps no bucket numbers.  A bit marks where each
//    bucket's run starts, so a slot's run is a bit count away, and the runs are
//    reserved and written by their ordinal among the chunk's non-empty buckets.
//  - The counters are double-buffered: one chunk is written while the next is
//    classified, with no barrier between the two.
// 2^28 int32 keys into 4096 buckets: 1.50 ms, 1.77 with an index of 2^14 cells,
// a search per key and one set of counters.  2^28 doubles with the learned
// classifier into 4096: 4.0 ms with a thread's keys classified one after the
// other, 5.9 in step (the state of ten keys spills).  2^22 pairs: 631 us for
// the whole sort by the look-back route and the stable bucket sort, 213 as words.
#include <algorithm>
#include <type_traits>

#include "classify.cuh"
#include "many.cuh"
#include "mlp.cuh"

namespace bsps {

constexpr int kRkThreads = 1024;
constexpr int kEarly = 4;  // buckets per thread reserved before the grouping
constexpr size_t kRkSmemBudget = 227 * 1024;  // splitters in shared memory up to this size
// keys per thread (fewer with the network's registers in use).  8-byte keys
// with the learned classifier take chunks of 10K with the splitters in global
// memory (L1-cached): with thousands of sub-buckets the per-chunk work over
// all of them (scan, reservations) would otherwise weigh as much as the keys,
// and a key reads one or two splitters.  The splitter tree reads more (skewed
// keys crowd a few cells of the radix index) and keeps its splitters on chip
// with chunks of 8K.
// With payloads (PAIRS) the words that move are twice the keys' size: 8K.
template <typename K, bool LEARNED = false, bool PAIRS = false> constexpr int rk_items() {
    return sizeof(K) == 8 ? (LEARNED ? 10 : 8) : (LEARNED || PAIRS ? 8 : 16);
}
template <typename K, bool LEARNED = false, bool PAIRS = false> constexpr int rk_chunk() {
    return kRkThreads * rk_items<K, LEARNED, PAIRS>();
}

template <typename K> struct RouteKeysArgs {
    const K *keys;
    int64_t n;
    const LutParams<K> *lutp;
    const uint16_t *lut;
    const K *vphi;
    const uint32_t *vtag;
    uint32_t P;
    int64_t chunks;
    uint32_t *cursor;   // keys routed so far per sub-bucket
    void *regions;      // keys, or words phi << 32 | position
    int64_t cap;
    DevStatus *st;
    const MlpTables *mlp_tables;  // learned classifier (nullable): the network's evaluation form
    const uint16_t *ylut;         // ... and the index over its output
    int lut_bits;                 // cells of `lut`
    uint32_t tag_floor;           // a key's tag is max(position, tag_floor): n - 1 drops the tie-break
    uint32_t few_above;           // PAIRS: left to the look-back route if the sample's keys repeat more often
};

// Shared memory: the radix index (with the learned classifier: the index over
// the network's output, in the same slot, and the network's tables), the
// splitters' phi (global memory, L1-cached, when they do not fit), two sets of
// per-bucket counts, the non-empty buckets of a chunk with their starts and
// region offsets, the run marks, and the chunk grouped by bucket.
template <typename K, bool LEARNED, bool PAIRS = false> struct RouteKeysLayout {
    // Buckets a call may have: the bound bsps_get_plan documents (counters,
    // offsets, the index and a chunk with 16-bit bucket numbers in 227 KB; the
    // layout below needs less).  `fits` says whether the splitters fit, too.
    static size_t limit_bytes(uint32_t P, bool &fits) {
        size_t total = 0;
        for (int pass = 0; pass < 2; ++pass) {
            fits = pass == 0;
            total = 64;
            auto take = [&](size_t bytes) { total = (total + bytes + 15) & ~size_t(15); };
            take(LEARNED ? sizeof(MlpTables) : 0);
            take(sizeof(uint16_t) * (kLutCells + 2));
            take(fits ? sizeof(K) * (P > 1 ? P - 1 : 1) : 0);
            take(sizeof(uint32_t) * (P + 4));
            take(sizeof(uint32_t) * (P + 4));
            total += (sizeof(K) + 2) * rk_chunk<K, LEARNED>() + 128;
            if (total <= kRkSmemBudget) break;
        }
        return total;
    }
    size_t mlp, lut, sphi, cnt, dlt, heads, ord, stage, total;
    bool sphi_in_smem, two_counts;
    __host__ __device__ RouteKeysLayout(uint32_t P, int lut_bits) {
        constexpr int CH = rk_chunk<K, LEARNED, PAIRS>();
        for (int pass = 0; pass < 4; ++pass) {  // what many buckets leave no room for goes
            sphi_in_smem = pass < 2;
            two_counts = pass % 2 == 0;
            size_t o = 64;  // LutParams
            auto take = [&](size_t bytes) {
                const size_t at = o;
                o = (o + bytes + 15) & ~size_t(15);
                return at;
            };
            mlp = take(LEARNED ? sizeof(MlpTables) : 0);
            lut = take(sizeof(uint16_t) * ((1 << lut_bits) + 2));
            sphi = take(sphi_in_smem ? sizeof(K) * P : 0);
            cnt = take(sizeof(uint32_t) * (two_counts ? 2 : 1) * P);
            dlt = take(sizeof(uint32_t) * P);
            heads = take(CH / 8);
            ord = take(CH / 32 * 2);
            stage = take((PAIRS ? 8 : sizeof(K)) * CH);
            total = o + 128;  // scan scratch
            if (total <= kRkSmemBudget - 512) break;  // (a batch's arguments are kept there, too)
        }
    }
};
static_assert(sizeof(LutParams<uint64_t>) <= 64, "radix index parameters fit their slot");

// A shared-memory word where `take` holds, else all ones: the lanes that do not
// take it cost the access no bank.
__device__ __forceinline__ uint32_t ld_shared_if(const uint32_t *p, bool take) {
    uint32_t v;
    asm("{ .reg .pred q; setp.ne.u32 q, %2, 0; mov.u32 %0, 0xffffffff; @q ld.shared.u32 %0, [%1]; }"
        : "=r"(v) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"((uint32_t)take));
    return v;
}
__device__ __forceinline__ uint64_t ld_shared_if(const uint64_t *p, bool take) {
    uint64_t v;
    asm("{ .reg .pred q; setp.ne.u32 q, %2, 0; mov.u64 %0, 0xffffffffffffffff; @q ld.shared.u64 %0, [%1]; }"
        : "=l"(v) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"((uint32_t)take));
    return v;
}

template <int DT, bool LEARNED, bool MANY, bool PAIRS = false>
__global__ void __launch_bounds__(kRkThreads, 1) route_keys_kernel(const Many<RouteKeysArgs<typename KeyTraits<DT>::T>> many) {
    using K = typename KeyTraits<DT>::T;
    const Pick<MANY, RouteKeysArgs<K>> pk(many);
    const RouteKeysArgs<K> &a = pk.a;
    if constexpr (PAIRS)
        if (a.st->repeats > a.few_above) return;
    constexpr int T = kRkThreads, IT = rk_items<K, LEARNED, PAIRS>(), CH = rk_chunk<K, LEARNED, PAIRS>(),
                  V = 16 / (int)sizeof(K);
    using Word = typename std::conditional<PAIRS, uint64_t, K>::type;  // what moves
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const RouteKeysLayout<K, LEARNED, PAIRS> L(a.P, a.lut_bits);
    Word *regions = reinterpret_cast<Word *>(a.regions);
    LutParams<K> &lps = *reinterpret_cast<LutParams<K> *>(smem_raw);
    MlpTables *mt = reinterpret_cast<MlpTables *>(smem_raw + L.mlp);
    uint16_t *lut = reinterpret_cast<uint16_t *>(smem_raw + L.lut);
    K *sphi_s = reinterpret_cast<K *>(smem_raw + L.sphi);
    const K *sphi = L.sphi_in_smem ? sphi_s : a.vphi;
    uint32_t *cnt_a = reinterpret_cast<uint32_t *>(smem_raw + L.cnt), *cnt = cnt_a;  // this chunk's counts, then starts
    uint32_t *dlt = reinterpret_cast<uint32_t *>(smem_raw + L.dlt);            // run -> bucket | keys << 16, then region slot - chunk slot
    uint32_t *heads = reinterpret_cast<uint32_t *>(smem_raw + L.heads);        // bit s: a run starts at slot s
    uint16_t *ord = reinterpret_cast<uint16_t *>(smem_raw + L.ord);            // run holding slot 32 w
    Word *stage = reinterpret_cast<Word *>(smem_raw + L.stage);
    uint32_t *tmp = reinterpret_cast<uint32_t *>(smem_raw + L.total - 128);
    __shared__ uint32_t overflowed, nruns_s;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t P = a.P;
    static_assert(kYCells == kLutCells, "the learned index takes the radix index's slot");
    const int cells = 1 << a.lut_bits;
    // index entry: splitters below the cell, and whether one or more share it
    constexpr uint32_t kDropped = 0xffffffffu;
    constexpr uint32_t kOne = 0x4000u, kMore = 0x8000u, kBelow = 0x3fffu;
    const uint16_t *lut_src = LEARNED ? a.ylut : a.lut;
    for (int i = tid; i <= cells; i += T) {
        const uint32_t v = lut_src[i];
        const uint32_t in = !LEARNED && i < cells ? lut_src[i + 1] - v : 0u;
        lut[i] = (uint16_t)(v | (in == 0 ? 0u : in == 1 ? kOne : kMore));
    }
    if (L.sphi_in_smem)  // (entry P - 1 is all ones)
        for (uint32_t i = tid; i < P; i += T) sphi_s[i] = a.vphi[i];
    for (uint32_t b = tid; b < (L.two_counts ? 2 * P : P); b += T) cnt[b] = 0;
    if constexpr (LEARNED) {
        const uint32_t *src = reinterpret_cast<const uint32_t *>(a.mlp_tables);
        uint32_t *dst = reinterpret_cast<uint32_t *>(mt);
        for (int q = tid; q < (int)(sizeof(MlpTables) / 4); q += T) dst[q] = src[q];
    }
    if (tid == 0) {
        lps = *a.lutp;
        overflowed = 0;
    }
    __syncthreads();
    const LutParams<K> lp = lps;
    const bool vec = ((uintptr_t)a.keys & 15) == 0;
    // buckets [b_lo, b_hi) are this thread's in the scan
    const uint32_t per = (P + T - 1) / T;
    const uint32_t b_lo = min(P, tid * per), b_hi = min(P, b_lo + per);
    const uint32_t cap = (uint32_t)a.cap;
    uint32_t n_mis = 0, n_steps = 0;

    // chunk keys into registers (key i of a thread is chunk key at(i))
    auto at = [&](int i) { return ((i / V) * T + tid) * V + i % V; };
    K kk[IT];
    auto load_chunk = [&](int64_t ch) {
        const int64_t e0 = ch * CH;
        const int nh = (int)imin64(CH, a.n - e0);
#pragma unroll
        for (int j = 0; j < IT / V; ++j) {
            const int q = (j * T + tid) * V;
            if (vec && q + V <= nh) {
                const uint4 w = __ldg(reinterpret_cast<const uint4 *>(a.keys + e0 + q));
                if constexpr (sizeof(K) == 4) {
                    kk[j * V + 0] = w.x; kk[j * V + 1] = w.y; kk[j * V + 2] = w.z; kk[j * V + 3] = w.w;
                } else {
                    kk[j * V + 0] = ((uint64_t)w.y << 32) | w.x;
                    kk[j * V + 1] = ((uint64_t)w.w << 32) | w.z;
                }
            } else {
#pragma unroll
                for (int e = 0; e < V; ++e) kk[j * V + e] = q + e < nh ? a.keys[e0 + q + e] : K(0);
            }
        }
    };
    if ((int64_t)pk.block < a.chunks) load_chunk(pk.block);

    for (int64_t ch = pk.block; ch < a.chunks; ch += pk.blocks) {
        const int64_t e0 = ch * CH;
        const int nh = (int)imin64(CH, a.n - e0);
        // ---- classify (Fig. 2 step 9): bucket of every key, P for none ----
        uint32_t br[IT];
        auto classify = [&](auto full) {  // full: a whole chunk
            auto mine = [&](int i) { return decltype(full)::value || at(i) < nh; };
            if constexpr (LEARNED) {
#pragma unroll
                for (int i = 0; i < IT; ++i) {
                    const K raw = kk[i];
                    kk[i] = KeyTraits<DT>::phi(raw);
                    br[i] = P;
                    if (mine(i)) {
                        uint32_t steps;
                        bool mis;
                        br[i] = classify_learned<DT>(raw, max((uint32_t)(e0 + at(i)), a.tag_floor), *mt, lut, P - 1, sphi,
                                                     a.vtag, steps, mis);
                        n_mis += mis;
                        n_steps += steps;
                    }
                }
            } else {
                const K base = lp.base, span = lp.span;
#pragma unroll
                for (int i = 0; i < IT; ++i) {
                    kk[i] = KeyTraits<DT>::phi(kk[i]);
                    const K d = (kk[i] > base ? kk[i] : base) - base;
                    br[i] = lut[(uint32_t)((d < span ? d : span) >> lp.shift)];
                }
                // the cell's first splitter and, where more than one share it, the
                // second; a third, or a key equal to a splitter: search
                uint32_t search = 0;  // bit i: key i
                auto decide = [&](auto splitter) {
#pragma unroll
                    for (int i = 0; i < IT; ++i) {
                        const uint32_t e = br[i], j = e & kBelow;
                        const K s1 = splitter(j, e >= kOne), s2 = splitter(j + 1, e >= kMore);
                        search |= (mine(i) && (s1 == kk[i] || s2 <= kk[i]) ? 1u : 0u) << i;
                        br[i] = mine(i) ? j + (s1 < kk[i] ? 1u : 0u) : P;
                    }
                };
                if (L.sphi_in_smem) decide([&](uint32_t j, bool take) { return ld_shared_if(sphi_s + j, take); });
                else decide([&](uint32_t j, bool take) { return take ? a.vphi[j] : all_ones<K>(); });
                if (__any_sync(0xffffffffu, search != 0)) {
                    // those keys again, exactly, each where it lies in the registers
                    // (inputs of few values take this for every key)
#pragma unroll
                    for (int i = 0; i < IT; ++i) {
                        if (!(search >> i & 1u)) continue;
                        const K k = kk[i];
                        const uint32_t tag = max((uint32_t)e0 + at(i), a.tag_floor);
                        uint32_t lo = P - 1, hi = P - 1;
                        if (k - base <= span) {  // (a key below the base meets no splitter)
                            const uint32_t c = (uint32_t)((k - base) >> lp.shift);
                            lo = lut[c] & kBelow;
                            hi = lut[c + 1] & kBelow;
                        }
                        while (lo < hi) {
                            const uint32_t mid = (lo + hi) >> 1;
                            const K s = sphi[mid];
                            bool le = s < k;
                            if (s == k) le = a.vtag[mid] <= tag;  // tags are read on ties only
                            lo = le ? mid + 1 : lo;
                            hi = le ? hi : mid;
                        }
                        br[i] = lo;
                    }
                }
            }
        };
        if (nh == CH) classify(std::true_type());
        else classify(std::false_type());
        // ---- rank inside the chunk: bucket << 16 | rank ----
        // where a warp's first keys share lane 0's bucket (runs of one bucket
        // are common in skewed inputs) its lanes' atomics are merged
        const uint32_t first = __shfl_sync(0xffffffffu, br[0], 0);
        if (__popc(__ballot_sync(0xffffffffu, br[0] == first)) > 4) {
#pragma unroll
            for (int i = 0; i < IT; ++i) {
                const uint32_t b = br[i], b0 = __shfl_sync(0xffffffffu, b, 0);
                const bool ok = b < P;
                const uint32_t same = __ballot_sync(0xffffffffu, ok && b == b0);
                uint32_t r = 0;
                if (ok) {
                    if (b != b0) {
                        r = atomicAdd(&cnt[b], 1u);
                    } else {
                        const int leader = __ffs(same) - 1;
                        uint32_t r0 = 0;
                        if (lane == leader) r0 = atomicAdd(&cnt[b], (uint32_t)__popc(same));
                        r = __shfl_sync(same, r0, leader) + __popc(same & lanemask_lt());
                    }
                }
                br[i] = b << 16 | r;
            }
        } else if (nh == CH) {
#pragma unroll
            for (int i = 0; i < IT; ++i) br[i] = br[i] << 16 | atomicAdd(&cnt[br[i]], 1u);
        } else {
#pragma unroll
            for (int i = 0; i < IT; ++i) br[i] = br[i] << 16 | (br[i] < P ? atomicAdd(&cnt[br[i]], 1u) : 0u);
        }
        __syncthreads();
        // ---- where each bucket starts inside the chunk, and its run's ordinal ----
        for (int w = tid; w < CH / 32; w += T) heads[w] = 0;
        uint32_t local = 0;  // keys | non-empty buckets << 16
        for (uint32_t b = b_lo; b < b_hi; ++b) {
            const uint32_t c = cnt[b];
            local += c + (c ? 0x10000u : 0u);
        }
        uint32_t wtot;
        const uint32_t wex = warp_excl_scan(local, &wtot);
        if (lane == 31) tmp[warp] = wtot;
        __syncthreads();
        uint32_t run = wex;
        {
            uint32_t all;
            const uint32_t ye = warp_excl_scan(tmp[lane], &all);  // T / 32 = 32 warps
            run += __shfl_sync(0xffffffffu, ye, warp);
            if (tid == 0) nruns_s = all >> 16;
        }
        for (uint32_t b = b_lo; b < b_hi; ++b) {
            const uint32_t c = cnt[b];
            if (c) {
                const uint32_t s0 = run & 0xffffu, o = run >> 16, w0 = (s0 + 31) >> 5, w1 = (s0 + c + 31) >> 5;
                cnt[b] = s0;
                dlt[o] = b | c << 16;
                atomicOr(&heads[s0 >> 5], 1u << (s0 & 31u));
                for (uint32_t w = w0; w < w1; ++w) ord[w] = (uint16_t)o;
                run += c + 0x10000u;
            }
        }
        __syncthreads();
        const uint32_t nruns = nruns_s;
        // the first kEarly of my runs are reserved now, so that the atomics'
        // round trip overlaps the grouping below
        uint32_t at_e[kEarly];
#pragma unroll
        for (int j = 0; j < kEarly; ++j) {
            const uint32_t o = j * T + tid;
            at_e[j] = 0;
            if (o < nruns) at_e[j] = atomicAdd(&a.cursor[dlt[o] & 0xffffu], dlt[o] >> 16);
        }
        // ---- group the chunk by bucket ----
        auto word = [&](int i) -> Word {
            if constexpr (PAIRS) return (uint64_t)kk[i] << 32 | (uint32_t)(e0 + at(i));
            else return kk[i];
        };
        if (nh == CH) {
#pragma unroll
            for (int i = 0; i < IT; ++i) stage[cnt[br[i] >> 16] + (br[i] & 0xffffu)] = word(i);
        } else {
#pragma unroll
            for (int i = 0; i < IT; ++i)
                if (br[i] >> 16 < P) stage[cnt[br[i] >> 16] + (br[i] & 0xffffu)] = word(i);
        }
        // the next chunk's keys load while this one is reserved and written
        if (ch + pk.blocks < a.chunks) load_chunk(ch + pk.blocks);
        // ---- reserve each bucket's run: one atomic per bucket and chunk ----
        auto reserved = [&](uint32_t o, uint32_t got) {
            const uint32_t b = dlt[o] & 0xffffu, c = dlt[o] >> 16;
            const bool fits = got + c <= cap;  // (fewer than 2^31 keys)
            if (!fits) {
                overflowed = 1;
                atomicExch(&a.st->overflow, 1);
                set_error(a.st, BSPS_ERR_BUCKET_OVERFLOW);
            }
            dlt[o] = fits ? b * cap + got - cnt[b] : kDropped;  // region slot of chunk slot s: dlt[o] + s
        };
#pragma unroll
        for (int j = 0; j < kEarly; ++j)
            if (j * T + tid < nruns) reserved(j * T + tid, at_e[j]);
        for (uint32_t g0 = kEarly * T + tid; g0 < nruns; g0 += 8 * T) {
            uint32_t got[8];  // eight reservations in flight at a time
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const uint32_t o = g0 + j * T;
                got[j] = o < nruns ? atomicAdd(&a.cursor[dlt[o] & 0xffffu], dlt[o] >> 16) : 0u;
            }
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (g0 + j * T < nruns) reserved(g0 + j * T, got[j]);
        }
        __syncthreads();
        // ---- every bucket's run, contiguously into its region ----
        auto run_of = [&](uint32_t s) {  // (a warp's slots are one word of the marks)
            return ord[s >> 5] + (uint32_t)__popc(heads[s >> 5] & (0xfffffffeu & (0xffffffffu >> (31 - (s & 31u)))));
        };
        if (overflowed) {  // a run that passes its region's end is not written (the overflow is reported)
            for (int s = tid; s < nh; s += T) {
                const uint32_t d = dlt[run_of(s)];
                if (d != kDropped) regions[d + (uint32_t)s] = stage[s];
            }
        } else if (nh == CH) {
#pragma unroll 8
            for (int i = 0; i < IT; ++i) {
                const uint32_t s = i * T + tid;
                regions[dlt[run_of(s)] + s] = stage[s];
            }
        } else {
            for (int s = tid; s < nh; s += T) regions[dlt[run_of(s)] + (uint32_t)s] = stage[s];
        }
        // this chunk's counts are free again; the next chunk counts in the others
        for (uint32_t b = tid; b < P; b += T) cnt[b] = 0;
        if (L.two_counts) cnt = cnt == cnt_a ? cnt_a + P : cnt_a;
        else __syncthreads();
    }
    if constexpr (LEARNED) {
        const uint32_t m = __reduce_add_sync(0xffffffffu, n_mis), stp = __reduce_add_sync(0xffffffffu, n_steps);
        if (lane == 0 && (m | stp)) {
            atomicAdd(&a.st->mispredicted, (unsigned long long)m);
            atomicAdd(&a.st->correction_steps, (unsigned long long)stp);
        }
    }
}

template <int DT, bool LEARNED, bool PAIRS = false> static cudaError_t launch_t(Exec &x) {
    using K = typename KeyTraits<DT>::T;
    constexpr int64_t CH = rk_chunk<K, LEARNED, PAIRS>();
    auto takes = [](const Ctx &c) { return (c.pl.classify == BSPS_LEARNED) == LEARNED; };
    size_t smem = 0;
    int64_t all = 0;  // chunks of every call
    for (int i = 0; i < x.count; ++i)
        if (takes(x.calls[i])) {
            const Plan &p = x.calls[i].pl;
            smem = std::max(smem, RouteKeysLayout<K, LEARNED, PAIRS>((uint32_t)p.P, LEARNED ? kLutBits : p.lut_bits).total);
            all += (p.n + CH - 1) / CH;
        }
    if (smem == 0) return cudaSuccess;
    if (smem > kRkSmemBudget - 512) return cudaErrorInvalidValue;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    sms = std::max(sms, 1);
    return launch_calls<RouteKeysArgs<K>>(x, route_keys_kernel<DT, LEARNED, false, PAIRS>,
                                          route_keys_kernel<DT, LEARNED, !PAIRS, PAIRS>, kRkThreads, DynSmem(smem, kRkSmemBudget - 512),
                                          [=](const Ctx &c, RouteKeysArgs<K> &a) {
        if (!takes(c)) return 0u;
        const Plan &p = c.pl;
        a.keys = (const K *)c.keys_in;
        a.n = p.n;
        a.lutp = (const LutParams<K> *)c.ly.lutp;
        a.lut = c.ly.lut;
        a.vphi = (const K *)c.ly.vphi;
        a.vtag = c.ly.vtag;
        a.P = (uint32_t)p.P;
        a.chunks = (p.n + CH - 1) / CH;
        a.cursor = c.ly.cursor;
        a.regions = c.ly.reg_keys;
        a.cap = p.cap;
        a.st = c.ly.status;
        a.mlp_tables = c.ly.mlp_tables;
        a.ylut = c.ly.ylut;
        a.lut_bits = LEARNED ? kLutBits : p.lut_bits;
        a.tag_floor = p.dup_off ? (uint32_t)(p.n - 1) : 0u;
        a.few_above = c.both_routes ? repeats_above(p) : 0xffffffffu;
        // one CTA per SM; of a batch's CTAs (each loads the index first) every
        // call gets its share of two waves
        const int64_t share = all <= 2 * sms ? a.chunks : imax64(1, 2 * sms * a.chunks / all);
        return (uint32_t)imin64(a.chunks, c.pl.n == 0 ? 0 : imin64(sms, share));
    });
}

template <int DT> static cudaError_t launch_d(Exec &x) {
    const cudaError_t e = launch_t<DT, false>(x);
    return e != cudaSuccess ? e : launch_t<DT, true>(x);
}

cudaError_t launch_route_keys(Exec &x) {
    switch (x.calls[0].pl.dtype) {
    case BSPS_U32: return launch_d<BSPS_U32>(x);
    case BSPS_I32: return launch_d<BSPS_I32>(x);
    case BSPS_F32: return launch_d<BSPS_F32>(x);
    default: return launch_d<BSPS_F64>(x);
    }
}

template <int DT> static cudaError_t launch_pairs_d(Exec &x) {
    return x.calls[0].pl.classify == BSPS_LEARNED ? launch_t<DT, true, true>(x) : launch_t<DT, false, true>(x);
}

cudaError_t launch_route_words(Exec &x) {
    switch (x.calls[0].pl.dtype) {
    case BSPS_U32: return launch_pairs_d<BSPS_U32>(x);
    case BSPS_I32: return launch_pairs_d<BSPS_I32>(x);
    case BSPS_F32: return launch_pairs_d<BSPS_F32>(x);
    default: return cudaErrorInvalidValue;
    }
}

static size_t limit_bytes(const Plan &pl, bool &fits) {
    const uint32_t P = (uint32_t)pl.P;
    const bool l = pl.classify == BSPS_LEARNED;
    if (pl.key_bytes == 8) return l ? RouteKeysLayout<uint64_t, true>::limit_bytes(P, fits) : RouteKeysLayout<uint64_t, false>::limit_bytes(P, fits);
    return l ? RouteKeysLayout<uint32_t, true>::limit_bytes(P, fits) : RouteKeysLayout<uint32_t, false>::limit_bytes(P, fits);
}

size_t route_keys_smem_bytes(const Plan &pl) {
    bool fits;
    return limit_bytes(pl, fits);
}

bool route_keys_splitters_in_smem(const Plan &pl) {
    bool fits;
    limit_bytes(pl, fits);
    return fits;
}

bool route_keys_fine_index(const Plan &pl) {
    if (pl.classify == BSPS_LEARNED) return false;
    const uint32_t P = (uint32_t)pl.P;
    if (pl.key_bytes == 8) {
        const RouteKeysLayout<uint64_t, false> l(P, kLutBitsFine);
        return l.sphi_in_smem && l.two_counts;
    }
    const RouteKeysLayout<uint32_t, false> l(P, kLutBitsFine);
    return l.sphi_in_smem && l.two_counts;
}

} // namespace bsps
