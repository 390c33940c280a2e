// kernels.cuh -- the plan of one sort call, the workspace layout, and the
// host-side launchers of each step of the path.
#pragma once

#include "common.cuh"

namespace bsps {

struct MlpNorm;

// Number of cells of the radix index placed in front of the splitter tree.
constexpr int kLutBits = 14;
constexpr int kLutCells = 1 << kLutBits;
constexpr int kLutBitsFine = kLutBits + 1;  // keys without payloads, where it fits (with 4096 splitters 7 of 8 cells
                                            // hold none, against 3 of 4: routing 2^28 keys 1.77 -> 1.66 ms)

// Routing geometry (Fig. 1 steps 9-11).
constexpr int kRouteThreads = 1024;
constexpr int kRouteTile = 65536;                           // keys per look-back tile
template <typename K> constexpr int route_items() { return sizeof(K) == 8 ? 4 : 8; }
template <typename K> constexpr int route_chunk() { return kRouteThreads * route_items<K>(); }
constexpr size_t kRouteSmemBudget = 220 * 1024;

// Bucket / block sort geometry (Fig. 1 step 3, Fig. 2 step 12): 1024-thread
// CTAs, keys per thread of the on-chip segment sort.
constexpr int kSortThreads = 1024;
constexpr int kRunItems32 = 10;        // block sort with input-slot companion, 4-byte keys
constexpr int kRunItems64 = 8;         // ... 8-byte keys
constexpr int kBucketItems32 = 14;     // sub-bucket sort, keys only, 4-byte keys
constexpr int kBucketItems64 = 10;     // ... 8-byte keys
constexpr int kPairItems32 = 12;       // sub-bucket sort with payload slots, 4-byte keys
constexpr int kPairItems64 = 8;        // ... 8-byte keys
constexpr int kKeysItems32 = 20;       // sizing of sub-buckets without payloads: 8 * 512 x 20 = 81,920 keys at most
constexpr int kKeysItems64 = 10;       // ... 8-byte keys (the counting sort takes any size; its stage holds 74,744 half
                                       // words of 4-byte keys, 37,368 of 8-byte keys, so this is about one or two parts)
constexpr int kSlowThreads = 512;      // out-of-core sort of an oversized sub-bucket
constexpr int kSlowItems = 8;

// Where the radix index sends a key: cells of width 2^shift above `base`.
template <typename K> struct LutParams {
    K base;        // phi of the smallest splitter
    K span;        // phi(largest splitter) - base
    uint32_t shift;
    uint32_t nsplit; // number of splitters (vbuckets - 1)
};

template <typename K> struct RecordBuffers {
    K *phi[2];
    uint32_t *tag[2];
};

// Dynamic shared memory of a launch, and the most that any launch of the kernel
// takes.  A kernel's limit belongs to the device, not to the launch: it is set
// to the most each time, so that two host threads whose calls differ in size
// cannot lower it between the other's setting and launch.
struct DynSmem {
    size_t bytes, most;
    DynSmem(size_t b) : bytes(b), most(b) {}
    DynSmem(size_t b, size_t m) : bytes(b), most(m) {}
    template <typename K> cudaError_t allow(K kernel) const {
        if (most <= 48 * 1024) return cudaSuccess;
        return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
    }
};

struct Plan {
    int64_t n, p, R, s, m, M, x, q, sample_size;
    int sampling, dtype, pairs, classify;
    int dup_off;       // keys compared by value alone (no tie-break by position)
    int merge;         // final step: merge of the sorted blocks' segments (Fig. 1 step 12)
    int seg_route;     // route by the sorted blocks' partition and segment copies (Fig. 1 steps 9-11)
    int pair_words;    // pairs are routed and sorted as words phi << 32 | position
    int keep_runs;     // the block sorts keep the sorted blocks (merge or seg_route)
    uint64_t seed;
    int64_t B;         // refine: sub-buckets per bucket
    int64_t P;         // vbuckets = p * B
    int64_t Q;         // sample records between consecutive splitters (q or s)
    int64_t cap;       // keys per sub-bucket region
    int run_cl;        // cluster size of the block sort (regular sampling)
    int bucket_cl;     // cluster size of the sub-bucket sort
    int64_t tiles;     // routing tiles
    int lut_bits;      // cells of the radix index: 2^lut_bits
    int key_bytes;
    size_t ws_bytes;
};

// Device pointers into the caller's workspace (all 256-byte aligned).
struct Layout {
    DevStatus *status;
    void *sphi[2];          // sample record phi (ping-pong), key width
    uint32_t *stag[2];      // sample record tag (ping-pong)
    void *pivots;           // scratch of the sample sort
    void *vphi;             // P-1 sub-bucket splitters, phi
    uint32_t *vtag;         // P-1 sub-bucket splitters, tag
    uint16_t *lut;          // 2^lut_bits + 1 entries (sub-bucket counts fit 16 bits)
    void *lutp;             // LutParams<K>
    uint32_t *state;        // tiles * P lookback words
    uint16_t *ids;          // tiles * kRouteTile sub-bucket ids (routing scratch)
    uint32_t *cursor;       // P keys routed per sub-bucket
    uint32_t *retry_flag;   // P: the keys-only sort gave the sub-bucket back
    uint32_t *retry_list;   // P: sub-buckets for the stable cluster sort
    uint32_t *run_retry;    // R: blocks the keys-only block sort gave back
    // learned classifier (classify == BSPS_LEARNED)
    float *mlp_params;                   // 1153
    float *mlp_part;                     // partial gradients of the training CTAs
    float *mlp_x, *mlp_y;                // training points
    int64_t *mlp_npts;
    struct MlpNorm *mlp_norm;
    void *mlp_opt;                       // gradient-descent state
    struct MlpTables *mlp_tables;        // the trained network's evaluation form
    float *mlp_ysplit;                   // the network's output for every splitter
    uint16_t *ylut;                      // index over the network's output (kYCells + 1)
    void *reg_keys;         // P * cap keys (phi), region v at v*cap
    uint32_t *reg_vals;     // P * cap payloads
    uint32_t *vsize;        // P sub-bucket sizes
    uint64_t *voff;         // P + 1 exclusive offsets
    uint32_t *slow_list;    // sub-buckets too large for the on-chip sort
    // the sorted blocks and their partition (keep_runs == 1)
    void *runs;                 // n keys (phi), block k's sorted keys at k*m
    uint32_t *runs_val;         // n payloads in the same order (pairs)
    uint32_t *rs_phi, *rs_tag;  // R * s: every block's own sample records, before the sample sort
    uint32_t *part;             // (P + 1) * R: c[k][v] at v * R + k
};

struct Ctx {
    Plan pl;
    Layout ly;
    const void *keys_in;
    const uint32_t *vals_in;
    void *keys_out;
    uint32_t *vals_out;
    int64_t *bucket_sizes;
    bsps_debug dbg;
    cudaStream_t stream;
    int both_routes;     // pairs: as words, or by the look-back route if the sample's keys repeat
};

// Internal record tag: the input position g for a key, n + k*M + j for the
// pad at local index j of virtual processor k; phi of a pad is all ones.
// (pad, phi, k*M+j) order == (phi', tag') order with these encodings.

// launchers (each returns cudaSuccess or the launch error); those that serve
// a single call and a batch's calls alike are in many.cuh
cudaError_t launch_sample(const Ctx &c);          // Fig. 1 steps 3-4
cudaError_t launch_route(const Ctx &c);           // Fig. 1 steps 9-11, with payloads
cudaError_t launch_debug(const Ctx &c);           // optional diagnostics
int mlp_train_kernels();                          // kernels launch_mlp_train queues
size_t mlp_opt_bytes();

// Byte counts of dynamic shared memory (host side).
size_t route_smem_bytes(const Plan &pl);
size_t sample_scratch_bytes(const Plan &p);         // Layout::pivots
int sample_final(const Plan &p);                    // the buffer the sorted sample ends in
int sample_sort_kernels(const Plan &p);
int run_keys_cluster(const Plan &p);               // keys-only block sort for regular sampling (0: not used)
bool counting_block_sort(const Ctx &c);            // kept blocks sorted by the counting sort (and tags recovered)
// merge final step (Fig. 1 steps 9-12)
cudaError_t launch_merge_partition(const Ctx &c); // c[k][v] and the sub-bucket sizes (into cursor)
cudaError_t launch_segment_copy(const Ctx &c);    // the route as segment copies into the regions
cudaError_t launch_merge_buckets(const Ctx &c);   // gather + stable merge per bucket
int merge_cluster(const Plan &pl);                // CTAs per bucket for a bound pl.cap (0: too large)
int64_t merge_capacity(int cl);                   // keys a cluster of cl CTAs merges
int64_t merge_runs_max();                         // largest R
// Pairs whose keys repeat are not routed as words where both routes are queued:
// the device leaves the work to the one that its sample names.  Neighbours in
// the sorted sample are compared; where at least half are equal, those that are
// not count the values, and the keys repeat if there are fewer than one for 400
// keys (2^24 pairs: of 300 copies 1764 us as words and 1981 by the look-back
// route, of 3000 copies 2274 and 1375).
constexpr int kRepeatProbes = 4096;
inline uint32_t repeat_probes(const Plan &p) { return (uint32_t)imax64(0, imin64(kRepeatProbes, p.sample_size - 1)); }
inline uint32_t repeats_above(const Plan &p) {
    const int64_t q = repeat_probes(p);
    return (uint32_t)imax64(q / 2, q - (int64_t)((double)q * p.n / (400.0 * p.sample_size)));
}
constexpr int64_t kPairWordsMax = 8192;           // largest P of pairs as words (index, splitters and a chunk on chip)
constexpr int64_t kSegRouteRunsMax = 16384;       // largest R of the segment-copy route (shared memory)
size_t route_keys_smem_bytes(const Plan &pl);
bool route_keys_fine_index(const Plan &pl);           // ... and a radix index of 2^kLutBitsFine cells
bool route_keys_splitters_in_smem(const Plan &pl);  // keys-only routing holds the splitters on chip

} // namespace bsps
