// batched.cu -- many independent keys-only sorts of uneven sizes in one call
// (no counterpart in the paper; each instance is the paper's sort, Fig. 2 /
// Fig. 3, with its own parameters).
//
// Small instances run the whole method on chip, one CTA per instance
// (small.cu), in one launch per shape.  The larger ones, with random sampling,
// run the single-call kernels together: every step of the path is one launch
// for all of them (many.cuh), in waves that reuse one workspace.  With regular
// sampling they run the single-call pipeline on several streams, recorded into
// one CUDA graph that later calls with the same arguments relaunch.
#include <algorithm>
#include <cstring>
#include <mutex>
#include <vector>

#include "many.cuh"
#include "small.cuh"

namespace bsps {

constexpr int kSmallMax = BSPS_BATCH_SMALL_MAX;    // keys of an on-chip instance
constexpr int kSampleMax = BSPS_BATCH_SAMPLE_MAX;  // sample records of an on-chip instance
constexpr int kLanesMax = 16;
constexpr size_t kWaveBytes = (size_t)32 << 20;      // workspace of a wave of larger instances, per lane of the table
constexpr size_t kTableBytes = 6144;                // argument tables of one larger instance, at most

// Folds instances' device statuses into the batch's, one thread each.
__device__ void fold_status(const DevStatus *from, DevStatus *into) {
    if (from->error) set_error(into, from->error);
    if (from->overflow) atomicExch(&into->overflow, 1);
    atomicAdd(&into->timeouts, from->timeouts);
    atomicAdd(&into->slow_buckets, from->slow_buckets);
    atomicMax(&into->max_bucket, from->max_bucket);
    atomicMax(&into->max_vbucket, from->max_vbucket);
    atomicAdd(&into->mispredicted, from->mispredicted);
    atomicAdd(&into->correction_steps, from->correction_steps);
}
__global__ void merge_status_kernel(const DevStatus *from, DevStatus *into) {
    if (threadIdx.x == 0) fold_status(from, into);
}
__global__ void merge_statuses_kernel(const DevStatus *const *from, int count, DevStatus *into) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < count) fold_status(from[i], into);
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
static int size_class(int64_t n) {
    int c = 0;
    while (((int64_t)1 << c) < n) ++c;
    return c;
}

static bool valid_tune(const bsps_tune *t) {
    if (!t || t->lanes < 1 || t->lanes > kLanesMax || t->small_max_log2 > 14 || t->learned_min_log2 < 0)
        return false;
    for (int c = 0; c < BSPS_BATCH_CLASSES; ++c)
        if (t->p[c] < 1 || t->p[c] > 65535) return false;
    return true;
}

struct Instance {
    int64_t off, n;
    bsps_params prm;
    bool small;
    int S, s;
};

struct BatchPlan {
    std::vector<Instance> inst;
    std::vector<SmallJob> jobs;
    std::vector<int64_t> bbase;
    int first[4] = {0, 0, 0, 0};  // the jobs of each on-chip shape (small.cuh), in `jobs`
    size_t lane_ws = 0, jobs_bytes = 0, total = 0;
    int lanes = 1;
    // random sampling: the larger instances by wave, their workspaces' offsets
    // in the wave's and the workspace of the largest wave
    std::vector<std::vector<int32_t>> waves;
    std::vector<size_t> ws_at, ws_of;
    size_t wave_ws = 0, tables_bytes = 0;
};

static int make_batch_plan(const int64_t *h_off, int32_t num, int32_t dtype, const bsps_params *prm,
                           const bsps_tune *t, BatchPlan &bp) {
    if (num < 0 || (num > 0 && !h_off) || !prm || !valid_tune(t)) return BSPS_ERR_INVALID_ARG;
    if (dtype < BSPS_U32 || dtype > BSPS_F64) return BSPS_ERR_UNSUPPORTED_DTYPE;
    if (num > 0 && h_off[0] != 0) return BSPS_ERR_INVALID_ARG;
    // the on-chip instances run the bucket-sort path with the tie-break
    if (prm->final_step != BSPS_FINAL_SORT || prm->duplicates != BSPS_DUP_TAGS) return BSPS_ERR_INVALID_ARG;
    bp.inst.resize(num);
    bp.bbase.assign(num + 1, 0);
    bp.jobs.clear();
    bp.lanes = t->lanes;
    size_t lane_ws = 0;
    const bool grouped = prm->sampling == BSPS_RANDOM;
    bp.ws_at.assign(num, 0);
    bp.ws_of.assign(num, 0);
    size_t largest = 0, sum = 0;
    std::vector<int32_t> larger;
    for (int32_t i = 0; i < num; ++i) {
        const int64_t n = h_off[i + 1] - h_off[i];
        if (n < 0) return BSPS_ERR_INVALID_ARG;
        Instance &I = bp.inst[i];
        I.off = h_off[i];
        I.n = n;
        I.prm = *prm;
        const int c = std::min(size_class(n), BSPS_BATCH_CLASSES - 1);
        I.prm.p = t->p[c];
        I.prm.seed = prm->seed + (uint64_t)i;
        if (t->learned_min_log2 > 0 && c >= t->learned_min_log2) I.prm.classify = BSPS_LEARNED;
        bp.bbase[i + 1] = bp.bbase[i] + I.prm.p;
        bsps_plan pl;
        const int rc = bsps_get_plan(n, dtype, &I.prm, 0, &pl);
        if (rc) return rc;
        I.s = (int)pl.s;
        I.S = (int)pl.sample_size;
        I.small = c <= t->small_max_log2 && n <= kSmallMax && dtype != BSPS_F64 &&
                  I.prm.sampling == BSPS_RANDOM && I.prm.classify == BSPS_TREE && I.prm.p <= kSmallBuckets &&
                  pl.sample_size <= kSampleMax;
        if (I.small) {
            SmallJob J = {};
            J.off = I.off;
            J.bbase = bp.bbase[i];
            J.seed = I.prm.seed;
            J.n = (int32_t)n;
            J.p = I.prm.p;
            J.s = (int32_t)pl.s;
            J.S = (int32_t)pl.sample_size;
            bp.jobs.push_back(J);
        } else {
            size_t w = 0;
            const int rc2 = bsps_workspace_size(n, dtype, &I.prm, 0, &w);
            if (rc2) return rc2;
            if (!grouped) {
                lane_ws = std::max(lane_ws, w);
            } else if (n > 0) {
                bp.ws_of[i] = (w + 255) & ~size_t(255);
                largest = std::max(largest, bp.ws_of[i]);
                sum += bp.ws_of[i];
                larger.push_back(i);
            }
        }
    }
    // waves of the larger instances: as many as a workspace for `lanes` of the
    // largest holds, or for all of them up to kWaveBytes a lane
    bp.wave_ws = std::max(std::min(sum, kWaveBytes * t->lanes), largest * t->lanes);
    size_t used = 0;
    for (const int32_t i : larger) {
        if (bp.waves.empty() || used + bp.ws_of[i] > bp.wave_ws) {
            bp.waves.emplace_back();
            used = 0;
        }
        bp.waves.back().push_back(i);
        bp.ws_at[i] = used;
        used += bp.ws_of[i];
    }
    // by shape, and inside a shape the largest first
    std::stable_sort(bp.jobs.begin(), bp.jobs.end(), [](const SmallJob &a, const SmallJob &b) {
        const int x = small_size(a.n, a.S), y = small_size(b.n, b.S);
        return x != y ? x < y : a.n > b.n;
    });
    for (const SmallJob &J : bp.jobs)
        for (int size = small_size(J.n, J.S) + 1; size <= 3; ++size) ++bp.first[size];
    auto up = [](size_t v) { return (v + 255) & ~size_t(255); };
    bp.lane_ws = up(lane_ws);
    bp.jobs_bytes = up(std::max<size_t>(1, bp.jobs.size()) * sizeof(SmallJob));
    bp.tables_bytes = up(larger.size() * kTableBytes);
    bp.total = up(sizeof(DevStatus)) + bp.jobs_bytes + bp.tables_bytes + bp.wave_ws + (bp.lane_ws ? bp.lane_ws * bp.lanes : 0);
    return BSPS_OK;
}

// Streams and events the call forks into (one set per device, made once).
struct LaneSet {
    bool made = false;
    cudaStream_t origin;  // the stream a recorded call is captured from
    cudaStream_t s[kLanesMax];
    cudaEvent_t fork, join[kLanesMax];
};
static LaneSet g_lanes[64];
static std::mutex g_mu;

// The last recorded graph and what it was recorded for.
struct GraphCache {
    std::vector<unsigned char> key;
    cudaGraphExec_t exec = nullptr;
};
static GraphCache g_graph[64];

static int lanes_for_device(LaneSet *&L) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return BSPS_ERR_CUDA;
    L = &g_lanes[dev];
    if (!L->made) {
        for (int i = 0; i < kLanesMax; ++i) {
            if (cudaStreamCreateWithFlags(&L->s[i], cudaStreamNonBlocking) != cudaSuccess) return BSPS_ERR_CUDA;
            if (cudaEventCreateWithFlags(&L->join[i], cudaEventDisableTiming) != cudaSuccess) return BSPS_ERR_CUDA;
        }
        if (cudaEventCreateWithFlags(&L->fork, cudaEventDisableTiming) != cudaSuccess) return BSPS_ERR_CUDA;
        if (cudaStreamCreateWithFlags(&L->origin, cudaStreamNonBlocking) != cudaSuccess) return BSPS_ERR_CUDA;
        L->made = true;
    }
    return BSPS_OK;
}

// Everything a call with regular sampling queues, on `stream` and the lanes
// forked from it.
static int enqueue_batch(const BatchPlan &bp, const void *in, void *out, int32_t dtype, int64_t *bsz,
                         unsigned char *ws, cudaStream_t stream, LaneSet *L) {
#define BSPS_CK(call)                                    \
    do {                                                 \
        if ((call) != cudaSuccess) return BSPS_ERR_CUDA; \
    } while (0)
    DevStatus *bst = (DevStatus *)ws;
    unsigned char *lane_ws = ws + ((sizeof(DevStatus) + 255) & ~size_t(255)) + bp.jobs_bytes + bp.tables_bytes + bp.wave_ws;
    BSPS_CK(cudaMemsetAsync(bst, 0, sizeof(DevStatus), stream));
    const int nl = bp.lane_ws ? bp.lanes : 0;
    BSPS_CK(cudaEventRecord(L->fork, stream));
    for (int l = 0; l < nl; ++l) BSPS_CK(cudaStreamWaitEvent(L->s[l], L->fork, 0));
    int l = 0;
    for (size_t i = 0; i < bp.inst.size(); ++i) {
        const Instance &I = bp.inst[i];  // (with regular sampling none runs on chip)
        unsigned char *w = lane_ws + (size_t)l * bp.lane_ws;
        const size_t kb = dtype == BSPS_F64 ? 8 : 4;
        const int rc = bsps_sort_keys((const unsigned char *)in + I.off * kb, (unsigned char *)out + I.off * kb, I.n,
                                      dtype, &I.prm, bsz ? bsz + bp.bbase[i] : nullptr, w, bp.lane_ws, L->s[l]);
        if (rc) return rc;
        merge_status_kernel<<<1, 32, 0, L->s[l]>>>((const DevStatus *)w, bst);
        BSPS_CK(cudaGetLastError());
        l = (l + 1) % nl;
    }
    for (int q = 0; q < nl; ++q) {
        BSPS_CK(cudaEventRecord(L->join[q], L->s[q]));
        BSPS_CK(cudaStreamWaitEvent(stream, L->join[q], 0));
    }
    return BSPS_OK;
#undef BSPS_CK
}

// Host memory to the device, in the stream's order.  A copy from pageable memory
// of up to 64 KB has been read when the call returns and waits for nothing; a
// larger one waits for the stream's earlier work on the host (128 KB behind 50
// ms of it: 48 ms, 64 KB: 18 us), so it goes in pieces.
static cudaError_t upload(void *to, const void *from, size_t bytes, cudaStream_t stream) {
    constexpr size_t kPiece = (size_t)64 << 10;
    for (size_t at = 0; at < bytes; at += kPiece) {
        const cudaError_t e = cudaMemcpyAsync((unsigned char *)to + at, (const unsigned char *)from + at,
                                              std::min(kPiece, bytes - at), cudaMemcpyHostToDevice, stream);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

static int sm_count() {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return std::max(sms, 1);
}

// The on-chip instances; their first launch clears the batch's status.  No more
// of them than SMs: one launch, an SM and its largest CTA to each, which ends
// first (8 instances of 2^8 to 2^12 keys 23 us, with CTAs of 256 threads 30), and
// launches of several shapes would run one after the other on a mostly idle GPU
// (10 instances of 2^8 to 2^14 keys: 51 + 46 + 46 us in three).  More: a launch
// per shape, several CTAs of the smaller shapes to an SM.  Short lists of jobs go
// with the launch, longer ones are uploaded to `djobs`.
static int run_on_chip(const BatchPlan &bp, const void *in, void *out, int32_t dtype, int64_t *bsz, DevStatus *bst,
                       SmallJob *djobs, cudaStream_t stream) {
    const int njobs = (int)bp.jobs.size();
    bool uploaded = false;
    DevStatus *clear = bst;
    auto launch = [&](int size, int first, int count) {
        if (count == 0) return cudaSuccess;
        const bool listed = count <= kSmallListed;
        if (!listed && !uploaded) {
            const cudaError_t e = upload(djobs, bp.jobs.data(), sizeof(SmallJob) * njobs, stream);
            if (e != cudaSuccess) return e;
            uploaded = true;
        }
        const cudaError_t e = launch_small_jobs(dtype, size, in, out, listed ? nullptr : djobs + first, &bp.jobs[first], count, bsz,
                                                clear, stream);
        clear = nullptr;
        return e;
    };
    if (njobs <= sm_count()) return launch(2, 0, njobs) == cudaSuccess ? BSPS_OK : BSPS_ERR_CUDA;
    for (int size = 2; size >= 0; --size)  // the largest first
        if (launch(size, bp.first[size], bp.first[size + 1] - bp.first[size]) != cudaSuccess) return BSPS_ERR_CUDA;
    return BSPS_OK;
}

// The on-chip instances and, wave by wave, the larger ones in one launch per
// step (random sampling).  The argument tables are gathered first and uploaded;
// nothing is kept between calls.
static int run_grouped(const BatchPlan &bp, const void *in, void *out, int32_t dtype, int64_t *bsz, unsigned char *ws,
                       cudaStream_t stream) {
#define BSPS_CK(call)                                    \
    do {                                                 \
        if ((call) != cudaSuccess) return BSPS_ERR_CUDA; \
    } while (0)
    DevStatus *bst = (DevStatus *)ws;
    const size_t at_jobs = (sizeof(DevStatus) + 255) & ~size_t(255);
    unsigned char *tables_at = ws + at_jobs + bp.jobs_bytes, *wave_ws = tables_at + bp.tables_bytes;
    const size_t kb = dtype == BSPS_F64 ? 8 : 4;
    std::vector<unsigned char> tables;
    std::vector<std::function<cudaError_t()>> later;
    for (const auto &wave : bp.waves) {
        std::vector<Ctx> calls(wave.size());
        std::vector<const DevStatus *> statuses;
        for (size_t k = 0; k < wave.size(); ++k) {
            const int32_t i = wave[k];
            const Instance &I = bp.inst[i];
            const int rc = prepare_keys_call(calls[k], (const unsigned char *)in + I.off * kb, (unsigned char *)out + I.off * kb,
                                             I.n, dtype, &I.prm, bsz ? bsz + bp.bbase[i] : nullptr, wave_ws + bp.ws_at[i],
                                             bp.ws_of[i], stream);
            if (rc) return rc;
            statuses.push_back(calls[k].ly.status);
        }
        Exec x = {calls.data(), (int)calls.size(), stream, true, &tables, tables_at, &later};
        const int rc = run_keys_calls(x);
        if (rc) return rc;
        const size_t at = x.put(statuses);
        const int count = (int)statuses.size();
        later.push_back([=]() -> cudaError_t {
            merge_statuses_kernel<<<(count + 127) / 128, 128, 0, stream>>>((const DevStatus *const *)(tables_at + at), count, bst);
            return cudaGetLastError();
        });
    }
    if (tables.size() > bp.tables_bytes) return BSPS_ERR_WORKSPACE_TOO_SMALL;
    if (bp.jobs.empty()) {
        BSPS_CK(cudaMemsetAsync(bst, 0, sizeof(DevStatus), stream));
    } else {
        const int rc = run_on_chip(bp, in, out, dtype, bsz, bst, (SmallJob *)(ws + at_jobs), stream);
        if (rc) return rc;
    }
    BSPS_CK(upload(tables_at, tables.data(), tables.size(), stream));
    for (const auto &f : later) BSPS_CK(f());
    for (size_t i = 0; i < bp.inst.size(); ++i)  // empty instances that are not on chip
        if (bp.inst[i].n == 0 && !bp.inst[i].small && bsz)
            BSPS_CK(cudaMemsetAsync(bsz + bp.bbase[i], 0, sizeof(int64_t) * bp.inst[i].prm.p, stream));
    return BSPS_OK;
#undef BSPS_CK
}

} // namespace bsps

using namespace bsps;

extern "C" {

int bsps_tune_default(bsps_tune *t) {
    if (!t) return BSPS_ERR_INVALID_ARG;
    std::memset(t, 0, sizeof(*t));
    for (int c = 0; c < BSPS_BATCH_CLASSES; ++c) {
        if (c <= 14) t->p[c] = c <= 9 ? 1 : 4;
        else t->p[c] = (int32_t)std::min<int64_t>(4096, std::max<int64_t>(16, ((int64_t)1 << c) >> 14));
    }
    t->small_max_log2 = 14;
    t->learned_min_log2 = 0;
    t->lanes = 8;
    return BSPS_OK;
}

int bsps_batch_bucket_base(const int64_t *h_offsets, int32_t num, const bsps_tune *t, int64_t *h_base) {
    if (!h_base || num < 0 || (num > 0 && !h_offsets) || !valid_tune(t)) return BSPS_ERR_INVALID_ARG;
    h_base[0] = 0;
    for (int32_t i = 0; i < num; ++i) {
        const int64_t n = h_offsets[i + 1] - h_offsets[i];
        if (n < 0) return BSPS_ERR_INVALID_ARG;
        h_base[i + 1] = h_base[i] + t->p[std::min(size_class(n), BSPS_BATCH_CLASSES - 1)];
    }
    return BSPS_OK;
}

int bsps_batch_workspace_size(const int64_t *h_offsets, int32_t num, int32_t dtype, const bsps_params *prm,
                              const bsps_tune *t, size_t *bytes) {
    if (!bytes) return BSPS_ERR_INVALID_ARG;
    BatchPlan bp;
    const int rc = make_batch_plan(h_offsets, num, dtype, prm, t, bp);
    if (rc) return rc;
    *bytes = bp.total;
    return BSPS_OK;
}

int bsps_sort_batched(const void *d_keys_in, void *d_keys_out, const int64_t *h_offsets, int32_t num,
                      int32_t dtype, const bsps_params *prm, const bsps_tune *t, int64_t *d_bucket_sizes,
                      void *d_ws, size_t ws_bytes, void *stream) {
    BatchPlan bp;
    int rc = make_batch_plan(h_offsets, num, dtype, prm, t, bp);
    if (rc) return rc;
    if (!d_ws || ws_bytes < bp.total) return BSPS_ERR_WORKSPACE_TOO_SMALL;
    if (((uintptr_t)d_ws & 255) != 0) return BSPS_ERR_INVALID_ARG;
    const int64_t nkeys = num > 0 ? h_offsets[num] : 0;
    if (nkeys > 0 && (!d_keys_in || !d_keys_out || d_keys_in == d_keys_out)) return BSPS_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    unsigned char *ws = (unsigned char *)d_ws;
    // under a caller's capture the table upload below would become a graph
    // node reading host memory this call does not keep
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cs) != cudaSuccess) return BSPS_ERR_CUDA;
    if (cs != cudaStreamCaptureStatusNone) return BSPS_ERR_CAPTURE;
    if (prm->sampling == BSPS_RANDOM) return run_grouped(bp, d_keys_in, d_keys_out, dtype, d_bucket_sizes, ws, st);
    std::lock_guard<std::mutex> lock(g_mu);
    LaneSet *L = nullptr;
    if ((rc = lanes_for_device(L))) return rc;

    // graph key: every argument the recorded work depends on
    std::vector<unsigned char> key;
    auto put = [&](const void *p, size_t b) {
        const unsigned char *c = (const unsigned char *)p;
        key.insert(key.end(), c, c + b);
    };
    put(&d_keys_in, sizeof(void *));
    put(&d_keys_out, sizeof(void *));
    put(&d_bucket_sizes, sizeof(void *));
    put(&d_ws, sizeof(void *));
    put(&num, sizeof(num));
    put(&dtype, sizeof(dtype));
    put(prm, sizeof(*prm));
    put(t, sizeof(*t));
    if (num > 0) put(h_offsets, sizeof(int64_t) * (size_t)(num + 1));
    int dev = 0;
    cudaGetDevice(&dev);
    GraphCache &G = g_graph[dev & 63];
    if (!G.exec || G.key != key) {
        if (G.exec) cudaGraphExecDestroy(G.exec);
        G.exec = nullptr;
        G.key.clear();
        // recorded from a private stream, so that any caller stream (the
        // legacy default stream included) can launch the graph
        if (cudaStreamBeginCapture(L->origin, cudaStreamCaptureModeThreadLocal) != cudaSuccess) return BSPS_ERR_CUDA;
        rc = enqueue_batch(bp, d_keys_in, d_keys_out, dtype, d_bucket_sizes, ws, L->origin, L);
        cudaGraph_t g = nullptr;
        const cudaError_t ec = cudaStreamEndCapture(L->origin, &g);
        if (rc) {
            if (g) cudaGraphDestroy(g);
            return rc;
        }
        if (ec != cudaSuccess || !g) return BSPS_ERR_CUDA;
        const cudaError_t ei = cudaGraphInstantiate(&G.exec, g, 0);
        cudaGraphDestroy(g);
        if (ei != cudaSuccess) {
            G.exec = nullptr;
            return BSPS_ERR_CUDA;
        }
        G.key = key;
    }
    return cudaGraphLaunch(G.exec, st) == cudaSuccess ? BSPS_OK : BSPS_ERR_CUDA;
}

// ---- autotuner ----
// Batch used to time size class c: enough instances of 2^c keys to fill the
// GPU, at most 2^24 keys in all.
static int tune_count(int c) { return (int)std::max<int64_t>(4, std::min<int64_t>(256, ((int64_t)1 << 24) >> c)); }

__global__ void tune_keys_kernel(uint32_t *k, int64_t words, uint64_t seed) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i * 4 >= words) return;
    uint64_t c[4] = {(uint64_t)i, 0, 0, 0};
    philox4x64_10(c, seed, 7);
    for (int w = 0; w < 4 && i * 4 + w < words; ++w) k[i * 4 + w] = (uint32_t)c[w];
}

int bsps_autotune_workspace_size(int32_t dtype, const bsps_params *prm, int32_t max_log2, size_t *bytes) {
    if (!bytes || !prm || max_log2 < 8 || max_log2 > 24) return BSPS_ERR_INVALID_ARG;
    const size_t kb = dtype == BSPS_F64 ? 8 : 4;
    size_t need = 0;
    std::vector<int64_t> off;
    for (int c = 8; c <= max_log2; ++c) {
        const int cnt = tune_count(c);
        off.assign(cnt + 1, 0);
        for (int i = 0; i < cnt; ++i) off[i + 1] = off[i] + ((int64_t)1 << c);
        bsps_tune t;
        bsps_tune_default(&t);
        t.small_max_log2 = -1;
        for (int32_t pc : {16, 64, 256, 1024, 4096}) {
            if (((int64_t)pc << 4) > ((int64_t)1 << c)) continue;
            t.p[c] = pc;
            size_t w = 0;
            const int rc = bsps_batch_workspace_size(off.data(), cnt, dtype, prm, &t, &w);
            if (rc) return rc;
            need = std::max(need, w);
        }
    }
    size_t keys_max = 0;
    for (int c = 8; c <= max_log2; ++c) keys_max = std::max(keys_max, ((size_t)tune_count(c) << c) * kb);
    *bytes = need + 2 * ((keys_max + 255) & ~size_t(255)) + 4096;
    return BSPS_OK;
}

int bsps_autotune_batched(int32_t dtype, const bsps_params *prm, int32_t max_log2, bsps_tune *t, void *d_ws,
                          size_t ws_bytes, void *stream) {
    if (!t || !prm || max_log2 < 8 || max_log2 > 24 || t->lanes < 1 || t->lanes > kLanesMax) return BSPS_ERR_INVALID_ARG;
    size_t need = 0;
    int rc = bsps_autotune_workspace_size(dtype, prm, max_log2, &need);
    if (rc) return rc;
    if (!d_ws || ws_bytes < need) return BSPS_ERR_WORKSPACE_TOO_SMALL;
    const size_t kb = dtype == BSPS_F64 ? 8 : 4;
    cudaStream_t st = (cudaStream_t)stream;
    size_t keys_max = 0;
    for (int c = 8; c <= max_log2; ++c) keys_max = std::max(keys_max, ((size_t)tune_count(c) << c) * kb);
    keys_max = (keys_max + 255) & ~size_t(255);
    unsigned char *kin = (unsigned char *)d_ws, *kout = kin + keys_max, *bws = kout + keys_max;
    const size_t bws_bytes = ws_bytes - 2 * keys_max;
    const int64_t words = (int64_t)(keys_max / 4);
    tune_keys_kernel<<<(unsigned)((words / 4 + 255) / 256 + 1), 256, 0, st>>>((uint32_t *)kin, words, prm->seed);
    if (cudaGetLastError() != cudaSuccess) return BSPS_ERR_CUDA;
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) return BSPS_ERR_CUDA;
    const bool onchip_ok = dtype != BSPS_F64 && prm->sampling == BSPS_RANDOM;
    int small_max = -1;
    bool small_run = true;
    std::vector<int64_t> off;
    for (int c = 8; c <= max_log2; ++c) {
        const int cnt = tune_count(c);
        off.assign(cnt + 1, 0);
        for (int i = 0; i < cnt; ++i) off[i + 1] = off[i] + ((int64_t)1 << c);
        float best = 1e30f;
        int best_p = t->p[c];
        bool best_chip = false;
        for (int chip = 0; chip <= 1; ++chip) {
            if (chip && !(onchip_ok && c <= 14)) continue;
            std::vector<int32_t> cands = chip ? std::vector<int32_t>{1, 2, 4, 8, 16}
                                              : std::vector<int32_t>{16, 64, 256, 1024, 4096};
            for (int32_t pc : cands) {
                if (!chip && ((int64_t)pc << 4) > ((int64_t)1 << c)) continue;
                bsps_tune tt = *t;
                tt.p[c] = pc;
                tt.small_max_log2 = chip ? 14 : -1;
                tt.learned_min_log2 = 0;
                if (chip) {  // the on-chip form must take every instance of the class
                    bsps_plan pl;
                    bsps_params q = *prm;
                    q.p = pc;
                    if (bsps_get_plan((int64_t)1 << c, dtype, &q, 0, &pl) || pl.sample_size > kSampleMax) continue;
                }
                size_t w = 0;
                if (bsps_batch_workspace_size(off.data(), cnt, dtype, prm, &tt, &w) || w > bws_bytes) continue;
                float ms[3];
                bool ok = true;
                for (int r = -1; r < 3 && ok; ++r) {  // one untimed call first
                    if (r >= 0 && cudaEventRecord(e0, st) != cudaSuccess) ok = false;
                    if (ok && bsps_sort_batched(kin, kout, off.data(), cnt, dtype, prm, &tt, nullptr, bws, bws_bytes, st))
                        ok = false;
                    if (ok && r >= 0) {
                        if (cudaEventRecord(e1, st) != cudaSuccess || cudaEventSynchronize(e1) != cudaSuccess ||
                            cudaEventElapsedTime(&ms[r], e0, e1) != cudaSuccess)
                            ok = false;
                    }
                }
                if (!ok) continue;
                std::sort(ms, ms + 3);
                if (ms[1] < best) {
                    best = ms[1];
                    best_p = pc;
                    best_chip = chip != 0;
                }
            }
        }
        t->p[c] = best_p;
        if (small_run && best_chip) small_max = c;
        else small_run = false;
    }
    // classes below the first timed one behave like it
    for (int c = 0; c < 8; ++c) t->p[c] = small_max >= 8 ? 1 : t->p[8];
    if (small_max >= 8) small_max = std::max(small_max, 7);
    t->small_max_log2 = small_max;
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return cudaStreamSynchronize(st) == cudaSuccess ? BSPS_OK : BSPS_ERR_CUDA;
}

} // extern "C"
