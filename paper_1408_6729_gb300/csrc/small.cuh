// small.cuh -- whole sorts on chip (small.cu).
#pragma once

#include "kernels.cuh"

namespace bsps {

constexpr int kSmallBuckets = 256;  // buckets of an on-chip sort

struct SmallJob {
    int64_t off;         // first key
    int64_t bbase;       // first bucket-size entry
    uint64_t seed;
    int64_t cap;         // keys a bucket may hold (single calls)
    int32_t n, p, s, S;  // keys, buckets, samples per bucket, sample records (s*p - 1)
};

// Jobs given to the launch itself, and the size of such a list (more are read
// from device memory).
constexpr int kSmallListed = 32;
struct SmallList {
    SmallJob job[kSmallListed];
};

// Keys a shape holds (kCountSmall, kCountMedium, kCountLarge of countsort.cuh).
constexpr int small_keys(int size) { return size == 0 ? 4096 : size == 1 ? 8192 : BSPS_BATCH_SMALL_MAX; }
int small_size(int64_t n, int64_t sample);  // the shape that takes n keys (without payloads: and that many sample records)

bool small_call(const Plan &p);
cudaError_t launch_small_call(const Ctx &c);
// njobs jobs of a batch, at `jobs` in device memory or (null) from `listed`;
// the batch's status block, if given, is cleared.
cudaError_t launch_small_jobs(int dtype, int size, const void *in, void *out, const SmallJob *jobs, const SmallJob *listed,
                              int njobs, int64_t *bsz, DevStatus *clear, cudaStream_t stream);

} // namespace bsps
