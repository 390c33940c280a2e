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

// Keys a shape holds (kCountSmall, kCountMedium, kCountLarge of countsort.cuh).
constexpr int small_keys(int size) { return size == 0 ? 4096 : size == 1 ? 8192 : BSPS_BATCH_SMALL_MAX; }
int small_size(int64_t n, int64_t sample);  // the shape that takes n keys (without payloads: and that many sample records)

bool small_call(const Plan &p);
cudaError_t launch_small_call(const Ctx &c);
cudaError_t launch_small_jobs(int dtype, int size, const void *in, void *out, const SmallJob *jobs, int njobs, int64_t *bsz,
                              cudaStream_t stream);

} // namespace bsps
