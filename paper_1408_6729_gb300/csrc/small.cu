// small.cu -- which inputs are sorted whole on chip, and their launches by key
// type; the kernels (small_sort.cuh) are compiled in a file for each type
// (small_*.cu), side by side.
#include <cstring>

#include "small_sort.cuh"

namespace bsps {

#define BSPS_SMALL(DT)                                                                                                    \
    extern template cudaError_t launch_small_keys_t<DT>(int, const void *, void *, const SmallJob *, int,                 \
                                                        const SmallList &, bool, int64_t *, DevStatus *, cudaStream_t);   \
    extern template cudaError_t launch_small_pairs_t<DT>(const Ctx &, const SmallJob &);
BSPS_SMALL(BSPS_U32)
BSPS_SMALL(BSPS_I32)
BSPS_SMALL(BSPS_F32)
#undef BSPS_SMALL

static cudaError_t launch_keys(int dtype, int size, const void *in, void *out, const SmallJob *jobs, int njobs,
                               const SmallList &list, bool batch, int64_t *bsz, DevStatus *st, cudaStream_t stream) {
    switch (dtype) {
    case BSPS_U32: return launch_small_keys_t<BSPS_U32>(size, in, out, jobs, njobs, list, batch, bsz, st, stream);
    case BSPS_I32: return launch_small_keys_t<BSPS_I32>(size, in, out, jobs, njobs, list, batch, bsz, st, stream);
    case BSPS_F32: return launch_small_keys_t<BSPS_F32>(size, in, out, jobs, njobs, list, batch, bsz, st, stream);
    default: return cudaErrorInvalidValue;
    }
}

int small_size(int64_t n, int64_t sample) {
    if (n <= small_keys(kCountSmall) && sample <= SmallKeysShape<kCountSmall>::kSample) return kCountSmall;
    if (n <= small_keys(kCountMedium) && sample <= SmallKeysShape<kCountMedium>::kSample) return kCountMedium;
    return kCountLarge;
}
static_assert(SmallKeysShape<kCountLarge>::kSample >= BSPS_BATCH_SAMPLE_MAX, "the records of a batch's instances");

cudaError_t launch_small_jobs(int dtype, int size, const void *in, void *out, const SmallJob *jobs, const SmallJob *listed,
                              int njobs, int64_t *bsz, DevStatus *clear, cudaStream_t stream) {
    SmallList list = {};
    if (!jobs) std::memcpy(list.job, listed, sizeof(SmallJob) * njobs);
    return launch_keys(dtype, size, in, out, jobs, njobs, list, true, bsz, clear, stream);
}

// The multi-kernel path's results in one launch: random sampling (with one
// bucket there are no splitters, so any sampling), the tie-break by position,
// no sub-buckets, no diagnostics asked for.
bool small_call(const Plan &p) {
    return p.n >= 1 && p.n <= BSPS_BATCH_SMALL_MAX && p.key_bytes == 4 && p.classify == BSPS_TREE && !p.dup_off && p.B == 1 &&
           (p.p == 1 || (p.sampling == BSPS_RANDOM && p.p <= kSmallBuckets && p.sample_size <= BSPS_BATCH_SAMPLE_MAX));
}

cudaError_t launch_small_call(const Ctx &c) {
    const Plan &p = c.pl;
    SmallJob J = {};
    J.seed = p.seed;
    J.n = (int32_t)p.n;
    J.p = (int32_t)p.p;
    J.s = (int32_t)imin64(p.s, INT32_MAX);
    J.S = (int32_t)imin64(p.sample_size, INT32_MAX);
    J.cap = p.cap;
    if (p.pairs) {
        switch (p.dtype) {
        case BSPS_U32: return launch_small_pairs_t<BSPS_U32>(c, J);
        case BSPS_I32: return launch_small_pairs_t<BSPS_I32>(c, J);
        default: return launch_small_pairs_t<BSPS_F32>(c, J);
        }
    }
    SmallList list = {};
    list.job[0] = J;
    return launch_keys(p.dtype, small_size(p.n, p.p > 1 ? p.sample_size : 0), c.keys_in, c.keys_out, nullptr, 1, list, false,
                       c.bucket_sizes, c.ly.status, c.stream);
}

} // namespace bsps
