// bucket.cu -- the final sort of every bucket by key type (bucket.cuh); the
// kernels of keys alone are compiled in a file for each type (bucket_*.cu),
// side by side.
#include "bucket.cuh"

namespace bsps {

extern template cudaError_t launch_bucket_keys_t<BSPS_U32>(Exec &x);
extern template cudaError_t launch_bucket_keys_t<BSPS_I32>(Exec &x);
extern template cudaError_t launch_bucket_keys_t<BSPS_F32>(Exec &x);
extern template cudaError_t launch_bucket_keys_t<BSPS_F64>(Exec &x);

cudaError_t launch_bucket_keys(Exec &x) {
    switch (x.calls[0].pl.dtype) {
    case BSPS_U32: return launch_bucket_keys_t<BSPS_U32>(x);
    case BSPS_I32: return launch_bucket_keys_t<BSPS_I32>(x);
    case BSPS_F32: return launch_bucket_keys_t<BSPS_F32>(x);
    default: return launch_bucket_keys_t<BSPS_F64>(x);
    }
}

template <int DT> static cudaError_t launch_pairs_cluster(Exec &x) {
    constexpr int IT = sizeof(typename KeyTraits<DT>::T) == 8 ? kPairItems64 : kPairItems32;
    switch (x.calls[0].pl.bucket_cl) {
    case 1: return launch_cluster<DT, true, 1, IT>(x);
    case 2: return launch_cluster<DT, true, 2, IT>(x);
    case 4: return launch_cluster<DT, true, 4, IT>(x);
    case 8: return launch_cluster<DT, true, 8, IT>(x);
    default: return cudaErrorInvalidValue;
    }
}

template <int DT> static cudaError_t launch_bucket_pairs_t(Exec &x) {
    using K = typename KeyTraits<DT>::T;
    const Ctx &c = x.calls[0];
    BucketArgs<K> a;
    bucket_args<DT>(c, a);
    // one-value sub-buckets are copied; the cluster sort takes the list of the others
    bucket_copy_kernel<DT, true><<<(unsigned)imin64(c.pl.P, 4 * (int64_t)sm_count()), kCopyThreads, 0, c.stream>>>(
        a, c.ly.retry_list, &c.ly.status->retry_count);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    e = launch_pairs_cluster<DT>(x);
    return e != cudaSuccess ? e : launch_slow<DT, true>(x);
}

cudaError_t launch_bucket_pairs(Exec &x) {
    switch (x.calls[0].pl.dtype) {
    case BSPS_U32: return launch_bucket_pairs_t<BSPS_U32>(x);
    case BSPS_I32: return launch_bucket_pairs_t<BSPS_I32>(x);
    case BSPS_F32: return launch_bucket_pairs_t<BSPS_F32>(x);
    default: return launch_bucket_pairs_t<BSPS_F64>(x);
    }
}

// The stable cluster sort alone, of the sub-buckets that pairs.cu lists when the
// keys repeat.
cudaError_t launch_repeats_cluster(Exec &x) {
    switch (x.calls[0].pl.dtype) {
    case BSPS_U32: return launch_pairs_cluster<BSPS_U32>(x);
    case BSPS_I32: return launch_pairs_cluster<BSPS_I32>(x);
    case BSPS_F32: return launch_pairs_cluster<BSPS_F32>(x);
    default: return cudaErrorInvalidValue;
    }
}

} // namespace bsps
