// bucket_i32.cu -- the final sort of int32 keys without payloads.
#include "bucket.cuh"

namespace bsps {

template cudaError_t launch_bucket_keys_t<BSPS_I32>(Exec &x);

} // namespace bsps
