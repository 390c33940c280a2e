// bucket_f32.cu -- the final sort of float32 keys without payloads.
#include "bucket.cuh"

namespace bsps {

template cudaError_t launch_bucket_keys_t<BSPS_F32>(Exec &x);

} // namespace bsps
