// bucket_u32.cu -- the final sort of uint32 keys without payloads.
#include "bucket.cuh"

namespace bsps {

template cudaError_t launch_bucket_keys_t<BSPS_U32>(Exec &x);

} // namespace bsps
