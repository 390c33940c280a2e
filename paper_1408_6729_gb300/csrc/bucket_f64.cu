// bucket_f64.cu -- the final sort of float64 keys without payloads.
#include "bucket.cuh"

namespace bsps {

template cudaError_t launch_bucket_keys_t<BSPS_F64>(Exec &x);

} // namespace bsps
