// small_u32.cu -- whole sorts of uint32 keys on chip.
#include "small_sort.cuh"

namespace bsps {

template cudaError_t launch_small_keys_t<BSPS_U32>(int, const void *, void *, const SmallJob *, int, const SmallList &, bool,
                                                     int64_t *, DevStatus *, cudaStream_t);
template cudaError_t launch_small_pairs_t<BSPS_U32>(const Ctx &, const SmallJob &);

} // namespace bsps
