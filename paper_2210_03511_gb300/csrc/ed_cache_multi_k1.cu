// Several-vector kernels of value kind 1 (real FP32).
#include "ed_cache_multi.cuh"

namespace ed {
template ed_status pass_multi_kind<1>(const CachePass&, bool, int, cudaStream_t);
template ed_status batch_multi_kind<1>(const BatchLaunch&, int, cudaStream_t);
}  // namespace ed
