// The fused CUDA-core Krylov power (stream_ga.cuh) on BF16 unfoldings.
#include "stream_ga.cuh"

namespace ttr {

template cudaError_t simt_ga<__nv_bfloat16>(const __nv_bfloat16*, int64_t, int64_t, const float*, int, int, float*, float*, int64_t, cudaStream_t);
template cudaError_t simt_ga_with_ctas<__nv_bfloat16>(const __nv_bfloat16*, int64_t, int64_t, const float*, int, int, float*, int64_t, float*, int64_t, cudaStream_t);

}  // namespace ttr
