// The fused CUDA-core Krylov power (stream_ga.cuh) on FP32 unfoldings, and
// its shape rules.
#include "stream_ga.cuh"

namespace ttr {

bool simt_ga_fused_ok(int64_t m, int b) { return m <= 256 && b <= 48 && ceil_div(m, 16) * ceil_div(b, 16) <= 48; }

int64_t simt_ga_partials(int64_t m, int64_t n, int b) {
  GaShape s;
  if (!ga_shape(m, n, b, &s)) return 0;
  int64_t tpc;
  int ctas;
  ga_plan(s, n, int64_t(1) << 30, &tpc, &ctas);
  return (int64_t)ctas * m * b;
}

template cudaError_t simt_ga<float>(const float*, int64_t, int64_t, const float*, int, int, float*, float*, int64_t, cudaStream_t);
template cudaError_t simt_ga_with_ctas<float>(const float*, int64_t, int64_t, const float*, int, int, float*, int64_t, float*, int64_t, cudaStream_t);

}  // namespace ttr
