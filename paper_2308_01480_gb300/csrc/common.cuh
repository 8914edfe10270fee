// Shared definitions for the TT-rBKI CUDA library (sm_103a).
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include "../../include/tt_rbki.h"

namespace ttr {

// Device status word values (mirrors tt_status where they overlap).
enum : int { DEV_OK = 0, DEV_BREAKDOWN = TT_EBREAKDOWN, DEV_NONFINITE = TT_ENONFINITE };

// Record the first non-OK status (later ones do not overwrite it).
__device__ __forceinline__ void set_status(int* status, int code) {
  if (status) atomicCAS(status, DEV_OK, code);
}

// Element loads/stores for the two storage types.
__device__ __forceinline__ float ld_elem(const float* p, int64_t i) { return p[i]; }
__device__ __forceinline__ float ld_elem(const __nv_bfloat16* p, int64_t i) {
  return __bfloat162float(p[i]);
}
__device__ __forceinline__ void st_elem(float* p, int64_t i, float v) { p[i] = v; }
__device__ __forceinline__ void st_elem(__nv_bfloat16* p, int64_t i, float v) {
  p[i] = __float2bfloat16_rn(v);
}

// Four consecutive elements (p aligned to four elements).
__device__ __forceinline__ void ld4(const float* p, float (&v)[4]) {
  const float4 x = *reinterpret_cast<const float4*>(p);
  v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
}
__device__ __forceinline__ void ld4(const __nv_bfloat16* p, float (&v)[4]) {
  const uint2 x = *reinterpret_cast<const uint2*>(p);
  v[0] = __uint_as_float(x.x << 16); v[1] = __uint_as_float(x.x & 0xffff0000u);
  v[2] = __uint_as_float(x.y << 16); v[3] = __uint_as_float(x.y & 0xffff0000u);
}

__device__ __forceinline__ void st4(float* p, const float (&v)[4]) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void st4(__nv_bfloat16* p, const float (&v)[4]) {
  __nv_bfloat162 h[2] = {__floats2bfloat162_rn(v[0], v[1]), __floats2bfloat162_rn(v[2], v[3])};
  *reinterpret_cast<uint2*>(p) = *reinterpret_cast<const uint2*>(h);
}

// Elements kept as loaded and converted when used: issue is in order, so a
// conversion next to a prefetching load would wait for it there.
__device__ __forceinline__ uint32_t ld_raw(const float* p) { return __float_as_uint(*p); }
__device__ __forceinline__ uint32_t ld_raw(const __nv_bfloat16* p) {
  return *reinterpret_cast<const unsigned short*>(p);
}
template <typename T>
__device__ __forceinline__ float from_raw(uint32_t x) {
  return __uint_as_float(sizeof(T) == 2 ? x << 16 : x);
}
// Four consecutive elements, p aligned to them: 4 words (FP32) or the first 2
// of r (BF16).
__device__ __forceinline__ void ld4_raw(const float* p, uint32_t* r) {
  const uint4 x = *reinterpret_cast<const uint4*>(p);
  r[0] = x.x; r[1] = x.y; r[2] = x.z; r[3] = x.w;
}
__device__ __forceinline__ void ld4_raw(const __nv_bfloat16* p, uint32_t* r) {
  const uint2 x = *reinterpret_cast<const uint2*>(p);
  r[0] = x.x; r[1] = x.y;
}
template <typename T>
__device__ __forceinline__ float4 from_raw4(const uint32_t* r) {
  if (sizeof(T) == 2)
    return make_float4(__uint_as_float(r[0] << 16), __uint_as_float(r[0] & 0xffff0000u), __uint_as_float(r[1] << 16),
                       __uint_as_float(r[1] & 0xffff0000u));
  return make_float4(__uint_as_float(r[0]), __uint_as_float(r[1]), __uint_as_float(r[2]), __uint_as_float(r[3]));
}

// Two FP32 multiply-adds in one instruction (each rounded as fmaf).
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("{\n .reg .b64 x, y, z;\n mov.b64 x, {%2, %3};\n mov.b64 y, {%4, %5};\n mov.b64 z, {%6, %7};\n"
      " fma.rn.f32x2 z, x, y, z;\n mov.b64 {%0, %1}, z;\n}\n"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return d;
}

// Deterministic pseudo-random value in [-1, 1) from two 64-bit words (a
// SplitMix64-style finaliser), for replacing numerically vanished basis
// columns by directions that carry no information of their own.
__device__ __forceinline__ float hash_uniform(uint64_t a, uint64_t b) {
  uint64_t z = a * 0x9E3779B97F4A7C15ull + b + 0x632BE59BD9B4E019ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  z ^= z >> 31;
  return (float)(z >> 40) * (1.0f / 8388608.0f) - 1.0f;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sum over the whole CTA; `red` holds >= 32 floats of shared scratch.
// Every thread receives the total.  Contains two __syncthreads().
__device__ __forceinline__ float block_sum(float v, float* red) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int nw = (blockDim.x + 31) >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (lane == 0) red[wid] = v;
  __syncthreads();
  float t = (lane < nw) ? red[lane] : 0.f;
  return warp_sum(t);
}

// Raises a kernel's dynamic shared-memory limit, once per kernel, to the
// largest the device allows next to the kernel's static shared memory.  One
// fixed limit (rather than one per launch) keeps every launch captured in a
// CUDA graph valid however the launches of other sizes that follow set it.
cudaError_t raise_smem_limit_ptr(const void* kernel);
template <typename Kernel>
inline cudaError_t raise_smem_limit(Kernel kernel) {
  return raise_smem_limit_ptr(reinterpret_cast<const void*>(kernel));
}
// That limit in bytes (0 without a device), for the rules that decide whether
// a shape fits the kernel.
size_t dynamic_smem_limit_ptr(const void* kernel);
template <typename Kernel>
inline size_t dynamic_smem_limit(Kernel kernel) {
  return dynamic_smem_limit_ptr(reinterpret_cast<const void*>(kernel));
}

__host__ __device__ inline int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }
__host__ __device__ inline int64_t imin(int64_t a, int64_t b) { return a < b ? a : b; }
__host__ __device__ inline int64_t imax(int64_t a, int64_t b) { return a > b ? a : b; }

}  // namespace ttr
