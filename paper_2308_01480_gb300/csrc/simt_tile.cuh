// The CUDA-core product P = A B^T over one column range, for the FP32 passes
// (sketch, Gram) and the BF16 unfoldings whose rows TMA cannot read.
//
// A (up to 8 TR rows) and B (up to TC CT rows) are both contiguous along the
// reduction, so a thread takes its operands as float4 along it: TR + TC
// 16-byte shared loads feed 4 TR TC multiply-adds.  (One scalar load per
// operand and element, 2 x VB tiles, made the passes bound by shared-memory
// instructions at an eighth of the FP32 rate.)  256 threads split into 8 row
// tiles x CT column tiles x KG = 32 / CT groups that take every KG-th group
// of four columns, so that a narrow output still occupies the CTA; the group
// sums are added in a fixed order.  Rows of the tiles are BK + 4 floats
// apart: eight lanes on eight consecutive rows hit eight different 16-byte
// banks.  The next chunk of columns is loaded into registers while the
// current one is multiplied.
#pragma once

#include "common.cuh"

namespace ttr {
namespace simt {

template <int TR_, int TC_, int CT_>
struct NtShape {
  static constexpr int TR = TR_, TC = TC_, CT = CT_;
  static constexpr int BM = 8 * TR, BN = TC * CT;
  static constexpr int KG = 32 / CT;
  static constexpr int BK = CT == 1 ? 128 : 64;
  static constexpr int KS = BK / (4 * KG);
  static constexpr int LD = BK + 4;
  static constexpr int GROUPS = CT >= 8 ? KG : 8;     // partial tiles left after the in-warp sums
  static constexpr int tile_floats(bool same) { return (BM + (same ? 0 : BN)) * LD; }
  static constexpr int smem_floats(bool same) {
    return tile_floats(same) > GROUPS * BM * BN ? tile_floats(same) : GROUPS * BM * BN;
  }
};

// ROWS x BK elements of a row-major matrix into registers: rows [0, rows)
// from A, columns [k0, kend), zero elsewhere.
template <typename T, int ROWS, int BK>
struct NtFetch {
  static constexpr int N4 = (ROWS * BK / 4 + 255) / 256;
  uint32_t r[4 * N4];
  // One pointer stepped from row to row; the step is opaque to the compiler,
  // which otherwise keeps the 16 to 32 row offsets of a tile in 64-bit
  // registers over the whole loop and spills the accumulators.
  __device__ __forceinline__ void load(const T* __restrict__ A, int64_t ld, int rows, int64_t k0, int64_t kend,
                                       bool vec) {
    if (vec) {
      constexpr int STEP = 1024 / BK;
      int64_t step = STEP * ld;
      asm volatile("" : "+l"(step));
      const int row = threadIdx.x / (BK / 4), c = (threadIdx.x % (BK / 4)) * 4;
      const bool in = k0 + c < kend;
      const T* p = A + (int64_t)row * ld + k0 + c;
#pragma unroll
      for (int u = 0; u < N4; ++u) {
#pragma unroll
        for (int t = 0; t < 4; ++t) r[4 * u + t] = 0u;
        if (in && row + u * STEP < rows) ld4_raw(p, r + 4 * u);
        p += step;
      }
    } else {
      constexpr int STEP = 256 / BK;
      int64_t step = STEP * ld;
      asm volatile("" : "+l"(step));
      const int row = threadIdx.x / BK, c = threadIdx.x % BK;
      const bool in = k0 + c < kend;
      const T* p = A + (int64_t)row * ld + k0 + c;
#pragma unroll
      for (int u = 0; u < 4 * N4; ++u) {
        r[u] = (in && row + u * STEP < rows) ? ld_raw(p) : 0u;
        p += step;
      }
    }
  }
  __device__ __forceinline__ void store(float* s, bool vec) const {
    constexpr int LD = BK + 4;
    if (vec) {
#pragma unroll
      for (int u = 0; u < N4; ++u) {
        const int e = threadIdx.x + 256 * u, row = e / (BK / 4), c = (e % (BK / 4)) * 4;
        if (row < ROWS)
          *reinterpret_cast<float4*>(s + row * LD + c) = from_raw4<T>(r + 4 * u);
      }
    } else {
#pragma unroll
      for (int u = 0; u < 4 * N4; ++u) {
        const int e = threadIdx.x + 256 * u, row = e / BK, c = e % BK;
        if (row < ROWS) s[row * LD + c] = from_raw<T>(r[u]);
      }
    }
  }
};

// acc[u][v] += sum over this thread's four-column groups of a shared tile
// pair: rows rt + RT u of As, rows ct + CT v of Bs.
template <int TR, int TC>
__device__ __forceinline__ void nt_step(float (&acc)[TR][TC], const float* a, int astep, const float* b, int bstep) {
  float4 av[TR];
#pragma unroll
  for (int u = 0; u < TR; ++u) av[u] = *reinterpret_cast<const float4*>(a + u * astep);
#pragma unroll
  for (int v = 0; v < TC; ++v) {
    const float4 bv = *reinterpret_cast<const float4*>(b + v * bstep);
#pragma unroll
    for (int u = 0; u < TR; ++u) {
      acc[u][v] = fmaf(av[u].x, bv.x, acc[u][v]);
      acc[u][v] = fmaf(av[u].y, bv.y, acc[u][v]);
      acc[u][v] = fmaf(av[u].z, bv.z, acc[u][v]);
      acc[u][v] = fmaf(av[u].w, bv.w, acc[u][v]);
    }
  }
}

// out(i, c, s): receives s = sum over columns [kbeg, kend) of A[i][k] B[c][k]
// for i < BM, c < BN (rows past rows_a / rows_b count as zero).  SAME: B is A
// (a diagonal tile of a Gram), read once.  va / vb: every row of A / B starts
// aligned to four elements and kbeg, kend are multiples of four.
template <class Sh, bool SAME, typename TA, typename TB, typename Out>
__device__ __forceinline__ void nt_tile(const TA* __restrict__ A, int64_t lda, int rows_a, const TB* __restrict__ B,
                                        int64_t ldb, int rows_b, int64_t kbeg, int64_t kend, bool va, bool vb,
                                        float* sm, Out out) {
  constexpr int TR = Sh::TR, TC = Sh::TC, CT = Sh::CT, BM = Sh::BM, BN = Sh::BN, BK = Sh::BK, LD = Sh::LD;
  float* As = sm;
  float* Bs = SAME ? sm : sm + BM * LD;
  const int tid = threadIdx.x, rt = tid & 7, q = tid >> 3, ct = q % CT, kg = q / CT;
  float acc[TR][TC];
#pragma unroll
  for (int u = 0; u < TR; ++u)
#pragma unroll
    for (int v = 0; v < TC; ++v) acc[u][v] = 0.f;
  NtFetch<TA, BM, BK> fa;
  NtFetch<TB, SAME ? 4 : BN, BK> fb;
  if (kbeg < kend) {
    fa.load(A, lda, rows_a, kbeg, kend, va);
    if constexpr (!SAME) fb.load(B, ldb, rows_b, kbeg, kend, vb);
  }
  for (int64_t k0 = kbeg; k0 < kend; k0 += BK) {
    __syncthreads();
    fa.store(As, va);
    if constexpr (!SAME) fb.store(Bs, vb);
    __syncthreads();
    if (k0 + BK < kend) {
      fa.load(A, lda, rows_a, k0 + BK, kend, va);
      if constexpr (!SAME) fb.load(B, ldb, rows_b, k0 + BK, kend, vb);
    }
#pragma unroll 1
    for (int s = 0; s < Sh::KS; ++s) {
      const int k4 = 4 * (kg + s * Sh::KG);
      nt_step<TR, TC>(acc, As + rt * LD + k4, 8 * LD, Bs + ct * LD + k4, CT * LD);
    }
  }
  // groups that share a warp are added by shuffles, the rest through shared memory
  if constexpr (CT <= 2) {
#pragma unroll
    for (int u = 0; u < TR; ++u)
#pragma unroll
      for (int v = 0; v < TC; ++v) {
        if constexpr (CT == 1) acc[u][v] += __shfl_xor_sync(0xffffffffu, acc[u][v], 8);
        acc[u][v] += __shfl_xor_sync(0xffffffffu, acc[u][v], 16);
      }
  }
  __syncthreads();
  const int g = CT >= 8 ? kg : (tid >> 5);
  const bool owner = CT >= 4 || (CT == 2 && !(tid & 16)) || (CT == 1 && !(tid & 24));
  if (owner) {
#pragma unroll
    for (int u = 0; u < TR; ++u)
#pragma unroll
      for (int v = 0; v < TC; ++v) sm[(g * BM + rt + 8 * u) * BN + ct + CT * v] = acc[u][v];
  }
  __syncthreads();
  for (int e = tid; e < BM * BN; e += 256) {
    float s = 0.f;
#pragma unroll
    for (int x = 0; x < Sh::GROUPS; ++x) s += sm[x * BM * BN + e];
    out(e / BN, e % BN, s);
  }
}

// Every row of a row-major matrix with this row length and base starts
// aligned to four elements.
template <typename T>
inline bool rows_aligned4(const T* A, int64_t ld) {
  return ld % 4 == 0 && reinterpret_cast<uintptr_t>(A) % (4 * sizeof(T)) == 0;
}

}  // namespace simt
}  // namespace ttr
