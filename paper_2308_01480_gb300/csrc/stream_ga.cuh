// CUDA-core fused Krylov power Y = C (C^T X) for m <= 256, b <= 48 (Alg. 3
// step 4): the FP32 form, and BF16 unfoldings the tensor cores do not take.
//
// Each column tile of C is read from memory once, into shared memory, and
// used by both products:
//   1  T = C_tile^T X: a lane owns two columns (one of a 32-column tile), a
//      warp TC1 columns of X (one of CG1 groups) and every RS-th row; the RS
//      partial tiles are added in order.  X is read as broadcasts.
//   2  Z += C_tile T^T as rows times rows (simt_tile.cuh): TR x TC register
//      tiles fed by 16-byte loads along the tile's columns, RT row tiles x
//      CT column tiles x KG groups of columns, kept in registers over all of
//      the CTA's tiles; the group sums are added in order at the end.
// Both phases do four or more multiply-adds per shared-memory instruction;
// the tile's width (128 columns, 64 above 128 rows) leaves room for two or
// more CTAs an SM, so that one CTA's loads overlap another's products.  A tile
// is a long chain for one CTA: unfoldings of up to 2,048 columns take tiles of
// 32 (120 x 504 at b = 45 24.4 -> 14.7), and above 128 rows and 12 columns of
// X also where 64 leave SMs without one (n < 9,728; 256 x 4,096 at b = 32
// 31.9 -> 18.9).  Wider tiles have fewer partials to add.
// Before, both products loaded their operands as scalars (one per 1 to 2
// multiply-adds for narrow blocks).  Measured (FP32, us): 45 x 4,100,625 at
// b = 6 1,230 -> 287 (738 MB, 2.6 TB/s; BF16, rows not aligned, 1,178 ->
// 287), 180 x 91,125 at b = 6 101 -> 31, 256 x 32,768 at b = 13 54 -> 29.
#pragma once

#include "cluster_la.cuh"
#include "common.cuh"
#include "kernels.h"
#include "simt_tile.cuh"

namespace ttr {

// Launch shape of one power.
struct GaShape {
  int rt, tr;       // row tiles per CTA, rows per tile: rt tr >= m
  int tc, ct;       // columns per tile, column tiles: tc ct >= b
  int tn;           // columns of C per tile
  int tc1, cg1;     // phase 1: columns of X per warp, groups
  int cw, rs;       // phase 1: warps across the tile's columns, row splits
  int kg;           // phase 2: groups over the tile's columns
  int mp, bp1, bn, ld;
  int ls;           // row stride of the group sums
  size_t off_x, off_t, off_p, smem;   // floats, floats, floats, bytes
};

inline bool ga_shape(int64_t m, int64_t n, int b, GaShape* s) {
  if (m < 1 || m > 256 || b < 1 || b > 48) return false;
  s->rt = m <= 64 ? 8 : m <= 128 ? 16 : 32;
  const bool tiny = n <= 2048;
  s->tr = tiny ? 8 : m <= 32 ? 4 : m <= 48 ? 6 : 8;
  s->tn = tiny ? 32 : m <= 128 ? 128 : b <= 12 || ceil_div(n, 64) >= 152 ? 64 : 32;
  if (b <= 4) { s->tc = 4; s->ct = 1; s->tc1 = 4; s->cg1 = 1; }
  else if (b <= 6) { s->tc = 6; s->ct = 1; s->tc1 = 8; s->cg1 = 1; }
  else if (b <= 8) { s->tc = 8; s->ct = 1; s->tc1 = 8; s->cg1 = 1; }
  else if (b <= 12) { s->tc = 6; s->ct = 2; s->tc1 = 12; s->cg1 = 1; }
  else if (b <= 16) { s->tc = 8; s->ct = 2; s->tc1 = 8; s->cg1 = 2; }
  else if (b <= 24) { s->tc = 6; s->ct = 4; s->tc1 = 12; s->cg1 = 2; }
  else if (b <= 32) { s->tc = 8; s->ct = 4; s->tc1 = 8; s->cg1 = 4; }
  else { s->tc = 6; s->ct = 8; s->tc1 = 12; s->cg1 = 4; }
  s->cw = s->tn >= 64 ? s->tn / 64 : 1;
  s->rs = 8 / (s->cw * s->cg1);
  s->kg = (int)imin(256 / (s->rt * s->ct), s->tn / 4);
  s->mp = s->rt * s->tr;
  s->bp1 = s->tc1 * s->cg1;
  s->bn = s->tc * s->ct;
  s->ld = s->tn + 4;
  s->off_x = (size_t)s->mp * s->ld;
  s->off_t = s->off_x + (size_t)((m + 3) / 4 * 4) * s->bp1;
  s->off_p = s->off_t + (size_t)s->bn * s->ld;
  const size_t tiles = s->off_p + (s->rs > 1 ? (size_t)s->rs * s->bp1 * s->tn : 0);
  // lanes hold consecutive rows: an odd stride keeps their stores in different
  // banks (a stride of bn = 32 made them take turns: 256 x 4,096 at b = 32
  // 35 us, so 28 with tiles of 64)
  s->ls = s->bn | 1;
  const size_t sums = (size_t)s->kg * s->mp * s->ls;
  s->smem = sizeof(float) * (tiles > sums ? tiles : sums);
  return true;
}

namespace {

// K elements a thread of a column tile of C (256 K / TN rows), all loads in
// flight together; rows are stepped by pointer.
template <typename T, int TN, int K>
struct GaLoad {
  static constexpr int rows = 256 * K / TN;
  uint32_t r[K];
  __device__ __forceinline__ void load(const T* __restrict__ C, int64_t n, int m, int wv, bool vec) {
    if (vec) {
      constexpr int STEP = 1024 / TN;
      const int row = threadIdx.x / (TN / 4), c = (threadIdx.x % (TN / 4)) * 4;
      const T* p = C + (int64_t)row * n + c;
      int64_t step = STEP * n;
      asm volatile("" : "+l"(step));       // no row offsets kept in registers
#pragma unroll
      for (int u = 0; u < K / 4; ++u) {
#pragma unroll
        for (int t = 0; t < 4; ++t) r[4 * u + t] = 0u;
        if (c < wv && row + u * STEP < m) ld4_raw(p, r + 4 * u);
        p += step;
      }
    } else {
      constexpr int STEP = 256 / TN;
      const int row = threadIdx.x / TN, c = threadIdx.x % TN;
      const T* p = C + (int64_t)row * n + c;
      int64_t step = STEP * n;
      asm volatile("" : "+l"(step));
#pragma unroll
      for (int u = 0; u < K; ++u) {
        r[u] = (c < wv && row + u * STEP < m) ? ld_raw(p) : 0u;
        p += step;
      }
    }
  }
  __device__ __forceinline__ void store(float* Cs, int m, bool vec) const {
    constexpr int LD = TN + 4;
    if (vec) {
      constexpr int STEP = 1024 / TN;
      const int row = threadIdx.x / (TN / 4), c = (threadIdx.x % (TN / 4)) * 4;
#pragma unroll
      for (int u = 0; u < K / 4; ++u)
        if (row + u * STEP < m)
          *reinterpret_cast<float4*>(Cs + (row + u * STEP) * LD + c) = from_raw4<T>(r + 4 * u);
    } else {
      constexpr int STEP = 256 / TN;
      const int row = threadIdx.x / TN, c = threadIdx.x % TN;
#pragma unroll
      for (int u = 0; u < K; ++u)
        if (row + u * STEP < m) Cs[(row + u * STEP) * LD + c] = from_raw<T>(r[u]);
    }
  }
};

// The m x wv column tile of an FP32 C with aligned rows straight to shared
// memory, every copy in flight (columns past wv become zero).  Element by
// element (rows not aligned) this was slower than loads in parts.
template <int TN>
__device__ __forceinline__ void ga_copy_async(float* Cs, const float* __restrict__ C, int64_t n, int m, int wv) {
  constexpr int LD = TN + 4, PER = TN / 4;
  const int c = (threadIdx.x % PER) * 4;
  const bool in = c < wv;                   // all four or none: n is a multiple of four
  for (int row = threadIdx.x / PER; row < m; row += 256 / PER)
    cp_async16z(Cs + row * LD + c, in ? C + (int64_t)row * n + c : C, in);
}

// PF > 0: the whole next tile (PF elements a thread) is loaded into registers
// while the current one is multiplied; 0: copied asynchronously (FP32, rows
// aligned) or loaded in parts of 16 elements.
template <typename TIn, int TR, int TC, int TC1, int TN, int PF>
__global__ void __launch_bounds__(256, 2) k_ga(const TIn* __restrict__ C, int64_t m64, int64_t n,
                                               const float* __restrict__ X, int ldx, int b, float* __restrict__ P,
                                               int64_t tiles_per_cta, const __grid_constant__ GaShape p, bool vec) {
  extern __shared__ __align__(16) float ga_sm[];
  float* Cs = ga_sm;
  float* Xs = ga_sm + p.off_x;
  float* Ts = ga_sm + p.off_t;
  float* Tp = ga_sm + p.off_p;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  constexpr int LD = TN + 4;
  const int m = (int)m64, BP1 = p.bp1;
  // X, all copies in flight beside the first tile's
  {
    const int dr = 256 / BP1, dc = 256 - dr * BP1;
    int r = tid / BP1, c = tid - r * BP1;
    for (int e = tid; e < m * BP1; e += 256) {
      const bool in = c < b;
      cp_async4(Xs + e, in ? X + (int64_t)r * ldx + c : X, in);
      r += dr;
      c += dc;
      if (c >= BP1) {
        c -= BP1;
        ++r;
      }
    }
  }
  for (int e = tid; e < (p.mp - m) * LD; e += 256) Cs[m * LD + e] = 0.f;
  for (int e = tid; e < p.bn * LD; e += 256) Ts[e] = 0.f;
  // phase 1: columns lane and lane + 32 of the warp's 64, rows rs0, rs0 + RS, ...
  const int cw = w % p.cw, cg = (w / p.cw) % p.cg1, rs0 = w / (p.cw * p.cg1);
  // phase 2
  const int rt = tid % p.rt, q = tid / p.rt, ct = q % p.ct, kg = q / p.ct;
  float acc[TR][TC];
#pragma unroll
  for (int u = 0; u < TR; ++u)
#pragma unroll
    for (int v = 0; v < TC; ++v) acc[u][v] = 0.f;
  const int64_t ntiles = ceil_div(n, TN);
  const int64_t t_beg = (int64_t)blockIdx.x * tiles_per_cta, t_end = imin(ntiles, t_beg + tiles_per_cta);
  const int ks = TN / (4 * p.kg);
  GaLoad<TIn, TN, PF ? PF : 16> ld;
  if constexpr (PF > 0) {
    if (t_beg < t_end) ld.load(C + t_beg * TN, n, m, (int)imin(TN, n - t_beg * TN), vec);
  }
  for (int64_t tile = t_beg; tile < t_end; ++tile) {
    const int64_t c0 = tile * TN;
    const int wv = (int)imin(TN, n - c0);     // columns of this tile
    __syncthreads();
    if constexpr (PF > 0) {
      ld.store(Cs, m, vec);
    } else if (sizeof(TIn) == 4 && vec) {
      ga_copy_async<TN>(Cs, reinterpret_cast<const float*>(C) + c0, n, m, wv);
    } else {
      GaLoad<TIn, TN, 16> part;
      for (int r0 = 0; r0 < m; r0 += GaLoad<TIn, TN, 16>::rows) {
        part.load(C + (int64_t)r0 * n + c0, n, m - r0, wv, vec);
        part.store(Cs + r0 * LD, m - r0, vec);
      }
    }
    cp_async_wait_all();                    // the tile's copies, and X's before the first
    __syncthreads();
    if constexpr (PF > 0) {
      if (tile + 1 < t_end) ld.load(C + c0 + TN, n, m, (int)imin(TN, n - c0 - TN), vec);
    }
    {
      constexpr bool kTwo = TN >= 64;          // columns of a lane
      float t0[TC1], t1[TC1];
#pragma unroll
      for (int c = 0; c < TC1; ++c) t0[c] = t1[c] = 0.f;
      const float* cc = Cs + rs0 * LD + cw * 64 + lane;
      const float* xx = Xs + rs0 * BP1 + cg * TC1;
      const int cstep = p.rs * LD, xstep = p.rs * BP1;
#pragma unroll 4
      for (int i = rs0; i < m; i += p.rs, cc += cstep, xx += xstep) {
        const float a0 = cc[0], a1 = kTwo ? cc[32] : 0.f;
#pragma unroll
        for (int c4 = 0; c4 < TC1 / 4; ++c4) {
          const float4 x = *reinterpret_cast<const float4*>(xx + 4 * c4);
          t0[4 * c4] = fmaf(a0, x.x, t0[4 * c4]);
          t0[4 * c4 + 1] = fmaf(a0, x.y, t0[4 * c4 + 1]);
          t0[4 * c4 + 2] = fmaf(a0, x.z, t0[4 * c4 + 2]);
          t0[4 * c4 + 3] = fmaf(a0, x.w, t0[4 * c4 + 3]);
          if constexpr (kTwo) {
            t1[4 * c4] = fmaf(a1, x.x, t1[4 * c4]);
            t1[4 * c4 + 1] = fmaf(a1, x.y, t1[4 * c4 + 1]);
            t1[4 * c4 + 2] = fmaf(a1, x.z, t1[4 * c4 + 2]);
            t1[4 * c4 + 3] = fmaf(a1, x.w, t1[4 * c4 + 3]);
          }
        }
      }
      if (p.rs > 1) {
        float* tp = Tp + (size_t)rs0 * BP1 * TN + cw * 64 + lane;
#pragma unroll
        for (int c = 0; c < TC1; ++c) {
          tp[(cg * TC1 + c) * TN] = t0[c];
          if constexpr (kTwo) tp[(cg * TC1 + c) * TN + 32] = t1[c];
        }
        __syncthreads();
        for (int e = tid; e < b * TN; e += 256) {
          float s = 0.f;
          for (int x = 0; x < p.rs; ++x) s += Tp[(size_t)x * BP1 * TN + e];
          const int c = e / TN;
          Ts[c * LD + (e - c * TN)] = s;
        }
      } else {
#pragma unroll
        for (int c = 0; c < TC1; ++c)
          if (cg * TC1 + c < b) {
            Ts[(cg * TC1 + c) * LD + cw * 64 + lane] = t0[c];
            if constexpr (kTwo) Ts[(cg * TC1 + c) * LD + cw * 64 + lane + 32] = t1[c];
          }
      }
    }
    __syncthreads();
    if (kg < p.kg) {                        // a short tile has fewer groups than the CTA
      for (int s = 0; s < ks; ++s) {
        const int k4 = 4 * (kg + s * p.kg);
        simt::nt_step<TR, TC>(acc, Cs + rt * LD + k4, p.rt * LD, Ts + ct * LD + k4, p.ct * LD);
      }
    }
  }
  // group sums in group order
  __syncthreads();
  if (kg < p.kg) {
#pragma unroll
    for (int u = 0; u < TR; ++u)
#pragma unroll
      for (int v = 0; v < TC; ++v)
        ga_sm[((size_t)kg * p.mp + rt + p.rt * u) * p.ls + ct + p.ct * v] = acc[u][v];
  }
  __syncthreads();
  float* out = P + (int64_t)blockIdx.x * m * b;
  for (int e = tid; e < m * b; e += 256) {
    const int i = e / b, c = e - i * b;
    float s = 0.f;
    for (int g = 0; g < p.kg; ++g) s += ga_sm[((size_t)g * p.mp + i) * p.ls + c];
    out[e] = s;
  }
}

template <typename TIn, int TR, int TC, int TC1, int TN, int PF>
cudaError_t ga_launch(const TIn* C, int64_t m, int64_t n, const float* X, int ldx, int b, float* P, int64_t tpc,
                      int ctas, const GaShape& s, cudaStream_t st) {
  const cudaError_t e = raise_smem_limit(k_ga<TIn, TR, TC, TC1, TN, PF>);
  if (e != cudaSuccess) return e;
  k_ga<TIn, TR, TC, TC1, TN, PF><<<ctas, 256, s.smem, st>>>(C, m, n, X, ldx, b, P, tpc, s, simt::rows_aligned4(C, n));
  return cudaGetLastError();
}

template <typename TIn, int TR, int TN, int PF>
cudaError_t ga_dispatch(const TIn* C, int64_t m, int64_t n, const float* X, int ldx, int b, float* P, int64_t tpc,
                        int ctas, const GaShape& s, cudaStream_t st) {
#define TTR_GA(TC, TC1) if (s.tc == TC && s.tc1 == TC1) return ga_launch<TIn, TR, TC, TC1, TN, PF>(C, m, n, X, ldx, b, P, tpc, ctas, s, st)
  TTR_GA(4, 4);
  TTR_GA(6, 8);
  TTR_GA(8, 8);
  TTR_GA(6, 12);
#undef TTR_GA
  return cudaErrorInvalidValue;
}

// CTAs of a power: what the chip holds at once, each over one contiguous
// range of tiles.
inline void ga_plan(const GaShape& s, int64_t n, int64_t max_ctas, int64_t* tpc, int* ctas) {
  const int64_t tiles = ceil_div(n, s.tn);
  const int64_t per_sm = s.smem <= 112 * 1024 ? 2 : 1;
  const int64_t want = imin(imin(tiles, per_sm * 152), max_ctas);
  *tpc = ceil_div(tiles, want);
  *ctas = (int)ceil_div(tiles, *tpc);
}

}  // namespace

template <typename TIn>
cudaError_t simt_ga_with_ctas(const TIn* C, int64_t m, int64_t n, const float* X, int ldx, int b,
                              float* partials, int64_t max_ctas, float* out, int64_t ldo, cudaStream_t st) {
  GaShape s;
  if (max_ctas < 1 || !ga_shape(m, n, b, &s)) return cudaErrorInvalidValue;
  int64_t tpc;
  int ctas;
  ga_plan(s, n, max_ctas, &tpc, &ctas);
  {
    ProfScope prof("gram_apply_simt", st, (double)m * n * sizeof(TIn) + (double)m * b * 4, 4.0 * m * n * b);
    note_launch("gram_apply_simt");
    const cudaError_t e = s.tn == 32    ? ga_dispatch<TIn, 8, 32, 0>(C, m, n, X, ldx, b, partials, tpc, ctas, s, st)
                          : s.tr == 4   ? ga_dispatch<TIn, 4, 128, 16>(C, m, n, X, ldx, b, partials, tpc, ctas, s, st)
                          : s.tr == 6   ? ga_dispatch<TIn, 6, 128, 24>(C, m, n, X, ldx, b, partials, tpc, ctas, s, st)
                          : s.rt == 8   ? ga_dispatch<TIn, 8, 128, 32>(C, m, n, X, ldx, b, partials, tpc, ctas, s, st)
                          : s.tn == 128 ? ga_dispatch<TIn, 8, 128, 0>(C, m, n, X, ldx, b, partials, tpc, ctas, s, st)
                                        : ga_dispatch<TIn, 8, 64, 0>(C, m, n, X, ldx, b, partials, tpc, ctas, s, st);
    if (e != cudaSuccess) return e;
  }
  return launch_reduce_partials(partials, ctas, m, b, out, ldo, st);
}

template <typename TIn>
cudaError_t simt_ga(const TIn* C, int64_t m, int64_t n, const float* X, int ldx, int b,
                    float* partials, float* out, int64_t ldo, cudaStream_t st) {
  return simt_ga_with_ctas(C, m, n, X, ldx, b, partials, int64_t(1) << 30, out, ldo, st);
}

}  // namespace ttr
