// CUDA-core projection S = X^T C (Alg. 3 step 10, and the first half of a
// Krylov power for tall unfoldings): the FP32 form, and BF16 unfoldings the
// tensor-core pass does not take.
//
// Every column of C is one column of S, so a thread keeps four whole
// columns (TC sums of each) in registers and reads C straight from global
// memory, coalesced along the row: C needs no shared memory and no barrier.
// X is the small operand: chunks of 16 rows are double-buffered in shared
// memory by each row group for itself (a barrier over the CTA per chunk held
// up the others) and read as broadcasts, one 16-byte load for 16
// multiply-adds, two to an instruction.  The next rows of C (16 to 32 elements
// a thread) are in flight while the current ones are multiplied.
// The eight warps of a CTA split into CG groups of output rows (b > 20), RG
// groups of rows of C (few columns: the groups' sums are added in order) and
// the rest over columns; when even that leaves the chip idle (n below
// 128 x 152 columns), the rows are also split over the grid and a second
// kernel adds the partials in split order.  Few rows of wide or short
// unfoldings take tiles of 64 columns with both operands in shared memory
// (k_proj_tile).
// Measured (FP32, us; before: 16 x 16 threads with both operands staged in
// shared memory and no split over rows unless n <= 512): 7680 x 2048 at
// b = 20 404 -> 25, 800 x 64,000 at b = 20 190 -> 87, 45 x 4,100,625 at
// b = 6 640 -> 208 (3.5 TB/s); BF16 715 -> 200.  What bounds it now is
// latency at one to two CTAs an SM.
#include "cluster_la.cuh"
#include "common.cuh"
#include "kernels.h"

namespace ttr {

namespace {

constexpr int PJ_RK = 16;   // rows of X per shared-memory chunk of a row group
constexpr int PJ_NC = 4;    // columns of C per thread

// VEC: every row of C (and of S) starts aligned to four elements, and the
// thread's columns are neighbours; otherwise they are 32 apart.  x16: rows
// of X are 16-byte aligned and b is a multiple of four.
template <typename TIn, typename TOut, int TC, int FR, int CTAS, bool VEC>
__global__ void __launch_bounds__(256, CTAS) k_proj(const TIn* __restrict__ C, int64_t m, int64_t n,
                                                    const float* __restrict__ X, int ldx, int b,
                                                    TOut* __restrict__ S, int64_t lds, int64_t rows_per,
                                                    int64_t split_stride, int CG, int RG, bool x16) {
  constexpr int NC = PJ_NC;
  extern __shared__ __align__(16) float pj_sm[];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int CW = 8 / (CG * RG);
  const int cw = w % CW, cg = (w / CW) % CG, rg = w / (CW * CG);
  const int BP = CG * TC;
  const int64_t col = (int64_t)blockIdx.x * (CW * 32 * NC) + cw * (32 * NC) + (VEC ? NC * lane : lane);
  S += (int64_t)blockIdx.y * split_stride;
  // this row group's rows [g0, g1) and its two chunk buffers; only the
  // group's warps synchronise
  const int64_t rbeg = (int64_t)blockIdx.y * rows_per, rend = imin(m, rbeg + rows_per);
  const int64_t gr = ceil_div(rend - rbeg, RG), g0 = rbeg + rg * gr, g1 = imin(rend, g0 + gr);
  const int nchunk = g0 < g1 ? (int)ceil_div(g1 - g0, PJ_RK) : 0;
  const int gt = 256 / RG;                      // threads of one group
  const int t = tid % gt;
  float* xbuf = pj_sm + (size_t)rg * 2 * PJ_RK * BP;
  auto group_sync = [&]() {
    if (gt == 32) __syncwarp();
    else asm volatile("bar.sync %0, %1;\n" ::"r"(1 + rg), "r"(gt) : "memory");
  };
  bool in[NC];
#pragma unroll
  for (int u = 0; u < NC; ++u) in[u] = VEC ? col < n : col + 32 * u < n;   // VEC: all four or none
  auto stage = [&](int ch) {
    float* xs = xbuf + (ch & 1) * PJ_RK * BP;
    const int64_t i0 = g0 + (int64_t)ch * PJ_RK;
    if (x16) {
      const int q = BP / 4;
      for (int e = t; e < PJ_RK * q; e += gt) {
        const int r = e / q, c = (e - r * q) * 4;
        const bool ok = i0 + r < g1 && c < b;
        cp_async16z(xs + 4 * e, ok ? X + (i0 + r) * ldx + c : X, ok);
      }
    } else {
      for (int e = t; e < PJ_RK * BP; e += gt) {
        const int r = e / BP, c = e - r * BP;
        const bool ok = i0 + r < g1 && c < b;
        cp_async4(xs + e, ok ? X + (i0 + r) * ldx + c : X, ok);
      }
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  auto fetch = [&](uint32_t (&v)[FR][NC], int64_t i0) {
    const TIn* p = C + i0 * n + col;
    const int left = (int)imin(FR, g1 - i0);
#pragma unroll
    for (int r = 0; r < FR; ++r) {
#pragma unroll
      for (int u = 0; u < NC; ++u) v[r][u] = 0u;
      if constexpr (VEC) {
        if (r < left && in[0]) ld4_raw(p, v[r]);
      } else {
#pragma unroll
        for (int u = 0; u < NC; ++u)
          if (r < left && in[u]) v[r][u] = ld_raw(p + 32 * u);
      }
      p += n;
    }
  };
  float2 acc[NC][TC / 2];
#pragma unroll
  for (int u = 0; u < NC; ++u)
#pragma unroll
    for (int c = 0; c < TC / 2; ++c) acc[u][c] = make_float2(0.f, 0.f);
  uint32_t cur[FR][NC], nxt[FR][NC] = {};
  if (nchunk > 0) {
    stage(0);
    fetch(cur, g0);
  }
  for (int ch = 0; ch < nchunk; ++ch) {
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    group_sync();
    if (ch + 1 < nchunk) stage(ch + 1);
    const int64_t i0 = g0 + (int64_t)ch * PJ_RK;
    const int rows = (int)imin(PJ_RK, g1 - i0);
    const float* xs = xbuf + (ch & 1) * PJ_RK * BP + cg * TC;
    for (int s = 0; s < rows; s += FR) {
      if (i0 + s + FR < g1) fetch(nxt, i0 + s + FR);
#pragma unroll
      for (int r = 0; r < FR; ++r) {
        float2 cv[NC];
        if constexpr (VEC) {
          const float4 f = from_raw4<TIn>(cur[r]);
          cv[0] = make_float2(f.x, f.x); cv[1] = make_float2(f.y, f.y);
          cv[2] = make_float2(f.z, f.z); cv[3] = make_float2(f.w, f.w);
        } else {
#pragma unroll
          for (int u = 0; u < NC; ++u) {
            const float f = from_raw<TIn>(cur[r][u]);
            cv[u] = make_float2(f, f);
          }
        }
#pragma unroll
        for (int c4 = 0; c4 < TC / 4; ++c4) {
          const float4 x = *reinterpret_cast<const float4*>(xs + (s + r) * BP + 4 * c4);
#pragma unroll
          for (int u = 0; u < NC; ++u) {
            acc[u][2 * c4] = fma2(make_float2(x.x, x.y), cv[u], acc[u][2 * c4]);
            acc[u][2 * c4 + 1] = fma2(make_float2(x.z, x.w), cv[u], acc[u][2 * c4 + 1]);
          }
        }
      }
#pragma unroll
      for (int r = 0; r < FR; ++r)
#pragma unroll
        for (int u = 0; u < NC; ++u) cur[r][u] = nxt[r][u];
    }
  }
  // sums of the row groups, added in group order
  for (int g = 1; g < RG; ++g) {
    __syncthreads();
    if (rg == g) {
#pragma unroll
      for (int u = 0; u < NC; ++u)
#pragma unroll
        for (int c = 0; c < TC / 2; ++c) {
          pj_sm[(u * TC + 2 * c) * gt + t] = acc[u][c].x;
          pj_sm[(u * TC + 2 * c + 1) * gt + t] = acc[u][c].y;
        }
    }
    __syncthreads();
    if (rg == 0) {
#pragma unroll
      for (int u = 0; u < NC; ++u)
#pragma unroll
        for (int c = 0; c < TC / 2; ++c) {
          acc[u][c].x += pj_sm[(u * TC + 2 * c) * gt + t];
          acc[u][c].y += pj_sm[(u * TC + 2 * c + 1) * gt + t];
        }
    }
  }
  if (rg != 0) return;
#pragma unroll
  for (int c = 0; c < TC; ++c) {
    const int row = cg * TC + c;
    if (row < b) {
      TOut* out = S + (int64_t)row * lds + col;
      if constexpr (VEC) {
        float v[4];
#pragma unroll
        for (int u = 0; u < NC; ++u) v[u] = (c & 1) ? acc[u][c / 2].y : acc[u][c / 2].x;
        if (in[0]) st4(out, v);
      } else {
#pragma unroll
        for (int u = 0; u < NC; ++u)
          if (in[u]) st_elem(out, 32 * u, (c & 1) ? acc[u][c / 2].y : acc[u][c / 2].x);
      }
    }
  }
}

// S (b x n) = sum over row splits of the partials P[y] (b x n), fixed order.
template <typename TOut>
__global__ void k_sum_splits(const float* __restrict__ P, int splits, int b, int64_t n, TOut* __restrict__ S,
                             int64_t lds) {
  const int64_t E = (int64_t)b * n;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < E; e += (int64_t)gridDim.x * blockDim.x) {
    // eight loads in flight, added in split order
    float acc = 0.f;
    int y = 0;
    for (; y + 8 <= splits; y += 8) {
      float v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = P[(int64_t)(y + u) * E + e];
#pragma unroll
      for (int u = 0; u < 8; ++u) acc += v[u];
    }
    for (; y < splits; ++y) acc += P[(int64_t)y * E + e];
    st_elem(S, (e / n) * lds + e % n, acc);
  }
}

// The form for at most 256 rows of wide or short unfoldings: 64 columns x
// 16 VB rows of S a CTA, both operands staged in shared memory 32 rows at a
// time (proj_tile says where).  Three or four CTAs an SM leave the registers for every
// load of a chunk to be in flight (at 32 they took turns: 64 x 16,384 at
// b = 20 8.1 us, 6.1 so).
template <typename TIn, typename TOut, int VB>
__global__ void __launch_bounds__(256, VB == 4 ? 4 : 3) k_proj_tile(const TIn* __restrict__ C, int64_t m, int64_t n,
                                                   const float* __restrict__ X, int ldx, int b, TOut* __restrict__ S,
                                                   int64_t lds) {
  constexpr int TN = 64, RC = 32, BP = 16 * VB;
  __shared__ float Cs[RC][TN];
  __shared__ float Xs[RC][BP];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int64_t col0 = (int64_t)blockIdx.x * TN;
  float acc[VB][4] = {};
  constexpr int NC = RC * TN / 256, NX = RC * BP / 256;   // tile entries per thread
  for (int64_t i0 = 0; i0 < m; i0 += RC) {
    uint32_t cl[NC];                                      // every load in flight before the first store
    float xl[NX];
#pragma unroll
    for (int u = 0; u < NC; ++u) {
      const int e = threadIdx.x + 256 * u, r = e / TN, c = e % TN;
      cl[u] = (i0 + r < m && col0 + c < n) ? ld_raw(C + (i0 + r) * n + col0 + c) : 0u;
    }
#pragma unroll
    for (int u = 0; u < NX; ++u) {
      const int e = threadIdx.x + 256 * u, r = e / BP, c = e % BP;
      xl[u] = (i0 + r < m && c < b) ? X[(i0 + r) * ldx + c] : 0.f;
    }
#pragma unroll
    for (int u = 0; u < NC; ++u) {
      const int e = threadIdx.x + 256 * u;
      Cs[e / TN][e % TN] = from_raw<TIn>(cl[u]);
    }
#pragma unroll
    for (int u = 0; u < NX; ++u) {
      const int e = threadIdx.x + 256 * u;
      Xs[e / BP][e % BP] = xl[u];
    }
    __syncthreads();
#pragma unroll 8
    for (int r = 0; r < RC; ++r) {
      float cv[4], xv[VB];
#pragma unroll
      for (int u = 0; u < 4; ++u) cv[u] = Cs[r][tx + 16 * u];
#pragma unroll
      for (int v = 0; v < VB; ++v) xv[v] = Xs[r][ty + 16 * v];
#pragma unroll
      for (int v = 0; v < VB; ++v)
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[v][u] = fmaf(xv[v], cv[u], acc[v][u]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int v = 0; v < VB; ++v) {
    const int row = ty + 16 * v;
    if (row >= b) continue;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int64_t col = col0 + tx + 16 * u;
      if (col < n) st_elem(S, (int64_t)row * lds + col, acc[v][u]);
    }
  }
}

// Where a CTA of 64 columns is the faster form.  Above 48 columns of X and
// rows, since four or eight warps would read each element of C for themselves
// (64 x 262,144 at b = 60: 84 us, 105 by the columns' form).  And for fewer
// than 128 x 152 columns, which leave the columns' form to a few rows per
// group and their sums: 20 x 504 at b = 14 2.6 us against 5.2, 130 x 8,069 at
// b = 30 8.1 against 12.2; the wider groups of 160 rows on, and 21 to 24
// columns, are as fast there or faster.
bool proj_tile(int64_t m, int64_t n, int b, int splits) {
  if (m > 256 || splits != 1) return false;
  if (b > 48 && m > 48) return true;
  if (n >= 128 * 152) return false;
  return m <= 64 || b > 24 || (b > 12 && b <= 20 && m <= 160);
}

// Row groups of a CTA.  Two CTAs an SM (narrow outputs): as few as give the
// chip both.  One: the least time by rounds of CTAs x (rows of a group + 40,
// the start and the sums of a CTA); asking for 304 CTAs of kernels that an SM
// holds one of left a second round of few (50 x 20,973 at b = 30: 164 CTAs
// 16.6 us, 82 of them 10.4).
int proj_row_groups(int64_t n, int64_t rows_per, int splits, int CG, int held) {
  constexpr int NC = PJ_NC;
  auto ctas = [&](int rg) { return ceil_div(n, (8 / (CG * rg)) * 32 * NC) * splits; };
  int RG = 1;
  if (held == 2) {
    while (CG * RG < 8 && rows_per >= 16 * RG && ctas(RG) < 2 * 152) RG *= 2;
    return RG;
  }
  int64_t least = -1;
  for (int rg = 1; CG * rg <= 8 && (rg == 1 || rows_per >= 8 * rg); rg *= 2) {
    const int64_t t = ceil_div(ctas(rg), 152) * (ceil_div(rows_per, rg) + 40);
    if (least < 0 || t <= least) {
      least = t;
      RG = rg;
    }
  }
  return RG;
}

template <typename TIn, typename TOut, int TC, bool VEC>
cudaError_t launch_proj(const TIn* C, int64_t m, int64_t n, const float* X, int ldx, int b, TOut* S, int64_t lds,
                        int64_t rows_per, int splits, int64_t split_stride, int CG, cudaStream_t st) {
  constexpr int NC = PJ_NC;
  // narrow outputs: two CTAs an SM; the wide ones hold their 48 to 96 sums and
  // 64 loads in one, as do 12 columns of rows that are read element by element
  // (with their column offsets they spilled at 128 registers: b = 10, rows not
  // aligned, BF16 0.77 of the time, 21 to 24 0.73)
  constexpr bool kOne = TC >= 16 || (TC == 12 && !VEC);
  constexpr int FR = kOne ? 8 : 4, CTAS = kOne ? 1 : 2;
  const int RG = proj_row_groups(n, rows_per, splits, CG, CTAS);
  const int cols = (8 / (CG * RG)) * 32 * NC;
  const bool x16 = b % 4 == 0 && ldx % 4 == 0 && reinterpret_cast<uintptr_t>(X) % 16 == 0;
  const size_t smem = sizeof(float) * (size_t)imax(RG * 2 * PJ_RK * CG * TC, RG > 1 ? (256 / RG) * NC * TC : 0);
  const dim3 grid((unsigned)ceil_div(n, cols), (unsigned)splits);
  k_proj<TIn, TOut, TC, FR, CTAS, VEC><<<grid, 256, smem, st>>>(C, m, n, X, ldx, b, S, lds, rows_per, split_stride,
                                                               CG, RG, x16);
  return cudaGetLastError();
}

template <typename TIn, typename TOut>
cudaError_t proj_dispatch(const TIn* C, int64_t m, int64_t n, const float* X, int ldx, int b, TOut* S, int64_t lds,
                          int64_t rows_per, int splits, int64_t split_stride, cudaStream_t st) {
  if (b > 64) return cudaErrorInvalidValue;
  if (proj_tile(m, n, b, splits)) {
    const unsigned ctas = (unsigned)ceil_div(n, 64);
    if (b <= 16) k_proj_tile<TIn, TOut, 1><<<ctas, 256, 0, st>>>(C, m, n, X, ldx, b, S, lds);
    else if (b <= 32) k_proj_tile<TIn, TOut, 2><<<ctas, 256, 0, st>>>(C, m, n, X, ldx, b, S, lds);
    else k_proj_tile<TIn, TOut, 4><<<ctas, 256, 0, st>>>(C, m, n, X, ldx, b, S, lds);
    return cudaGetLastError();
  }
  const bool vec = n % 4 == 0 && lds % 4 == 0 && split_stride % 4 == 0 &&
                   reinterpret_cast<uintptr_t>(C) % (4 * sizeof(TIn)) == 0 &&
                   reinterpret_cast<uintptr_t>(S) % (4 * sizeof(TOut)) == 0;
#define TTR_PJ(TC, CG, VEC) \
  return launch_proj<TIn, TOut, TC, VEC>(C, m, n, X, ldx, b, S, lds, rows_per, splits, split_stride, CG, st)
#define TTR_PJ2(TC, CG)              \
  do {                               \
    if (vec) TTR_PJ(TC, CG, true);   \
    TTR_PJ(TC, CG, false);           \
  } while (0)
  if (b <= 4) TTR_PJ2(4, 1);
  if (b <= 8) TTR_PJ2(8, 1);
  if (b <= 12) TTR_PJ2(12, 1);
  if (b <= 16) TTR_PJ2(16, 1);
  if (b <= 20) TTR_PJ2(20, 1);
  if (b <= 24) TTR_PJ2(12, 2);
  if (b <= 32) TTR_PJ2(16, 2);
  if (b <= 40) TTR_PJ2(20, 2);
  if (b <= 48) {
    // element by element, reading C by four column groups costs more than 24
    // columns' sums: 200 x 83,885 at b = 45 (BF16) 158 us by four, so 78
    if (vec) TTR_PJ(12, 4, true);
    TTR_PJ(24, 2, false);
  }
  TTR_PJ2(16, 4);
#undef TTR_PJ2
#undef TTR_PJ
}

}  // namespace

// Row splits over the grid: one when the columns alone fill the chip.
int64_t simt_proj_splits(int64_t m, int64_t n) {
  const int64_t wide = ceil_div(n, 128);
  if (m < 256 || wide >= 152) return 1;
  return imax(1, imin(imin(2 * 152 / wide, ceil_div(m, 32)), 64));
}

template <typename TIn, typename TOut>
cudaError_t simt_proj(const TIn* C, int64_t m, int64_t n, const float* X, int ldx, int b, TOut* S,
                      int64_t lds, cudaStream_t st, float* partials) {
  const int64_t splits0 = partials ? simt_proj_splits(m, n) : 1;
  const int64_t rows_per = ceil_div(m, splits0), splits = ceil_div(m, rows_per);
  ProfScope prof("proj_simt", st, (double)m * n * sizeof(TIn) + (double)m * b * 4 + (double)b * n * sizeof(TOut),
                 2.0 * m * n * b);
  if (splits == 1) {
    note_launch("proj_simt");
    return proj_dispatch<TIn, TOut>(C, m, n, X, ldx, b, S, lds, m, 1, 0, st);
  }
  const int64_t E = (int64_t)b * n;
  note_launch("proj_simt", 2);
  const cudaError_t e = proj_dispatch<TIn, float>(C, m, n, X, ldx, b, partials, n, rows_per, (int)splits, E, st);
  if (e != cudaSuccess) return e;
  k_sum_splits<TOut><<<(int)imin(ceil_div(E, 256), 4 * 152), 256, 0, st>>>(partials, (int)splits, b, n, S, lds);
  return cudaGetLastError();
}

template cudaError_t simt_proj<float, float>(const float*, int64_t, int64_t, const float*, int, int, float*, int64_t, cudaStream_t, float*);
template cudaError_t simt_proj<float, __nv_bfloat16>(const float*, int64_t, int64_t, const float*, int, int, __nv_bfloat16*, int64_t, cudaStream_t, float*);
template cudaError_t simt_proj<__nv_bfloat16, float>(const __nv_bfloat16*, int64_t, int64_t, const float*, int, int, float*, int64_t, cudaStream_t, float*);
template cudaError_t simt_proj<__nv_bfloat16, __nv_bfloat16>(const __nv_bfloat16*, int64_t, int64_t, const float*, int, int, __nv_bfloat16*, int64_t, cudaStream_t, float*);

}  // namespace ttr
