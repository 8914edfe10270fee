// CUDA-core (SIMT) streaming passes over an unfolding C (m x n, row-major):
// the plain FP32 form of the passes of Alg. 3, and the form used for BF16
// shapes the tensor-core kernels do not cover.
//   cs    : Y = C S^T          (Alg. 3 step 4: the sketch C W with S = W^T,
//                               or the second half of a power)
//   gram  : G = C C^T          (exhaustion route: all of R^m is Krylov; and
//                               the tiles of the Gram-power route)
// (the projection is stream_proj.cu, the fused power stream_ga.cuh).
// Both are products of rows with rows (simt_tile.cuh).  Reductions over n are
// split across CTAs into per-CTA partials that a second kernel sums in a
// fixed order, so results are bit-reproducible.
// Measured (FP32, us; before: 2 x VB register tiles on scalar shared loads):
// the sketch of 45 x 4,100,625 at b = 6 965 -> 183 (4.0 TB/s), of
// 800 x 64,000 at b = 20 259 -> 68 and at b = 30 262 -> 103, of 7680 x 2048
// at b = 20 91 -> 26; the Gram of 32 x 1,048,576 181 -> 62, of 45 x 4,100,625
// 1,020 -> 474.  BF16, rows not aligned: the sketch of 45 x 4,100,625
// 951 -> 173, of 80 x 794,155 at b = 28 398 -> 202.
#include "common.cuh"
#include "kernels.h"
#include "simt_tile.cuh"

namespace ttr {

namespace {

// ---------------------------------------------------------------- cs
// P[split][i][c] = sum_{col in split} C[i][col] S[c][col], i in the CTA's
// row tile; grid = (row tiles, splits).
template <class Sh, typename TIn>
__global__ void __launch_bounds__(256, 2) k_cs(const TIn* __restrict__ C, int64_t m, int64_t n,
                                               const float* __restrict__ S, int64_t lds, int b,
                                               float* __restrict__ P, int64_t cols_per_split, bool va, bool vb) {
  extern __shared__ __align__(16) float nt_sm[];
  const int64_t row0 = (int64_t)blockIdx.x * Sh::BM;
  const int64_t cbeg = (int64_t)blockIdx.y * cols_per_split, cend = imin(n, cbeg + cols_per_split);
  const int rows = (int)imin(Sh::BM, m - row0);
  float* out = P + ((int64_t)blockIdx.y * m + row0) * b;
  simt::nt_tile<Sh, false>(C + row0 * n, n, rows, S, lds, b, cbeg, cend, va, vb, nt_sm,
                           [&](int i, int c, float s) {
                             if (i < rows && c < b) out[(int64_t)i * b + c] = s;
                           });
}

// ---------------------------------------------------------------- gram
// P[item] (T x T, T = Sh::BM) = rows I of C times rows J of C, transposed,
// over the item's column range; tiles I <= J enumerated J-major.
template <class Sh, typename TIn>
__global__ void __launch_bounds__(256, 2) k_gram_tiles_simt(const TIn* __restrict__ C, int64_t m, int64_t n, int splits,
                                                            float* __restrict__ P, bool vec) {
  extern __shared__ __align__(16) float nt_sm[];
  constexpr int T = Sh::BM;
  static_assert(Sh::BN == T, "square tiles");
  const int t = (int)blockIdx.x / splits, s = (int)blockIdx.x % splits;
  int J = 0;
  while ((J + 1) * (J + 2) / 2 <= t) ++J;
  const int I = t - J * (J + 1) / 2;
  const int64_t chunks = ceil_div(n, Sh::BK);
  const int64_t c0 = chunks * s / splits * Sh::BK, c1 = imin(n, chunks * (s + 1) / splits * Sh::BK);
  const int ra = (int)imin(T, m - (int64_t)I * T), rb = (int)imin(T, m - (int64_t)J * T);
  const TIn* A = C + (int64_t)I * T * n;
  const TIn* B = C + (int64_t)J * T * n;
  float* out = P + (size_t)blockIdx.x * T * T;
  auto put = [&](int i, int c, float v) { out[i * T + c] = v; };
  if (I == J) simt::nt_tile<Sh, true>(A, n, ra, A, n, ra, c0, c1, vec, vec, nt_sm, put);
  else simt::nt_tile<Sh, false>(A, n, ra, B, n, rb, c0, c1, vec, vec, nt_sm, put);
}

// As below for few splits: one thread per entry, in split order.
template <int T>
__global__ void __launch_bounds__(256) k_gram_simt_reduce_few(const float* __restrict__ P, int64_t m, int splits,
                                                              float* __restrict__ G) {
  const int i = blockIdx.y;
  const int j = (int)(blockIdx.x * blockDim.x + threadIdx.x);
  if (j < i || j >= m) return;
  const int I = i / T, J = j / T;
  const int t = J * (J + 1) / 2 + I;
  const float* src = P + (size_t)t * splits * T * T + (size_t)(i - T * I) * T + (j - T * J);
  float s = 0.f;
#pragma unroll 8
  for (int k = 0; k < splits; ++k) s += src[(size_t)k * T * T];
  G[(int64_t)i * m + j] = s;
  if (j != i) G[(int64_t)j * m + i] = s;
}

// G[i][j] = G[j][i] = sum over the splits of tile(i, j), i <= j: eight warps
// of a block take every eighth split of 32 consecutive j, in four chains, and
// the warp sums are added in a fixed tree (one thread per entry left the
// short Grams waiting on a chain of hundreds of loads).
template <int T>
__global__ void __launch_bounds__(256) k_gram_simt_reduce(const float* __restrict__ P, int64_t m, int splits,
                                                          float* __restrict__ G) {
  __shared__ float red[8][33];
  const int i = blockIdx.y, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int j = (int)blockIdx.x * 32 + lane;
  if ((int)blockIdx.x * 32 + 31 < i) return;
  const bool live = j >= i && j < m;
  float a[4] = {0.f, 0.f, 0.f, 0.f};
  if (live) {
    const int I = i / T, J = j / T;
    const int t = J * (J + 1) / 2 + I;
    const float* src = P + (size_t)t * splits * T * T + (size_t)(i - T * I) * T + (j - T * J);
    int k = w;
    for (; k + 24 < splits; k += 32) {
#pragma unroll
      for (int u = 0; u < 4; ++u) a[u] += src[(size_t)(k + 8 * u) * T * T];
    }
    for (; k < splits; k += 8) a[0] += src[(size_t)k * T * T];
  }
  red[w][lane] = (a[0] + a[1]) + (a[2] + a[3]);
  __syncthreads();
  if (w == 0 && live) {
    const float s = ((red[0][lane] + red[1][lane]) + (red[2][lane] + red[3][lane])) +
                    ((red[4][lane] + red[5][lane]) + (red[6][lane] + red[7][lane]));
    G[(int64_t)i * m + j] = s;
    if (j != i) G[(int64_t)j * m + i] = s;
  }
}

// ---------------------------------------------------------------- reduce
// out[r * ldo + c] = sum_{s < S} P[s][r][c] (fixed order), r < rows, c < cols.
// A block takes 32 consecutive elements (lane = element, each load of a warp
// one 128-byte row of a partial); warp w sums the partials w, w + 8, ... in
// four interleaved chains, and the eight warp sums are added in a fixed
// tree: every element sees the same order whatever the grid, so reruns are
// bit-identical, and a short element range still spreads over eight warps.
constexpr int RED_WARPS = 8;

__device__ __forceinline__ float strided_sum_warp(const float* __restrict__ p, int n, int64_t stride, int w) {
  float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
  int k = w;
  for (; k + 3 * RED_WARPS < n; k += 4 * RED_WARPS) {
    a0 += p[(int64_t)k * stride];
    a1 += p[(int64_t)(k + RED_WARPS) * stride];
    a2 += p[(int64_t)(k + 2 * RED_WARPS) * stride];
    a3 += p[(int64_t)(k + 3 * RED_WARPS) * stride];
  }
  for (; k < n; k += RED_WARPS) a0 += p[(int64_t)k * stride];
  return (a0 + a1) + (a2 + a3);
}

// base(e) + k * stride is partial k of element e (k < n); out[e] = the sum.
template <typename Base>
__device__ __forceinline__ void reduce_elements(Base base, int n, int64_t stride, int64_t E, int cols,
                                                float* __restrict__ out, int64_t ldo) {
  __shared__ float red[RED_WARPS][33];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int64_t e0 = (int64_t)blockIdx.x * 32; e0 < E; e0 += (int64_t)gridDim.x * 32) {
    const int64_t e = e0 + lane;
    red[w][lane] = (e < E) ? strided_sum_warp(base(e), n, stride, w) : 0.f;
    __syncthreads();
    if (w == 0 && e < E) {
      const float t = ((red[0][lane] + red[1][lane]) + (red[2][lane] + red[3][lane])) +
                      ((red[4][lane] + red[5][lane]) + (red[6][lane] + red[7][lane]));
      out[(e / cols) * ldo + e % cols] = t;
    }
    __syncthreads();
  }
}

struct PartialsFlat {
  const float* P;
  __device__ const float* operator()(int64_t e) const { return P + e; }
};
struct PartialsGrouped {   // element e's row group g = e / cols / group_rows starts at slot g
  const float* P;
  int64_t E, cols, group_rows;
  __device__ const float* operator()(int64_t e) const { return P + (e / cols / group_rows) * E + e; }
};

__global__ void __launch_bounds__(32 * RED_WARPS) k_reduce_partials(const float* __restrict__ P, int S, int64_t rows,
                                                                    int cols, float* __restrict__ out, int64_t ldo) {
  const int64_t E = rows * cols;
  reduce_elements(PartialsFlat{P}, S, E, E, cols, out, ldo);
}

// As above for at most eight partials, which leave most of the eight warps
// idle: one thread per element, in partial order (two partials of 7680 x 20:
// 5.8 us by warps; the 7680 x 2048 call with five of them 796 us, so 771).
__global__ void __launch_bounds__(256) k_reduce_few(const float* __restrict__ P, int S, int64_t rows, int cols,
                                                    float* __restrict__ out, int64_t ldo) {
  const int64_t E = rows * cols;
  const bool dense = ldo == cols;
  for (int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x; e < E; e += (int64_t)gridDim.x * 256) {
    float v[8];
#pragma unroll
    for (int s = 0; s < 8; ++s) v[s] = (s < S) ? P[s * E + e] : 0.f;
    float a = v[0];
#pragma unroll
    for (int s = 1; s < 8; ++s)
      if (s < S) a += v[s];
    if (dense) {
      out[e] = a;
    } else {
      const int64_t r = e / cols;
      out[r * ldo + (e - r * cols)] = a;
    }
  }
}

// out[r][c] = sum over the CTAs of r's row group (slot j * groups + g) of
// their partials; the CTAs of a group write only that group's rows.
__global__ void __launch_bounds__(32 * RED_WARPS) k_reduce_grouped(const float* __restrict__ P, int per, int groups,
                                                                   int64_t rows, int cols, int64_t group_rows,
                                                                   float* __restrict__ out, int64_t ldo) {
  const int64_t E = rows * cols;
  reduce_elements(PartialsGrouped{P, E, cols, group_rows}, per, (int64_t)groups * E, E, cols, out, ldo);
}

}  // namespace

// ======================================================================
// Launchers
// ======================================================================
static void reduce_launch(const float* P, int S, int64_t rows, int cols, float* out, int64_t ldo,
                          cudaStream_t st) {
  int64_t E = rows * cols;
  if (S <= 8) {
    k_reduce_few<<<(int)imin(ceil_div(E, 256), 152 * 8), 256, 0, st>>>(P, S, rows, cols, out, ldo);
  } else {
    const int blocks = (int)imin(ceil_div(E, 32), 4096);
    k_reduce_partials<<<blocks, 32 * RED_WARPS, 0, st>>>(P, S, rows, cols, out, ldo);
  }
  note_launch("reduce_partials");
}

cudaError_t launch_reduce_partials(const float* P, int S, int64_t rows, int cols, float* out, int64_t ldo,
                                   cudaStream_t st) {
  reduce_launch(P, S, rows, cols, out, ldo, st);
  return cudaGetLastError();
}

cudaError_t launch_reduce_partials_grouped(const float* P, int per, int groups, int64_t rows, int cols,
                                           int64_t group_rows, float* out, int64_t ldo, cudaStream_t st) {
  const int64_t E = rows * cols;
  note_launch("reduce_partials");
  k_reduce_grouped<<<(int)imin(ceil_div(E, 32), 4096), 32 * RED_WARPS, 0, st>>>(P, per, groups, rows, cols,
                                                                                group_rows, out, ldo);
  return cudaGetLastError();
}

namespace {

// Rows of a cs tile: the shortest of 32, 48 and 64 that takes all rows, else 64.
int cs_tile_rows(int64_t m) { return m <= 32 ? 32 : m <= 48 ? 48 : 64; }

// Two CTAs an SM in all, a split at least 256 columns.
int64_t cs_splits(int64_t m, int64_t n) {
  const int64_t rt = ceil_div(m, cs_tile_rows(m));
  return imax(1, imin(imax(1, 2 * 152 / rt), ceil_div(n, 256)));
}

template <class Sh, typename TIn>
cudaError_t cs_launch(const TIn* C, int64_t m, int64_t n, const float* S, int64_t lds, int b, float* P, int splits,
                      cudaStream_t st) {
  const int64_t per = ceil_div(ceil_div(n, Sh::BK), splits) * Sh::BK;
  constexpr size_t smem = sizeof(float) * Sh::smem_floats(false);
  if (smem > 48 * 1024) {
    const cudaError_t e = raise_smem_limit(k_cs<Sh, TIn>);
    if (e != cudaSuccess) return e;
  }
  // vector loads end with the row only where n is a multiple of four, however S is spaced
  k_cs<Sh, TIn><<<dim3((unsigned)ceil_div(m, Sh::BM), (unsigned)splits), 256, smem, st>>>(
      C, m, n, S, lds, b, P, per, simt::rows_aligned4(C, n), n % 4 == 0 && simt::rows_aligned4(S, lds));
  return cudaGetLastError();
}

template <int TR, typename TIn>
cudaError_t cs_dispatch(const TIn* C, int64_t m, int64_t n, const float* S, int64_t lds, int b, float* P, int splits,
                        cudaStream_t st) {
#define TTR_CS(TC, CT) return cs_launch<simt::NtShape<TR, TC, CT>>(C, m, n, S, lds, b, P, splits, st)
  if (b <= 4) TTR_CS(4, 1);
  if (b <= 6) TTR_CS(6, 1);
  if (b <= 8) TTR_CS(8, 1);
  if (b <= 12) TTR_CS(6, 2);
  if (b <= 16) TTR_CS(8, 2);
  if (b <= 20) TTR_CS(5, 4);
  if (b <= 24) TTR_CS(3, 8);
  if (b <= 32) TTR_CS(4, 8);
  if (b <= 40) TTR_CS(5, 8);
  if (b <= 48) TTR_CS(6, 8);
  if (b <= 64) TTR_CS(4, 16);
#undef TTR_CS
  return cudaErrorInvalidValue;
}

}  // namespace

template <typename TIn>
cudaError_t simt_cs(const TIn* C, int64_t m, int64_t n, const float* S, int64_t lds, int b,
                    float* partials, float* out, int64_t ldo, cudaStream_t st) {
  const int splits = (int)cs_splits(m, n);
  {
    ProfScope prof("cs_simt", st, (double)m * n * sizeof(TIn) + (double)b * n * 4, 2.0 * m * n * b);
    note_launch("cs_simt");
    const int rows = cs_tile_rows(m);
    const cudaError_t e = rows == 32   ? cs_dispatch<4>(C, m, n, S, lds, b, partials, splits, st)
                          : rows == 48 ? cs_dispatch<6>(C, m, n, S, lds, b, partials, splits, st)
                                       : cs_dispatch<8>(C, m, n, S, lds, b, partials, splits, st);
    if (e != cudaSuccess) return e;
  }
  reduce_launch(partials, splits, m, b, out, ldo, st);
  return cudaGetLastError();
}

int64_t simt_cs_partials(int64_t m, int64_t n, int b) { return cs_splits(m, n) * m * b; }

// ---------------------------------------------------------------- gram
namespace {

// Tile edge, tiles of the upper triangle and splits of the columns.
struct GramPlan {
  int edge, tiles, splits;
};

// One tile of 16 or 32 for the shortest; else of 48 and 64 the edge, and of
// the splits that give every SM one CTA or two, those with the least time by
//   (chunks of a CTA + 1/2) x (1.85 per two CTAs an SM holds, 1 for one alone)
// plus one where more than eight partials are left to add, with a chunk of a
// 64-row tile 1.6 times a 48-row one (the ratios measured at 200 to 1,000
// rows).  The splits go down to one chunk, since a short Gram is one chain of
// chunks.  A fixed minimum of 256 columns a split and the edge by padding alone
// gave 700 columns of 39 rows three CTAs (9.5 us, so 5.7) and 800 x 8,000
// one CTA of 48 rows an SM (276 us, 176 as 64-row tiles in three splits).
GramPlan gram_plan(int64_t m, int64_t n) {
  const int64_t chunks = ceil_div(n, 64);
  GramPlan best = {};
  double least = 0.;
  for (const int edge : {16, 32, 48, 64}) {
    if (m <= 32 ? edge != (m <= 16 ? 16 : 32) : edge < 48) continue;
    const int64_t nT = ceil_div(m, edge), tiles = nT * (nT + 1) / 2;
    for (const int64_t ctas : {152, 304}) {
      int64_t splits = imax(1, imin(ctas / tiles, chunks));
      const int64_t per = ceil_div(chunks, splits);
      splits = ceil_div(chunks, per);
      const int64_t held = ceil_div(tiles * splits, 152);     // CTAs of the fullest SM
      const double t = (per + 0.5) * ((held / 2) * 1.85 + held % 2) * (edge == 64 ? 1.6 : 1.) + (splits > 8);
      if (best.edge == 0 || t < least) {
        least = t;
        best = {edge, (int)tiles, (int)splits};
      }
    }
  }
  return best;
}

template <class Sh, typename TIn>
cudaError_t gram_launch(const TIn* C, int64_t m, int64_t n, int tiles, int splits, float* P, float* G,
                        cudaStream_t st) {
  constexpr size_t smem = sizeof(float) * Sh::smem_floats(false);
  if (smem > 48 * 1024) {
    const cudaError_t e = raise_smem_limit(k_gram_tiles_simt<Sh, TIn>);
    if (e != cudaSuccess) return e;
  }
  k_gram_tiles_simt<Sh, TIn><<<tiles * splits, 256, smem, st>>>(C, m, n, splits, P, simt::rows_aligned4(C, n));
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  note_launch("gram_reduce");
  if (splits <= 8)   // 800 rows, 2 splits: 5.7 us against 13.8 by eight warps
    k_gram_simt_reduce_few<Sh::BM><<<dim3((unsigned)ceil_div(m, 256), (unsigned)m), 256, 0, st>>>(P, m, splits, G);
  else
    k_gram_simt_reduce<Sh::BM><<<dim3((unsigned)ceil_div(m, 32), (unsigned)m), 256, 0, st>>>(P, m, splits, G);
  return cudaGetLastError();
}

}  // namespace

template <typename TIn>
cudaError_t simt_gram(const TIn* C, int64_t m, int64_t n, float* partials, float* out, cudaStream_t st,
                      const char* family) {
  const GramPlan p = gram_plan(m, n);
  ProfScope prof(family, st, (double)m * n * sizeof(TIn), 2.0 * m * m * n);
  note_launch(family);
  switch (p.edge) {
    case 16: return gram_launch<simt::NtShape<2, 8, 2>>(C, m, n, p.tiles, p.splits, partials, out, st);
    case 32: return gram_launch<simt::NtShape<4, 8, 4>>(C, m, n, p.tiles, p.splits, partials, out, st);
    case 48: return gram_launch<simt::NtShape<6, 6, 8>>(C, m, n, p.tiles, p.splits, partials, out, st);
    default: return gram_launch<simt::NtShape<8, 4, 16>>(C, m, n, p.tiles, p.splits, partials, out, st);
  }
}

int64_t simt_gram_partials(int64_t m, int64_t n) {
  const GramPlan p = gram_plan(m, n);
  return (int64_t)p.tiles * p.splits * p.edge * p.edge;
}

// Explicit instantiations.
template cudaError_t simt_cs<float>(const float*, int64_t, int64_t, const float*, int64_t, int, float*, float*, int64_t, cudaStream_t);
template cudaError_t simt_cs<__nv_bfloat16>(const __nv_bfloat16*, int64_t, int64_t, const float*, int64_t, int, float*, float*, int64_t, cudaStream_t);
template cudaError_t simt_gram<float>(const float*, int64_t, int64_t, float*, float*, cudaStream_t, const char*);
template cudaError_t simt_gram<__nv_bfloat16>(const __nv_bfloat16*, int64_t, int64_t, float*, float*, cudaStream_t, const char*);

}  // namespace ttr
