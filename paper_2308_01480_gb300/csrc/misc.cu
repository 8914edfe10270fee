// Input-side kernels: the Gaussian test matrices of Alg. 3 step 3 drawn on
// the device, and the canonicalising permute/convert of a strided tensor.
#include "common.cuh"
#include "kernels.h"

namespace ttr {

// Philox4x32 with 10 rounds, from its published definition (Salmon, Moraes,
// Dror, Shaw, SC'11): per round the two multiplications give high and low
// halves that are mixed with the other two words and the round key; the key
// advances by the two Weyl increments between rounds.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
    const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
    c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  return c;
}

// (0,1) uniform with 24 significant bits: exact in binary32.
__device__ __forceinline__ float u01(uint32_t x) {
  return ((float)(x >> 9) + 0.5f) * 1.1920928955078125e-07f;  // 2^-23
}

// Box-Muller (1958): (u1, u2) -> sqrt(-2 ln u1) (cos 2 pi u2, sin 2 pi u2).
__device__ __forceinline__ float2 box_muller(uint32_t a, uint32_t b) {
  const float rad = sqrtf(-2.f * logf(u01(a)));
  float s, c;
  sincospif(2.f * u01(b), &s, &c);
  return make_float2(rad * c, rad * s);
}

// Omega_k entry (i, c) written at out[i * si + c * sc], i < n, c < b.  With
// a slab (w > 0) the n local rows are the rows (i / w) nd + lo + i % w of
// the full Omega_k: the columns of the unfolding whose last index lies in
// [lo, lo + w) of a last mode of size nd, in their order.
// A thread draws four columns (one Philox block) of one row at a time, the
// column group from the grid's second dimension: with a 64-bit division and
// remainder per draw 4,100,625 x 6 (FP32) took 88 us, so 70; the rest is the
// transform.
template <typename T>
__global__ void __launch_bounds__(256) k_omega(uint64_t seed, uint32_t mode, int64_t n, int b, T* __restrict__ out,
                                               int64_t si, int64_t sc, int64_t w, int64_t nd, int64_t lo) {
  const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
  for (int g = (int)blockIdx.y; 4 * g < b; g += (int)gridDim.y) {
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) {
      const int64_t gi = (w > 0) ? (i / w) * nd + lo + i % w : i;   // row of the full Omega_k
      const uint4 x =
          philox4x32_10(make_uint4((uint32_t)gi, (uint32_t)((uint64_t)gi >> 32), (uint32_t)g, mode), k0, k1);
      const float2 z01 = box_muller(x.x, x.y);
      const float2 z23 = box_muller(x.z, x.w);
      const float z[4] = {z01.x, z01.y, z23.x, z23.y};
      T* p = out + i * si + (int64_t)(4 * g) * sc;
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        if (4 * g + t < b) st_elem(p, 0, z[t]);
        p += sc;
      }
    }
  }
}

cudaError_t launch_omega(uint64_t seed, int mode, int64_t n, int b, void* out, int dtype, int64_t si,
                         int64_t sc, cudaStream_t st, int64_t slab_w, int64_t slab_nd, int64_t slab_lo) {
  const int groups = (b + 3) / 4;
  const dim3 grid((unsigned)imax(1, imin(ceil_div(n, 256), imax(1, 152 * 16 / groups))),
                  (unsigned)imin(groups, 65535));
  ProfScope prof("omega_philox", st, (double)n * b * (dtype == TT_BF16 ? 2 : 4), 0);
  note_launch("omega_philox");
  if (dtype == TT_BF16)
    k_omega<__nv_bfloat16><<<grid, 256, 0, st>>>(seed, (uint32_t)mode, n, b, (__nv_bfloat16*)out, si, sc, slab_w,
                                                 slab_nd, slab_lo);
  else
    k_omega<float><<<grid, 256, 0, st>>>(seed, (uint32_t)mode, n, b, (float*)out, si, sc, slab_w, slab_nd, slab_lo);
  return cudaGetLastError();
}

// Transposed copy of an explicit Omega (n x b row-major, b <= 64) into the
// b x n layout read by the sketch pass, with dtype conversion.  HBM bounds
// it: a CTA reads the b TR contiguous floats of TR rows in order, keeps them
// transposed in shared memory (odd row stride: no bank conflicts on the way
// in) and writes each column's TR entries together.  524,288 x 40 to BF16:
// one strided element a thread took 116 us, this 26 us.
template <typename T>
__global__ void __launch_bounds__(256) k_transpose_in(const float* __restrict__ src, int64_t n, int b,
                                                      T* __restrict__ dst, bool pair) {
  constexpr int TR = 128;
  extern __shared__ float omt[];               // [b][TR + 1]
  const int64_t r0 = (int64_t)blockIdx.x * TR;
  const int rows = (int)imin(TR, n - r0);
  const float* s = src + r0 * b;
  const int total = rows * b, dc = 256 % b, dr = 256 / b;
  int c = threadIdx.x % b, r = threadIdx.x / b;
  for (int e = threadIdx.x; e < total; e += 4 * 256) {
    float v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = (e + 256 * u < total) ? s[e + 256 * u] : 0.f;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (e + 256 * u < total) omt[c * (TR + 1) + r] = v[u];
      c += dc;
      r += dr;
      if (c >= b) {
        c -= b;
        ++r;
      }
    }
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  for (int col = threadIdx.x >> 5; col < b; col += 8) {
    const float* t = omt + col * (TR + 1);
    T* out = dst + (int64_t)col * n + r0;
    if constexpr (sizeof(T) == 2) {
      if (pair) {                              // n even: rows, and pairs in them, are 4-byte aligned
#pragma unroll
        for (int u = 0; u < TR / 64; ++u) {
          const int i = 2 * lane + 64 * u;
          if (i < rows) *reinterpret_cast<__nv_bfloat162*>(out + i) = __floats2bfloat162_rn(t[i], t[i + 1]);
        }
        continue;
      }
    }
#pragma unroll
    for (int u = 0; u < TR / 32; ++u) {
      const int i = lane + 32 * u;
      if (i < rows) st_elem(out, i, t[i]);
    }
  }
}

cudaError_t launch_omega_transpose_any(const float* src, int64_t n, int b, void* dst, int dtype, cudaStream_t st) {
  if (b < 1 || b > 64) return cudaErrorInvalidValue;
  const dim3 grid((unsigned)ceil_div(n, 128));
  const size_t smem = sizeof(float) * (size_t)b * 129;
  note_launch("omega_transpose");
  if (dtype == TT_BF16)
    k_transpose_in<__nv_bfloat16><<<grid, 256, smem, st>>>(src, n, b, (__nv_bfloat16*)dst,
                                                           n % 2 == 0 && reinterpret_cast<uintptr_t>(dst) % 4 == 0);
  else
    k_transpose_in<float><<<grid, 256, smem, st>>>(src, n, b, (float*)dst, false);
  return cudaGetLastError();
}

// ------------------------------------------------------------ permute/convert
// A dense copy with its modes in another order.  The copy moves every byte
// once, so HBM bounds it; what it must avoid is index arithmetic per element
// and loads or stores that use a few bytes of each 32-byte sector.  The host
// first drops modes of size one and merges neighbouring destination modes
// that are also neighbours in the source, then picks by the source stride of
// the innermost destination mode:
//   rows   it is 1: both sides run along the same mode; 4 elements a thread
//          where every row starts aligned, else 1
//   tiles  another mode has the smallest stride and both modes hold at least
//          kPermTileMin entries: tiles of these two modes go through shared
//          memory, so that loads run along the source's fastest mode and
//          stores along the destination's
//   generic  the rest (a fastest mode too short to fill a quarter of a
//          warp's load): one element a thread at a time
// Indices are 32-bit with division by multiplication; a copy of 2^31
// elements or more takes the generic kernel with 64-bit division.
// Measured, 256 x 256 x 64 x 32 FP32 to BF16 in mode order (4, 2, 1, 3):
// one element a thread with 64-bit divisions took 2,235 us (360 GB/s);
// tiles take 167 us (4,820 GB/s, 0.71 of the measured copy rate).
constexpr int kPermMax = 8;
constexpr int64_t kPermTileMin = 8;

// n / d for n < 2^31 as a multiply-high, an add and a shift (d >= 1), after
// Granlund and Montgomery, Division by Invariant Integers using Multiplication
// (1994).
struct FastDiv {
  uint32_t d, mul, sh;
};
inline FastDiv fast_div(uint32_t d) {
  FastDiv f;
  f.d = d;
  f.sh = 0;
  while ((1ull << f.sh) < d) ++f.sh;
  f.mul = (uint32_t)(((1ull << 32) * ((1ull << f.sh) - d)) / d + 1);
  return f;
}
__device__ __forceinline__ uint32_t div_by(uint32_t n, const FastDiv& f) { return (__umulhi(n, f.mul) + n) >> f.sh; }

struct PermArgs {
  int d;
  int64_t ddims[kPermMax];     // destination mode sizes
  int64_t sstride[kPermMax];   // source stride of destination mode j
  FastDiv div[kPermMax];       // of ddims (32-bit kernels)
};

// Source offset of the element whose destination index over modes [0, d) is e.
__device__ __forceinline__ int64_t perm_offset(const PermArgs& a, int d, uint32_t e) {
  int64_t off = 0;
  for (int j = d - 1; j >= 0; --j) {
    const uint32_t q = div_by(e, a.div[j]);
    off += (int64_t)(e - q * a.div[j].d) * a.sstride[j];
    e = q;
  }
  return off;
}

template <typename TS, typename TD>
__global__ void k_permute_wide(const TS* __restrict__ src, TD* __restrict__ dst, int64_t total, PermArgs a) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    int64_t rem = e, off = 0;
    for (int j = a.d - 1; j >= 0; --j) {
      const int64_t idx = rem % a.ddims[j];
      rem /= a.ddims[j];
      off += idx * a.sstride[j];
    }
    st_elem(dst, e, ld_elem(src, off));
  }
}

template <typename TS, typename TD>
__global__ void __launch_bounds__(256) k_permute_generic(const TS* __restrict__ src, TD* __restrict__ dst,
                                                         uint32_t total, const __grid_constant__ PermArgs a) {
  const uint32_t step = gridDim.x * 256u;
  for (uint32_t e = blockIdx.x * 256u + threadIdx.x; e < total; e += 4 * step) {
    float v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const uint32_t x = e + (uint32_t)u * step;
      v[u] = (x < total) ? ld_elem(src, perm_offset(a, a.d, x)) : 0.f;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const uint32_t x = e + (uint32_t)u * step;
      if (x < total) st_elem(dst, (int64_t)x, v[u]);
    }
  }
}

// Innermost destination mode contiguous in the source.  vecs: vectors of V
// elements in all; per_row: its division by the vectors of one row.
template <typename TS, typename TD, int V>
__global__ void __launch_bounds__(256) k_permute_rows(const TS* __restrict__ src, TD* __restrict__ dst, uint32_t vecs,
                                                      FastDiv per_row, const __grid_constant__ PermArgs a) {
  constexpr int U = 4;                       // vectors in flight per thread
  const uint32_t step = gridDim.x * 256u;
  for (uint32_t e = blockIdx.x * 256u + threadIdx.x; e < vecs; e += U * step) {
    float v[U][V];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const uint32_t x = e + (uint32_t)u * step;
      if (x < vecs) {
        const uint32_t row = div_by(x, per_row);
        const TS* p = src + perm_offset(a, a.d - 1, row) + (int64_t)(x - row * per_row.d) * V;
        if constexpr (V == 4) ld4(p, v[u]);
        else v[u][0] = ld_elem(p, 0);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const uint32_t x = e + (uint32_t)u * step;
      if (x < vecs) {
        if constexpr (V == 4) st4(dst + (int64_t)x * 4, v[u]);
        else st_elem(dst, (int64_t)x, v[u][0]);
      }
    }
  }
}

struct PermTile {
  uint32_t S, J;          // sizes of mode s (smallest source stride) and of the innermost mode
  uint32_t nts, ntj;      // tiles along each
  FastDiv fts, ftj;
  PermArgs o;             // the other modes, in destination order
  int64_t odst[kPermMax]; // their destination strides
  int64_t sj;             // source stride of the innermost mode
  int64_t ss;             // source stride of mode s
  int64_t ds;             // destination stride of mode s
  uint32_t tiles;
};

// TJ x TSZ tiles: 256 threads read rows of TSZ source-contiguous entries
// (lane = mode s) into shared memory and write rows of TJ entries (lane = the
// innermost mode), two to a 4-byte store for BF16 where rows are even (PAIR).
// The odd row stride keeps both directions free of bank conflicts, but for the
// paired stores of 64-entry rows, whose two reads each take two turns (entries
// 32 apart share a bank); 8 to 16 loads a thread are in flight.
template <typename TS, typename TD, int TSZ, int TJ, bool PAIR>
__global__ void __launch_bounds__(256) k_permute_tiles(const TS* __restrict__ src, TD* __restrict__ dst,
                                                       const __grid_constant__ PermTile p) {
  __shared__ float t[TJ][TSZ + 1];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (uint32_t tile = blockIdx.x; tile < p.tiles; tile += gridDim.x) {
    uint32_t q = div_by(tile, p.ftj);
    const uint32_t j0 = (tile - q * p.ntj) * TJ;
    uint32_t o = div_by(q, p.fts);
    const uint32_t s0 = (q - o * p.nts) * TSZ;
    int64_t so = (int64_t)s0 * p.ss + (int64_t)j0 * p.sj, dof = (int64_t)s0 * p.ds + j0;
    for (int j = p.o.d - 1; j >= 0; --j) {
      const uint32_t n = div_by(o, p.o.div[j]);
      const uint32_t idx = o - n * p.o.div[j].d;
      so += (int64_t)idx * p.o.sstride[j];
      dof += (int64_t)idx * p.odst[j];
      o = n;
    }
    const TS* ps = src + so;
    TD* pd = dst + dof;
    const int S = (int)min(p.S - s0, (uint32_t)TSZ), J = (int)min(p.J - j0, (uint32_t)TJ);
    constexpr int NS = TSZ / 32, NJ = TJ / 8;
    float v[NJ][NS];
#pragma unroll
    for (int a = 0; a < NJ; ++a)
#pragma unroll
      for (int b = 0; b < NS; ++b) {
        const int j = w + 8 * a, s = lane + 32 * b;
        v[a][b] = (j < J && s < S) ? ld_elem(ps, (int64_t)j * p.sj + (int64_t)s * p.ss) : 0.f;
      }
#pragma unroll
    for (int a = 0; a < NJ; ++a)
#pragma unroll
      for (int b = 0; b < NS; ++b) t[w + 8 * a][lane + 32 * b] = v[a][b];
    __syncthreads();
    if constexpr (PAIR) {
      constexpr int HW = TJ / 2;             // pairs in a row: 16 or 32 lanes
      constexpr int RPW = 32 / HW;
      const int jp = lane % HW, sub = lane / HW;
#pragma unroll
      for (int a = 0; a < TSZ / (8 * RPW); ++a) {
        const int s = (w + 8 * a) * RPW + sub;
        if (s < S && 2 * jp < J)
          *reinterpret_cast<__nv_bfloat162*>(pd + (int64_t)s * p.ds + 2 * jp) =
              __floats2bfloat162_rn(t[2 * jp][s], t[2 * jp + 1][s]);
      }
    } else {
#pragma unroll
      for (int a = 0; a < TSZ / 8; ++a)
#pragma unroll
        for (int b = 0; b < TJ / 32; ++b) {
          const int s = w + 8 * a, j = lane + 32 * b;
          if (s < S && j < J) st_elem(pd, (int64_t)s * p.ds + j, t[j][s]);
        }
    }
    __syncthreads();
  }
}

template <typename TS, typename TD>
static cudaError_t permute_typed(const TS* src, TD* dst, int64_t total, PermArgs a, cudaStream_t st) {
  // merge destination modes that are neighbours in the source as well
  PermArgs c = {};
  for (int j = 0; j < a.d; ++j) {
    if (a.ddims[j] == 1) continue;
    if (c.d > 0 && c.sstride[c.d - 1] == a.sstride[j] * a.ddims[j]) {
      c.ddims[c.d - 1] *= a.ddims[j];
      c.sstride[c.d - 1] = a.sstride[j];
    } else {
      c.ddims[c.d] = a.ddims[j];
      c.sstride[c.d] = a.sstride[j];
      ++c.d;
    }
  }
  if (c.d == 0) {
    c.d = 1;
    c.ddims[0] = 1;
    c.sstride[0] = 1;
  }
  constexpr int kCtas = 152 * 8;
  if (total >= (int64_t(1) << 31)) {
    k_permute_wide<TS, TD><<<152 * 32, 256, 0, st>>>(src, dst, total, c);
    return cudaGetLastError();
  }
  for (int j = 0; j < c.d; ++j) c.div[j] = fast_div((uint32_t)c.ddims[j]);
  const int last = c.d - 1;
  if (c.sstride[last] == 1) {
    bool v4 = c.ddims[last] % 4 == 0 && (uintptr_t)src % (4 * sizeof(TS)) == 0 && (uintptr_t)dst % (4 * sizeof(TD)) == 0;
    for (int j = 0; j < last; ++j) v4 = v4 && c.sstride[j] % 4 == 0;
    const uint32_t vecs = (uint32_t)(v4 ? total / 4 : total);
    const FastDiv per_row = fast_div((uint32_t)(v4 ? c.ddims[last] / 4 : c.ddims[last]));
    const int grid = (int)imin(ceil_div(vecs, 1024), kCtas);
    if (v4) k_permute_rows<TS, TD, 4><<<grid, 256, 0, st>>>(src, dst, vecs, per_row, c);
    else k_permute_rows<TS, TD, 1><<<grid, 256, 0, st>>>(src, dst, vecs, per_row, c);
    return cudaGetLastError();
  }
  int s = last;
  for (int j = 0; j < c.d; ++j)
    if (c.sstride[j] > 0 && (c.sstride[s] == 0 || c.sstride[j] < c.sstride[s])) s = j;
  if (s == last || c.ddims[s] < kPermTileMin || c.ddims[last] < kPermTileMin) {
    k_permute_generic<TS, TD><<<(int)imin(ceil_div(total, 1024), kCtas), 256, 0, st>>>(src, dst, (uint32_t)total, c);
    return cudaGetLastError();
  }
  PermTile p = {};
  p.S = (uint32_t)c.ddims[s];
  p.J = (uint32_t)c.ddims[last];
  p.ss = c.sstride[s];
  p.sj = c.sstride[last];
  int64_t dstride = 1, outer = 1;
  int64_t ds[kPermMax];
  for (int j = last; j >= 0; --j) {
    ds[j] = dstride;
    dstride *= c.ddims[j];
  }
  p.ds = ds[s];
  for (int j = 0; j < last; ++j)
    if (j != s) {
      p.o.ddims[p.o.d] = c.ddims[j];
      p.o.sstride[p.o.d] = c.sstride[j];
      p.o.div[p.o.d] = c.div[j];
      p.odst[p.o.d] = ds[j];
      ++p.o.d;
      outer *= c.ddims[j];
    }
  const int tsz = p.S > 32 ? 64 : 32, tj = p.J > 32 ? 64 : 32;
  p.nts = (uint32_t)ceil_div(p.S, tsz);
  p.ntj = (uint32_t)ceil_div(p.J, tj);
  p.fts = fast_div(p.nts);
  p.ftj = fast_div(p.ntj);
  p.tiles = (uint32_t)(outer * p.nts * p.ntj);   // each tile holds at least one element: < 2^31
  const int grid = (int)imin(p.tiles, 2 * kCtas);
  const bool pair = sizeof(TD) == 2 && p.J % 2 == 0 && (uintptr_t)dst % 4 == 0;
#define TTR_PT(A, B)                                                                              \
  do {                                                                                            \
    if constexpr (sizeof(TD) == 2) {                                                              \
      if (pair) {                                                                                 \
        k_permute_tiles<TS, TD, A, B, true><<<grid, 256, 0, st>>>(src, dst, p);                   \
        return cudaGetLastError();                                                                \
      }                                                                                           \
    }                                                                                             \
    k_permute_tiles<TS, TD, A, B, false><<<grid, 256, 0, st>>>(src, dst, p);                      \
  } while (0)
  if (tsz == 64 && tj == 64) TTR_PT(64, 64);
  else if (tsz == 64) TTR_PT(64, 32);
  else if (tj == 64) TTR_PT(32, 64);
  else TTR_PT(32, 32);
#undef TTR_PT
  return cudaGetLastError();
}

cudaError_t launch_permute(const void* src, int sdt, void* dst, int ddt, const int64_t* dims,
                           const int64_t* sstrides, const int* perm, int d, cudaStream_t st) {
  PermArgs a = {};
  a.d = d;
  int64_t total = 1;
  for (int j = 0; j < d; ++j) {
    const int s = perm ? perm[j] : j;
    a.ddims[j] = dims[s];
    a.sstride[j] = sstrides[s];
    total *= dims[s];
  }
  if (total == 0) return cudaSuccess;
  note_launch("permute_convert");
  if (sdt == TT_F32 && ddt == TT_F32) return permute_typed((const float*)src, (float*)dst, total, a, st);
  if (sdt == TT_F32 && ddt == TT_BF16) return permute_typed((const float*)src, (__nv_bfloat16*)dst, total, a, st);
  if (sdt == TT_BF16 && ddt == TT_BF16)
    return permute_typed((const __nv_bfloat16*)src, (__nv_bfloat16*)dst, total, a, st);
  if (sdt == TT_BF16 && ddt == TT_F32) return permute_typed((const __nv_bfloat16*)src, (float*)dst, total, a, st);
  return cudaErrorInvalidValue;
}

}  // namespace ttr

// ---------------------------------------------------------------- test aid
namespace ttr {

// Every CTA fills its whole dynamic shared memory with `value`; with one
// maximal CTA per SM and several waves, each SM's shared memory ends up
// holding the pattern, so a later kernel that reads shared memory it never
// wrote sees it.
__global__ void k_fill_shared(uint32_t bits, int words) {
  extern __shared__ uint32_t fill_sm[];
  volatile uint32_t* p = fill_sm;   // volatile: the stores are the point
  for (int i = threadIdx.x; i < words; i += blockDim.x) p[i] = bits;
}

}  // namespace ttr

extern "C" tt_status tt_debug_fill_shared(uint32_t bits, void* stream) {
  int dev = 0, sms = 0, maxsm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&maxsm, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
    ttr::set_last_error("tt_debug_fill_shared: device query failed");
    return TT_ECUDA;
  }
  const size_t bytes = (size_t)maxsm / 16 * 16;
  if (cudaFuncSetAttribute(ttr::k_fill_shared, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) !=
      cudaSuccess) {
    ttr::set_last_error("tt_debug_fill_shared: cudaFuncSetAttribute failed");
    return TT_ECUDA;
  }
  ttr::k_fill_shared<<<4 * sms, 1024, bytes, (cudaStream_t)stream>>>(bits, (int)(bytes / 4));
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    ttr::set_last_error(cudaGetErrorString(e));
    return TT_ECUDA;
  }
  return TT_OK;
}
