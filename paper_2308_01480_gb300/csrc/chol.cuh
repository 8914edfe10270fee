// Cholesky factorisation of a small symmetric positive definite Gram matrix
// and the inverse of its triangular factor, by one CTA in shared memory
// (used by the block orthonormalisation of Alg. 3 step 5).
#pragma once

#include "common.cuh"

namespace ttr {

// G (b x b, row stride ldg, upper triangle used) = R^T R.  R is written to
// R (row stride ldr, upper triangle; its lower triangle is zeroed) and
// T = R^{-1} (b x b, row stride ldt, upper triangular) to T.  G is destroyed.
// A pivot below 1e-6 of diag0[j] (or non-positive) raises *flag (when
// report) and is replaced by 1 so the factorisation completes.
// One barrier per column: row j of R is formed from the unscaled row j of G
// while the trailing block (rows and columns > j) is updated in place.
__device__ inline void chol_inv_cta(float* G, int ldg, int b, const float* diag0, float* R, int ldr, float* T,
                                    int ldt, int* flag, bool report, unsigned long long* badmask = nullptr) {
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = blockDim.x >> 5;
  __syncthreads();
  for (int j = 0; j < b; ++j) {
    float dj = G[j * ldg + j];
    if (!(dj > 1e-6f * diag0[j])) {
      if (report && tid == 0 && flag) atomicExch(flag, 1);
      if (badmask && tid == 0) atomicOr(badmask, 1ull << j);
      dj = 1.f;
    }
    const float rj = sqrtf(dj), inv = 1.f / rj, inv2 = inv * inv;
    for (int l = j + tid; l < b; l += blockDim.x) R[j * ldr + l] = (l == j) ? rj : G[j * ldg + l] * inv;
    for (int l = tid; l < j; l += blockDim.x) R[j * ldr + l] = 0.f;
    for (int i = j + 1 + wid; i < b; i += nw) {
      const float gi = G[j * ldg + i] * inv2;
      for (int l = i + lane; l < b; l += 32) G[i * ldg + l] -= gi * G[j * ldg + l];
    }
    __syncthreads();
  }
  // T = R^{-1}: one thread per column, back substitution in shared memory
  for (int c = tid; c < b; c += blockDim.x) {
    for (int i = b - 1; i > c; --i) T[i * ldt + c] = 0.f;
    for (int i = c; i >= 0; --i) {
      float s0 = (i == c) ? 1.f : 0.f, s1 = 0.f;
      int l = i + 1;
      for (; l + 1 <= c; l += 2) {
        s0 -= R[i * ldr + l] * T[l * ldt + c];
        s1 -= R[i * ldr + l + 1] * T[(l + 1) * ldt + c];
      }
      if (l <= c) s0 -= R[i * ldr + l] * T[l * ldt + c];
      T[i * ldt + c] = (s0 + s1) / R[i * ldr + i];
    }
  }
  __syncthreads();
}


// Cholesky factorisation G = R^T R and the triangular inverse T = R^-1 of a
// b x b Gram, b <= W (W = 16 or 32), by the first two warps of the CTA, both
// in one sweep over the columns (no triangular solve follows).
//
// Warp 0 factors.  Lane l holds column l of the upper triangle of G in a
// register window that slides down one row per step: at step j,
// a[s] = G[j + s][l], so the pivot row is always a[0] and every register
// index is a compile-time constant while the column loop runs at run time.
// Row j of R, shifted so that it starts at R[j][j + 1], goes to a
// 16-byte-aligned shared row, which every lane reads back as W / 4 vector
// broadcasts to update its window.  The next pivot needs only lane j + 1's own
// entries (G[j+1][j+1] - R[j][j+1]^2, the product the window update forms),
// so its broadcast and reciprocal square root run while the row travels.
// Warp 1 inverts, up to four rows behind (named barriers 1 .. 8, one per four
// rows: warp 0 arrives, warp 1 waits).  Lane l holds row l of V, started as
// the identity, as the window v[s] = V[l][j + s]: T[l][j] = V[l][j] / R[j][j]
// is final at step j, and V[l][j + s] -= R[j][j + s] T[l][j]
// (T[:, c] = (e_c - sum_{j < c} R[j][c] T[:, j]) / R[c][c], i.e. T R = I).
// T is staged transposed (conflict-free) and written by the whole CTA.
// Entries past row or column b are exact zeros in the shared rows and in the
// windows, so the sums run over full vectors without changing a bit of the
// result.  Pivot square roots and reciprocals use the hardware reciprocal
// square root (a few ulp), which the following Cholesky QR passes absorb.  A
// pivot below 1e-6 of diag0 (or non-positive) raises *flag when report and
// is replaced by 1.
//
// The step's latency decides the time, and one warp doing both sweeps in
// turn pays it twice: b = 30 alone took 15.1K cycles on one warp, 7.7K on two
// (bit-identical).
template <int W>
struct CholShared {
  float rows[W][W];      // rows[j][s] = R[j][j + 1 + s], zero past column b
  float inv[W];          // 1 / R[j][j]
  float Tt[W][33];       // Tt[j][l] = T[l][j]
};

template <int W>
__device__ __forceinline__ void chol_warp(CholShared<W>& sh, const float* G, int ldg, int b, const float* diag0,
                                          int* flag, bool report, unsigned long long* badmask, int bit0) {
  const unsigned full = 0xffffffffu;
  const int l = threadIdx.x & 31;
  float a[W];
#pragma unroll
  for (int i = 0; i < W; ++i) a[i] = (i <= l && l < b) ? G[i * ldg + l] : 0.f;
  const float d0 = (l < b) ? diag0[l] : 1.f;
  float djj = __shfl_sync(full, a[0], 0);
  const float dref0 = __shfl_sync(full, d0, 0);
  bool low = !(djj > 1e-6f * dref0);
  unsigned bad = low ? 1u : 0u;
  djj = low ? 1.f : djj;
  float inv = rsqrtf(djj);
#pragma unroll 1
  for (int j = 0; j < b; ++j) {
    const float rjl = (l > j) ? a[0] * inv : ((l == j) ? djj * inv : 0.f);   // R[j][l]
    // lane l > j holds entry l - j - 1; the others zero the rest of the row
    if (l < W) sh.rows[j][l > j ? l - j - 1 : W - 1 - l] = (l > j) ? rjl : 0.f;
    if (l == 0) sh.inv[j] = inv;
    __syncwarp();
    const int nx = (j + 1) & 31;
    const float cand = __shfl_sync(full, fmaf(-rjl, rjl, a[1]), nx);
    const float dref = __shfl_sync(full, d0, nx);
    const float4* rv = reinterpret_cast<const float4*>(sh.rows[j]);
    float4 r4[W / 4];
#pragma unroll
    for (int q = 0; q < W / 4; ++q) r4[q] = rv[q];
    // issue is in order: the next pivot before the window update, so that it
    // fills the wait for the row and its square root runs under the update
    low = !(cand > 1e-6f * dref);
    bad |= (low && j + 1 < b) ? (1u << nx) : 0u;
    djj = low ? 1.f : cand;
    inv = rsqrtf(djj);
#pragma unroll
    for (int q = 0; q < W / 4; ++q) {
      const float rr[4] = {r4[q].x, r4[q].y, r4[q].z, r4[q].w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int s = 4 * q + e + 1;
        if (s < W) a[s - 1] = fmaf(-rr[e], rjl, a[s]);   // G[j + s][l] -= R[j][j + s] R[j][l], slid down a row
      }
    }
    a[W - 1] = 0.f;
    if ((j & 3) == 3 || j == b - 1)
      asm volatile("bar.arrive %0, 64;\n" ::"r"(1 + (j >> 2)) : "memory");
  }
  if (report && bad && l == 0 && flag) atomicExch(flag, 1);
  if (badmask && bad && l == 0) atomicOr(badmask, (unsigned long long)bad << bit0);
}

template <int W>
__device__ __forceinline__ void inv_warp(CholShared<W>& sh, int b) {
  const int l = threadIdx.x & 31;
  float v[W];
#pragma unroll
  for (int i = 0; i < W; ++i) v[i] = (i == l && l < b) ? 1.f : 0.f;
#pragma unroll 1
  for (int j = 0; j < b; ++j) {
    if ((j & 3) == 0) asm volatile("bar.sync %0, 64;\n" ::"r"(1 + (j >> 2)) : "memory");
    const float4* rv = reinterpret_cast<const float4*>(sh.rows[j]);
    const float inv = sh.inv[j];
    float4 r4[W / 4];
#pragma unroll
    for (int q = 0; q < W / 4; ++q) r4[q] = rv[q];
    const float t = v[0] * inv;                          // T[l][j]
#pragma unroll
    for (int q = 0; q < W / 4; ++q) {
      const float rr[4] = {r4[q].x, r4[q].y, r4[q].z, r4[q].w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int s = 4 * q + e + 1;
        if (s < W) v[s - 1] = fmaf(-rr[e], t, v[s]);
      }
    }
    v[W - 1] = 0.f;
    sh.Tt[j][l] = t;
  }
}

// One per kernel, shared by both widths: no call is inside another.
__device__ __forceinline__ float* chol_shared_words() {
  static_assert(sizeof(CholShared<16>) <= sizeof(CholShared<32>), "the wide form is the larger");
  __shared__ __align__(16) float words[sizeof(CholShared<32>) / sizeof(float)];
  return words;
}
template <int W>
__device__ __forceinline__ CholShared<W>& chol_shared() {
  return *reinterpret_cast<CholShared<W>*>(chol_shared_words());
}

// Out of line (one copy per kernel, its own register allocation).
template <int W>
static __device__ __noinline__ void chol_inv_pair(CholShared<W>& sh, const float* G, int ldg, int b,
                                                  const float* diag0, int* flag, bool report,
                                                  unsigned long long* badmask, int bit0) {
  if (threadIdx.x < 32) chol_warp<W>(sh, G, ldg, b, diag0, flag, report, badmask, bit0);
  else inv_warp<W>(sh, b);
}

// Called by every thread of the CTA after a barrier: warps 0 and 1 work, then
// all threads write T (zero below the diagonal); no barrier at the end.
template <int W>
static __device__ __forceinline__ void chol_inv_cta_w(const float* G, int ldg, int b, const float* diag0, float* T,
                                                      int ldt, int* flag, bool report, unsigned long long* badmask,
                                                      int bit0) {
  CholShared<W>& sh = chol_shared<W>();
  if (threadIdx.x < 64) chol_inv_pair<W>(sh, G, ldg, b, diag0, flag, report, badmask, bit0);
  __syncthreads();
  const int lane = threadIdx.x & 31;
  if (lane < b)
    for (int r = threadIdx.x >> 5; r < b; r += blockDim.x >> 5)
      T[r * ldt + lane] = (lane >= r) ? sh.Tt[lane][r] : 0.f;
}
static __device__ __forceinline__ void chol_inv_two_warps(const float* G, int ldg, int b, const float* diag0, float* T,
                                                          int ldt, int* flag, bool report,
                                                          unsigned long long* badmask, int bit0) {
  if (b <= 16) chol_inv_cta_w<16>(G, ldg, b, diag0, T, ldt, flag, report, badmask, bit0);
  else chol_inv_cta_w<32>(G, ldg, b, diag0, T, ldt, flag, report, badmask, bit0);
}

// chol_inv_cta's contract for b <= 32 in a CTA of at least two warps, except
// that R itself is not written: the CTA synchronises, warps 0 and 1 factor and
// invert, the CTA synchronises.
__device__ __forceinline__ void chol_inv_warp32_call(const float* G, int ldg, int b, const float* diag0, float* T,
                                                     int ldt, int* flag, bool report,
                                                     unsigned long long* badmask = nullptr) {
  __syncthreads();
  chol_inv_two_warps(G, ldg, b, diag0, T, ldt, flag, report, badmask, 0);
  __syncthreads();
}

// 32 < b <= 64 in two column blocks (first 32, then b2 = b - 32), the two
// diagonal blocks by the two-warp routine and the coupling products by the
// whole CTA (of R only R12 is written):  R11 = chol(G11), T11 = R11^-1;  R12 = T11^T G12;
// G22 <- G22 - R12^T R12;  R22 = chol(G22), T22 = R22^-1;
// T12 = -(T11 R12) T22.  G (upper triangle used) is destroyed.
static __device__ __noinline__ void chol_inv_blocked64(float* G, int ldg, int b, const float* diag0, float* R, int ldr, float* T,
                                          int ldt, int* flag, bool report, unsigned long long* badmask) {
  const int tid = threadIdx.x, nt = blockDim.x, b2 = b - 32;
  __syncthreads();
  chol_inv_two_warps(G, ldg, 32, diag0, T, ldt, flag, report, badmask, 0);
  __syncthreads();
  // R12[i][c] = sum_{k <= i} T11[k][i] G[k][32 + c]; zero R21 and T21
  for (int x = tid; x < 32 * b2; x += nt) {
    const int i = x / b2, c = x % b2;
    float acc = 0.f;
    for (int k = 0; k <= i; ++k) acc = fmaf(T[k * ldt + i], G[k * ldg + 32 + c], acc);
    R[i * ldr + 32 + c] = acc;
    R[(32 + c) * ldr + i] = 0.f;
    T[(32 + c) * ldt + i] = 0.f;
  }
  __syncthreads();
  // Schur complement, upper triangle, in place
  for (int x = tid; x < b2 * b2; x += nt) {
    const int i = x / b2, c = x % b2;
    if (c < i) continue;
    float acc = G[(32 + i) * ldg + 32 + c];
    for (int k = 0; k < 32; ++k) acc = fmaf(-R[k * ldr + 32 + i], R[k * ldr + 32 + c], acc);
    G[(32 + i) * ldg + 32 + c] = acc;
  }
  __syncthreads();
  chol_inv_two_warps(G + 32 * ldg + 32, ldg, b2, diag0 + 32, T + 32 * ldt + 32, ldt, flag, report, badmask, 32);
  __syncthreads();
  // X = T11 R12 (T11 upper: k >= i) into the place of G12, which is no
  // longer needed, then T12 = -X T22 (T22 upper: k <= c)
  for (int x = tid; x < 32 * b2; x += nt) {
    const int i = x / b2, c = x % b2;
    float acc = 0.f;
    for (int k = i; k < 32; ++k) acc = fmaf(T[i * ldt + k], R[k * ldr + 32 + c], acc);
    G[i * ldg + 32 + c] = acc;
  }
  __syncthreads();
  for (int x = tid; x < 32 * b2; x += nt) {
    const int i = x / b2, c = x % b2;
    float acc = 0.f;
    for (int k = 0; k <= c; ++k) acc = fmaf(G[i * ldg + 32 + k], T[(32 + k) * ldt + 32 + c], acc);
    T[i * ldt + 32 + c] = -acc;
  }
  __syncthreads();
}

// The fastest routine for the CTA at hand (chol_inv_cta's contract, R only as
// scratch): two warps for b <= 32, two such column blocks for b <= 64.
__device__ inline void chol_inv_fast(float* G, int ldg, int b, const float* diag0, float* R, int ldr, float* T,
                                     int ldt, int* flag, bool report, unsigned long long* badmask = nullptr) {
  if (b <= 32) chol_inv_warp32_call(G, ldg, b, diag0, T, ldt, flag, report, badmask);
  else if (b <= 64) chol_inv_blocked64(G, ldg, b, diag0, R, ldr, T, ldt, flag, report, badmask);
  else chol_inv_cta(G, ldg, b, diag0, R, ldr, T, ldt, flag, report, badmask);
}

// Pivoted variant for a block that keeps only c <= b columns (the Krylov
// dimension cap): greedy symmetric pivoting on the largest remaining
// diagonal of G (b x b, full symmetric storage, row stride ldg) selects c
// columns; R (c x c, row stride ldr) is the Cholesky factor of the selected
// columns' Gram and Tf (b x bt, row stride ldt, zeroed here) maps the b
// columns to the c kept ones: Tf[perm[i]][j] = (R^{-1})[i][j] for i, j < c.
// perm (b ints of shared memory) receives the pivot order.  A pivot below
// 1e-6 of its original diagonal (or non-positive) raises *flag when report.
__device__ inline void pchol_select_cta(float* G, int ldg, int b, int c, const float* diag0, float* R, int ldr,
                                        float* Tf, int ldt, int bt, int* perm, float* dsw, int* flag,
                                        bool report, unsigned long long* badmask = nullptr) {
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = blockDim.x >> 5;
  __shared__ int s_piv;
  for (int i = tid; i < b; i += blockDim.x) {
    perm[i] = i;
    dsw[i] = diag0[i];
  }
  __syncthreads();
  for (int j = 0; j < c; ++j) {
    if (wid == 0) {
      float best = -1.f;
      int bi = j;
      for (int i = j + lane; i < b; i += 32) {
        const float v = G[i * ldg + i];
        if (v > best) { best = v; bi = i; }
      }
      for (int o = 16; o > 0; o >>= 1) {
        const float ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
      }
      if (lane == 0) s_piv = bi;
    }
    __syncthreads();
    const int pv = s_piv;
    if (pv != j) {
      // symmetric swap of rows and columns j <-> pv
      for (int l = tid; l < b; l += blockDim.x) {
        const float t = G[j * ldg + l]; G[j * ldg + l] = G[pv * ldg + l]; G[pv * ldg + l] = t;
      }
      __syncthreads();
      for (int l = tid; l < b; l += blockDim.x) {
        const float t = G[l * ldg + j]; G[l * ldg + j] = G[l * ldg + pv]; G[l * ldg + pv] = t;
      }
      if (tid == 0) {
        const int t = perm[j]; perm[j] = perm[pv]; perm[pv] = t;
        const float d = dsw[j]; dsw[j] = dsw[pv]; dsw[pv] = d;
      }
      __syncthreads();
    }
    float dj = G[j * ldg + j];
    if (!(dj > 1e-6f * dsw[j])) {
      if (report && tid == 0 && flag) atomicExch(flag, 1);
      if (badmask && tid == 0) atomicOr(badmask, 1ull << j);
      dj = 1.f;
    }
    const float rj = sqrtf(dj), inv = 1.f / rj, inv2 = inv * inv;
    for (int l = j + tid; l < c; l += blockDim.x) R[j * ldr + l] = (l == j) ? rj : G[j * ldg + l] * inv;
    for (int l = tid; l < j; l += blockDim.x) R[j * ldr + l] = 0.f;
    // full trailing update (later swaps need whole rows and columns)
    for (int i = j + 1 + wid; i < b; i += nw) {
      const float gi = G[j * ldg + i] * inv2;
      for (int l = j + 1 + lane; l < b; l += 32) G[i * ldg + l] -= gi * G[j * ldg + l];
    }
    __syncthreads();
  }
  for (int x = tid; x < b * ldt; x += blockDim.x) Tf[x] = 0.f;
  __syncthreads();
  // (R^{-1}) column by column; row i of it lands on row perm[i] of Tf
  for (int col = tid; col < c; col += blockDim.x) {
    float t[64];
    for (int i = col; i >= 0; --i) {
      float s0 = (i == col) ? 1.f : 0.f;
      for (int l = i + 1; l <= col; ++l) s0 -= R[i * ldr + l] * t[l];
      t[i] = s0 / R[i * ldr + i];
    }
    for (int i = 0; i <= col; ++i) Tf[perm[i] * ldt + col] = t[i];
  }
  (void)bt;
  __syncthreads();
}

}  // namespace ttr
