// Top-r eigenpairs of the small symmetric Rayleigh-Ritz matrix (Alg. 3
// steps 6-8), k <= 160, in two one-CTA kernels.  The first holds H in
// registers: 8 warps, thread (warp w, lane l) owning the entries
// (l + 32 a, w + 8 c), a < KT = ceil(k / 32), c < 4 KT.  The second (16
// warps, so that the register-resident Cholesky of step 4 fits) does steps
// 2-5.
//
//  1. Householder tridiagonalisation, two barriers per column (below).  The
//     reflectors go to global scratch.
//  2. Bisection by Sturm counts: one round with a count at each of 512
//     points over the Gershgorin interval, then each warp refines the
//     brackets of two wanted eigenvalues at once by three rounds of 33-point
//     multisection.
//  3. Inverse iteration on the tridiagonal T (pivoted LU), one thread per
//     wanted eigenvalue, two rounds of one solve each, and
//  4. after each round an orthonormalisation of the r vectors by Cholesky
//     QR twice (columns in descending eigenvalue order, so the result is
//     the Gram-Schmidt basis), or Gram-Schmidt twice when a Cholesky pivot
//     is too small.
//  5. Back-transformation by the stored reflectors, sixteen at a time, all
//     vectors together.
#include <float.h>

#include <utility>

#include "chol.cuh"
#include "cluster_la.cuh"
#include "common.cuh"
#include "kernels.h"
#include "sturm.cuh"

namespace ttr {

namespace {

constexpr int ER_KTMAX = 5;
constexpr int ER_TRI_WARPS = 8;          // warps of the tridiagonalisation CTA (16 measured slower)

// Compile-time loop: f(integral_constant<int, 0>) ... f(<N - 1>), so that
// register-tile indices are constants however large the unrolled body.
template <int I>
struct CIdx {
  static constexpr int value = I;
  __host__ __device__ constexpr operator int() const { return I; }
};
template <typename F, int... I>
__device__ __forceinline__ void sfor_impl(F& f, std::integer_sequence<int, I...>) {
  (f(CIdx<I>{}), ...);
}
template <int N, typename F>
__device__ __forceinline__ void sfor(F&& f) {
  sfor_impl(f, std::make_integer_sequence<int, N>{});
}

__device__ __forceinline__ float warp_min_f(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float warp_max_f(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
// Pivoted LU of T - lam I, one thread per vector: row i of w holds
// (1 / pivot, two upper diagonals, multiplier), bit i & 7 of ex[i / 8] whether
// rows were exchanged; tiny pivots replaced by +-tiny.  Rows k .. kp - 1 (kp a
// multiple of 8) are zero, so that the solves need no bounds checks.  A chain
// of k steps whose latency is the time: the exchange is a selection (lanes
// that exchange and lanes that do not would otherwise take turns) and the
// reciprocals of both candidate pivots are taken before it is known.
__device__ __forceinline__ float rcp_pivot(float p, float tiny) {
  return __fdividef(1.f, (fabsf(p) < tiny) ? copysignf(tiny, p) : p);
}
__device__ void tri_lu(const float* __restrict__ d, const float* __restrict__ e, int k, int kp, float lam, float tiny,
                       float4* __restrict__ w, uint32_t* __restrict__ ex) {
  float alpha = d[0] - lam, beta = (k > 1) ? e[0] : 0.f, sub = beta;
  uint32_t bits = 0u;
  for (int i = 0; i + 1 < k; ++i) {
    const float a1 = d[i + 1] - lam, c1 = e[i + 1];        // e[k - 1] is zero
    const float rs = rcp_pivot(sub, tiny), ra = rcp_pivot(alpha, tiny);
    const bool keep = fabsf(alpha) >= fabsf(sub);
    const float rp = keep ? ra : rs;
    const float li = (keep ? sub : alpha) * rp;
    const float up = keep ? beta : a1, lo = keep ? a1 : beta;
    w[i] = make_float4(rp, up, keep ? 0.f : c1, li);
    bits |= keep ? 0u : (1u << (i & 7));
    if ((i & 7) == 7) {
      ex[i >> 3] = bits;
      bits = 0u;
    }
    alpha = fmaf(-li, up, lo);
    beta = keep ? c1 : -li * c1;
    sub = c1;
  }
  w[k - 1] = make_float4(rcp_pivot(alpha, tiny), 0.f, 0.f, 0.f);
  ex[(k - 1) >> 3] = bits;
  for (int i = k; i < kp; ++i) w[i] = make_float4(0.f, 0.f, 0.f, 0.f);
}

// x <- (T - lam I)^-1 x (x zero from k to kp), returning max |x_i|; eight rows
// of the factors and of x in registers at a time, since a store to x between
// two loads would make each row wait for shared memory.
__device__ float tri_lu_solve(const float4* __restrict__ w, const uint32_t* __restrict__ ex, int kp,
                              float* __restrict__ x) {
  float xi = x[0];
  for (int i0 = 0; i0 < kp; i0 += 8) {
    float lv[8], xn[8];
    const uint32_t bits = ex[i0 >> 3];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      lv[q] = w[i0 + q].w;
      xn[q] = x[i0 + q + 1];
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const bool swap = bits & (1u << q);
      const float top = swap ? xn[q] : xi, low = swap ? xi : xn[q];
      xn[q] = top;
      xi = fmaf(-lv[q], top, low);
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) x[i0 + q] = xn[q];
  }
  float x1 = 0.f, x2 = 0.f, mx = 0.f;
  for (int i0 = kp - 8; i0 >= 0; i0 -= 8) {
    float4 f[8];
    float xv[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      f[q] = w[i0 + q];
      xv[q] = x[i0 + q];
    }
#pragma unroll
    for (int q = 7; q >= 0; --q) {
      const float v = fmaf(-f[q].y, x1, fmaf(-f[q].z, x2, xv[q])) * f[q].x;
      xv[q] = v;
      mx = fmaxf(mx, fabsf(v));
      x2 = x1;
      x1 = v;
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) x[i0 + q] = xv[q];
  }
  return mx;
}

}  // namespace

// Reflectors per group of the back-transformation.
constexpr int ER_GB = 16;

// Shared memory of k_eig_vectors (float offsets).  The vectors' rows have an
// odd stride and the inverse-iteration factors' rows one of 4 mod 32 floats:
// one thread per vector walks its row, so neither meets a bank conflict.  The
// vectors' rows are zero from k on (up to 32 KT and one more).
struct ErLayout {
  int ldx, ldw, kp, groups;
  size_t V, tau, d, e, de, lam, red, cnt, ex, X, X2, G, T, S, D, C, total;
};
__host__ __device__ inline ErLayout er_layout(int KM, int k, int r) {
  ErLayout L;
  L.kp = (k + 7) & ~7;
  L.ldx = KM + 1;
  L.ldw = 4 * ((L.kp + 7) & ~7) + 4;
  L.groups = k > 2 ? (k - 2 + ER_GB - 1) / ER_GB : 0;
  size_t o = 0;
  auto take = [&](size_t n) { const size_t at = o; o += (n + 3) & ~size_t(3); return at; };
  // the reflectors (step 5) and the inverse-iteration factors (step 3) are
  // never live together: one region holds both.  Reads of whole 32-entry
  // chunks run up to 31 floats past the last reflector, which are zeroed.
  const size_t v = (size_t)k * k + 32, w = (size_t)r * L.ldw;
  L.V = take(v > w ? v : w);
  L.tau = take(KM);
  L.d = take(KM);
  L.e = take(KM);
  L.de = take(2 * (size_t)(KM + 4) + 4) + 2;   // de + 1 on a 16-byte boundary
  L.lam = take(32);
  L.red = take(64);
  L.cnt = take(512);
  L.ex = take(32 * 21);
  L.X = take((size_t)r * L.ldx);
  L.X2 = take((size_t)r * L.ldx);
  L.G = take(36 * 33);
  L.T = take(33 * 32);
  L.S = take((size_t)L.groups * ER_GB * (ER_GB + 1));
  L.D = take(ER_GB * 36);
  L.C = take(ER_GB * 36);
  L.total = o + 4;       // the last word: a flag
  return L;
}

// Sum over the 32 lanes of NV values x[0..NV) (NV a power of two <= 32) with
// the transposing butterfly: at each level a lane keeps half of its values
// and sends the other half, so after log2(NV) levels every lane holds one
// partial sum; the remaining levels are plain butterflies.  Lane l ends with
// the total of value (l >> (5 - log2 NV)).
template <int NV>
__device__ __forceinline__ float lane_transpose_sum(float (&x)[NV]) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  float cur[NV];
  sfor<NV>([&](auto i) { cur[i] = x[i]; });
  int n = NV, o = 16;
  // levels that halve the value count (compile-time sizes via sfor)
  sfor<5>([&](auto lvl) {
    constexpr int L = decltype(lvl)::value;
    constexpr int N = NV >> L;          // values held before this level
    if constexpr (N >= 2) {
      constexpr int H = N / 2;
      const int off = 16 >> L;
      const bool up = lane & off;
      sfor<H>([&](auto i) {
        const float send = up ? cur[i] : cur[i + H];
        const float keep = up ? cur[i + H] : cur[i];
        cur[i] = keep + __shfl_xor_sync(full, send, off);
      });
    } else {
      const int off = 16 >> L;
      cur[0] += __shfl_xor_sync(full, cur[0], off);
    }
  });
  (void)n;
  (void)o;
  return cur[0];
}

// Step 1 in one CTA of 8 warps: T = (d, e) and the reflectors (row j of
// Vg = v_j, tau[j]) to global scratch.  Thread (warp w, lane l) holds the
// entries (l + 32 a, w + 8 c), a < KR, c < 4 KR, so every column lives in one
// warp and each thread carries 20 KR entries (the per-column reductions,
// broadcasts and barriers are spread over many multiply-adds).  Per column
// two barriers:
//   M  every warp forms tau (H v)_c for its columns c (H is symmetric, so the
//      column dot is the row product) and its share of v^T H v, reduced over
//      the lanes by one transposing butterfly;
//   U  every thread applies H -= v w^T + w v^T, w = p - (tau/2)(v^T p) v,
//      to its entries of the trailing block: the four column slots that hold
//      the next column first, then
//   R  the warp owning the next column forms its reflector (v and tau) from
//      its registers and publishes it while the others finish U.
// The column time is the chain barrier, M, barrier, the next column's update,
// R; v and p are kept in shared memory in column order and, for the 20
// broadcasts of a warp's own columns, also warp by warp, so that five
// 16-byte loads fetch them.  With R after all of U, scalar broadcasts and three
// operations per entry in U a column of k = 150 took 1,300 (late) to 3,100
// (early) cycles, 139 us in all; 1,050 to 2,500 and 122 us so.
// Tiles of finished rows (32-row blocks) and columns (8-column slots) are
// skipped at compile time: the column loop is split into 32-column segments.
template <int KR, int NW>
__global__ void __launch_bounds__(NW * 32, 1) k_eig_tridiag8(const float* __restrict__ Hin, int64_t ldh, int k,
                                                        float* __restrict__ Vg, float* __restrict__ tau_g,
                                                        float* __restrict__ d_g, float* __restrict__ e_g) {
  constexpr int SPS = 32 / NW;            // column slots per warp in a 32-column segment
  constexpr int KC = SPS * KR;
  constexpr int KM = 32 * KR;
  static_assert(SPS == 4, "a segment's slots of a warp are one 16-byte load");
  __shared__ __align__(16) float vs[2][KM];    // v in column order
  __shared__ __align__(16) float vw[2][KM];    // v, warp by warp: entry (i % NW) KC + i / NW
  __shared__ __align__(16) float ps[KM];
  __shared__ __align__(16) float pw[KM];
  __shared__ float wsum[NW];
  __shared__ float scal[2];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;

  float A[KR][KC];   // A[a][c] = H[lane + 32 a][w + NW c]
  sfor<KR>([&](auto a) {
    sfor<KC>([&](auto c) {
      const int i = lane + 32 * a, j = w + NW * c;
      A[a][c] = (i < k && j < k) ? 0.5f * (Hin[(int64_t)i * ldh + j] + Hin[(int64_t)j * ldh + i]) : 0.f;
    });
  });
  const int z0 = (k >= 2) ? (k - 2) * k : 0;
  for (int x = z0 + tid; x < k * k; x += NW * 32) Vg[x] = 0.f;
  sfor<KR>([&](auto seg) {
    constexpr int S = decltype(seg)::value;
    const int jend = min(32 * S + 32, k - 2);
    // R: the reflector of column j (slot j / NW of warp j % NW, inside this segment)
    auto reflector = [&](int j) {
      const int t = (j / NW) - SPS * S;   // 0 .. SPS - 1
      float colv[KR];
      sfor<KR>([&](auto a) {
        float x = 0.f;
        if constexpr (a >= S) {
          sfor<SPS>([&](auto u) {
            if (t == u) x = A[a][SPS * S + u];
          });
        }
        colv[a] = x;
      });
      float part = 0.f, sel = 0.f;
      const int a1 = (j + 1) >> 5;
      sfor<KR>([&](auto a) {
        if constexpr (a >= S) {
          const float x = colv[a];
          const int i = lane + 32 * a;
          if (i >= j + 2 && i < k) part = fmaf(x, x, part);
          if (a == a1) sel = x;
        }
      });
      const float x0 = __shfl_sync(0xffffffffu, sel, (j + 1) & 31);
      const float sigma = warp_sum(part);
      float tt = 0.f, iv = 0.f, beta = x0;
      if (sigma > 0.f) {
        const float s2 = fmaf(x0, x0, sigma);
        const float mu = s2 * rsqrtf(s2);
        const float v0 = (x0 <= 0.f) ? x0 - mu : __fdividef(-sigma, x0 + mu);
        tt = __fdividef(2.f * v0 * v0, fmaf(v0, v0, sigma));
        beta = mu;
        iv = __fdividef(1.f, v0);
      }
      float v[KR];
      sfor<KR>([&](auto a) {
        const int i = lane + 32 * a;
        v[a] = (a < S) ? 0.f : ((i == j + 1) ? 1.f : ((i > j + 1 && i < k) ? colv[a] * iv : 0.f));
        vs[j & 1][i] = v[a];
        vw[j & 1][(lane % NW) * KC + (lane / NW) + SPS * a] = v[a];
      });
      if (lane == 0) {
        scal[j & 1] = tt;
        tau_g[j] = tt;
        e_g[j] = beta;
      }
      sfor<KR>([&](auto a) {
        const int i = lane + 32 * a;
        if (i < k) Vg[(size_t)j * k + i] = (tt != 0.f) ? v[a] : 0.f;
        if constexpr (a >= S) {
          if (i == j) d_g[j] = colv[a];
        }
      });
    };
    if (32 * S < jend && w == (32 * S) % NW) reflector(32 * S);
    for (int j = 32 * S; j < jend; ++j) {
      __syncthreads();
      const float tau = scal[j & 1];
      const bool next = j + 1 < jend && w == ((j + 1) % NW);
      if (tau == 0.f) {                      // the same decision in every thread
        if (next) reflector(j + 1);
        continue;
      }
      // M: (H v)_c for this thread's live columns, its share of v^T H v
      constexpr int LIVE = KC - SPS * S;
      float vr[KR], vc[KC];
      sfor<KR>([&](auto a) { vr[a] = (a >= S) ? vs[j & 1][lane + 32 * a] : 0.f; });
      sfor<KR>([&](auto q) {
        if constexpr (q >= S) {
          const float4 x = *reinterpret_cast<const float4*>(&vw[j & 1][w * KC + 4 * q]);
          vc[4 * q] = x.x; vc[4 * q + 1] = x.y; vc[4 * q + 2] = x.z; vc[4 * q + 3] = x.w;
        } else {
          vc[4 * q] = vc[4 * q + 1] = vc[4 * q + 2] = vc[4 * q + 3] = 0.f;
        }
      });
      float hv[LIVE], part = 0.f;
      sfor<LIVE>([&](auto c) {
        float acc = 0.f;
        sfor<KR>([&](auto a) {
          if constexpr (a >= S) acc = fmaf(A[a][SPS * S + c], vr[a], acc);
        });
        hv[c] = acc;
        part = fmaf(vc[SPS * S + c], acc, part);
      });
      // lane totals of the live columns in butterflies of 16, 8 or 4
      auto publish = [&](auto first, auto count) {
        constexpr int F = decltype(first)::value, N = decltype(count)::value;
        float x[N];
        sfor<N>([&](auto c) {
          if constexpr (F + c < LIVE) x[c] = hv[F + c];
          else x[c] = 0.f;
        });
        const float tot = lane_transpose_sum<N>(x);
        constexpr int shift = (N == 16) ? 1 : (N == 8) ? 2 : 3;
        const int vi = SPS * S + F + (lane >> shift);
        if ((lane & ((1 << shift) - 1)) == 0 && vi < KC) {
          const int col = w + NW * vi;
          const float pv = (col > j && col < k) ? tau * tot : 0.f;
          ps[col] = pv;
          pw[w * KC + vi] = pv;
        }
      };
      if constexpr (LIVE > 16) {
        publish(CIdx<0>{}, CIdx<16>{});
        publish(CIdx<16>{}, CIdx<4>{});
      } else if constexpr (LIVE > 8) {
        publish(CIdx<0>{}, CIdx<16>{});
      } else if constexpr (LIVE > 4) {
        publish(CIdx<0>{}, CIdx<8>{});
      } else {
        publish(CIdx<0>{}, CIdx<4>{});
      }
      const float share = warp_sum(part);
      if (lane == 0) wsum[w] = share;
      __syncthreads();
      // U: rank-2 update of the live tiles
      float vhv = 0.f;
#pragma unroll
      for (int q = 0; q < NW; ++q) vhv += wsum[q];
      const float K = 0.5f * tau * tau * vhv;
      float wr[KR], wc[KC];
      sfor<KR>([&](auto a) { wr[a] = (a >= S) ? fmaf(-K, vr[a], ps[lane + 32 * a]) : 0.f; });
      sfor<KR>([&](auto q) {
        if constexpr (q >= S) {
          const float4 x = *reinterpret_cast<const float4*>(&pw[w * KC + 4 * q]);
          wc[4 * q] = fmaf(-K, vc[4 * q], x.x);
          wc[4 * q + 1] = fmaf(-K, vc[4 * q + 1], x.y);
          wc[4 * q + 2] = fmaf(-K, vc[4 * q + 2], x.z);
          wc[4 * q + 3] = fmaf(-K, vc[4 * q + 3], x.w);
        }
      });
      auto update = [&](auto c) {
        sfor<KR>([&](auto a) {
          if constexpr (a >= S) {
            A[a][c] = fmaf(-vr[a], wc[c], A[a][c]);
            A[a][c] = fmaf(-wr[a], vc[c], A[a][c]);
          }
        });
      };
      sfor<SPS>([&](auto u) { update(CIdx<SPS * S + decltype(u)::value>{}); });
      if (next) reflector(j + 1);
      sfor<KC>([&](auto c) {
        if constexpr (c >= SPS * S + SPS) update(c);
      });
    }
    __syncthreads();                         // the last column's p and v are read before the next segment's
  });
  // trailing 2 x 2 (or 1 x 1) block, written by the owners of its entries
  sfor<KR>([&](auto a) {
    sfor<KC>([&](auto c) {
      const int i = lane + 32 * a, jj = w + NW * c;
      if (k >= 2 && i == k - 2 && jj == k - 2) d_g[k - 2] = A[a][c];
      if (k >= 2 && i == k - 1 && jj == k - 2) e_g[k - 2] = A[a][c];
      if (i == k - 1 && jj == k - 1) d_g[k - 1] = A[a][c];
    });
  });
  if (tid == 0) {
    if (k >= 2) tau_g[k - 2] = 0.f;
    e_g[k - 1] = 0.f;
    tau_g[k - 1] = 0.f;
  }
}

// sum_i a[u][i] b[v][i] of four rows with four rows, lanes along i, for the
// 32-entry chunks c0 .. KT - 1 (rows of b zero past their end): all loads
// unconditional (a condition on each made an inner product of 150 entries
// take 3.2K cycles).  put(u, v, total) is called by one lane in two.
template <int KT, typename Put>
__device__ __forceinline__ void warp_dots4(const float* const (&a)[4], const float* const (&b)[4], int c0, Put put) {
  const int lane = threadIdx.x & 31;
  float acc[16];
#pragma unroll
  for (int t = 0; t < 16; ++t) acc[t] = 0.f;
#pragma unroll
  for (int c = 0; c < KT; ++c) {
    if (c >= c0) {                       // warp-uniform
      float x[4], y[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) x[u] = a[u][32 * c + lane];
#pragma unroll
      for (int u = 0; u < 4; ++u) y[u] = b[u][32 * c + lane];
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[4 * u + v] = fmaf(x[u], y[v], acc[4 * u + v]);
    }
  }
  const float tot = lane_transpose_sum<16>(acc);
  if (!(lane & 1)) put(lane >> 3, (lane >> 1) & 3, tot);
}

// Steps 2-5 in one CTA of 16 warps, from T and the reflectors in global
// scratch (the reflectors are staged in shared memory).  Every step is a
// chain of short dependent operations, so latency decides: k = 150, r = 20
// took 238K cycles (115 us) with divided Sturm ratios, branching LU, bounds
// checks in the solves and one thread per inner product, 157K (77 us) so.
template <int KT>
__global__ void __launch_bounds__(512, 1) k_eig_vectors(const float* __restrict__ Vg, const float* __restrict__ tau_g,
                                                       const float* __restrict__ d_g, const float* __restrict__ e_g,
                                                       int k, int r, float* __restrict__ V, int ldv,
                                                       float* __restrict__ evals) {
  constexpr int NW = 16;
  constexpr int KM = 32 * KT;
  constexpr int NT = 32 * NW;
  extern __shared__ __align__(16) float sm[];
  const ErLayout L = er_layout(KM, k, r);
  float* Vs = sm + L.V;                   // [k][k], row j = reflector v_j
  float* Wk = sm + L.V;                   // [r][ldw] inverse-iteration factors, rows of float4
  uint32_t* exb = reinterpret_cast<uint32_t*>(sm + L.ex);   // [r][21] exchange bits
  float* tau = sm + L.tau;
  float* d = sm + L.d;
  float* e = sm + L.e;
  float2* de = reinterpret_cast<float2*>(sm + L.de);   // scaled (d_i, e_{i-1}^2)
  float* lam = sm + L.lam;
  float* red = sm + L.red;
  int* cnt = reinterpret_cast<int*>(sm + L.cnt);       // [512]
  float* G = sm + L.G;                    // [32][33]
  float* Tm = sm + L.T;                   // [32][33]
  int* sflag = reinterpret_cast<int*>(sm + L.total - 4);
  const int tid = threadIdx.x, lane = tid & 31, ty = tid >> 5;
  const int ldx = L.ldx;
  for (int i = tid; i < k; i += NT) {
    tau[i] = tau_g[i];
    d[i] = d_g[i];
    e[i] = e_g[i];
  }
  if (tid == 0) *sflag = 0;
  __syncthreads();

  // ---------------------------------------------------------------- 2
  float glo = FLT_MAX, ghi = -FLT_MAX, amax = 0.f;
  for (int i = tid; i < k; i += NT) {
    const float off = (i > 0 ? fabsf(e[i - 1]) : 0.f) + fabsf(e[i]);
    glo = fminf(glo, d[i] - off);
    ghi = fmaxf(ghi, d[i] + off);
    amax = fmaxf(amax, fmaxf(fabsf(d[i]), fabsf(e[i])));
  }
  glo = warp_min_f(glo);
  ghi = warp_max_f(ghi);
  amax = warp_max_f(amax);
  if (lane == 0) {
    red[ty] = glo;
    red[32 + ty] = ghi;
    cnt[ty] = __float_as_int(amax);
  }
  __syncthreads();
  glo = warp_min_f(lane < NW ? red[lane] : FLT_MAX);
  ghi = warp_max_f(lane < NW ? red[32 + lane] : -FLT_MAX);
  amax = warp_max_f(lane < NW ? __int_as_float(cnt[lane]) : 0.f);
  const float tnorm = fmaxf(amax, FLT_MIN);
  const float pivmin = FLT_MIN * fmaxf(1.f, tnorm * tnorm);
  // T scaled by a power of two (exact) to largest entry in [1, 2)
  const unsigned ex = min(__float_as_uint(tnorm) & 0x7f800000u, 0x7e800000u);
  const float up = __uint_as_float(0x7f000000u - ex), down = __uint_as_float(ex);
  const int groups4 = (k + 2) / 4;        // 1 + 4 groups4 >= k rows
  for (int i = tid; i < 1 + 4 * groups4; i += NT) {
    de[i] = (i < k) ? sturm_row(d[i] * up, i > 0 ? e[i - 1] * up : 0.f) : sturm_row(16.f, 0.f);
  }
  __syncthreads();
  const float pad = 4.f * FLT_EPSILON;
  const float lo0 = glo * up - pad, hi0 = ghi * up + pad;
  const float step = (hi0 - lo0) * (1.f / (float)(NT + 1));
  cnt[tid] = sturm(de, groups4, fmaf((float)(tid + 1), step, lo0));
  __syncthreads();
  // a warp refines the brackets of eigenvalues ty and ty + NW together
  // (two independent Sturm chains in flight)
  {
    const int j0 = ty, j1 = ty + NW;
    const bool has0 = j0 < r, has1 = j1 < r;
    auto bracket = [&](int jj, float& lo, float& hi) {
      const int want = k - jj;             // count reaching k - j brackets the j-th largest
      int first = NT;
#pragma unroll
      for (int u = NW - 1; u >= 0; --u) {
        const unsigned ge = __ballot_sync(0xffffffffu, cnt[32 * u + lane] >= want);
        if (ge) first = 32 * u + __ffs(ge) - 1;
      }
      lo = (first == 0) ? lo0 : fmaf((float)first, step, lo0);
      hi = (first == NT) ? hi0 : fmaf((float)(first + 1), step, lo0);
    };
    auto narrow = [&](int c, int want, float x, float& lo, float& hi) {
      const unsigned ge = __ballot_sync(0xffffffffu, c >= want);
      const int sidx = ge ? (__ffs(ge) - 1) : 32;
      const float xs = __shfl_sync(0xffffffffu, x, sidx < 32 ? sidx : 31);
      const float xp = __shfl_sync(0xffffffffu, x, sidx > 0 ? sidx - 1 : 0);
      if (sidx == 32) lo = xs;
      else {
        hi = xs;
        if (sidx > 0) lo = xp;
      }
    };
    float lo_0 = 0.f, hi_0 = 0.f, lo_1 = 0.f, hi_1 = 0.f;
    if (has0) bracket(j0, lo_0, hi_0);
    if (has1) bracket(j1, lo_1, hi_1);
    // three rounds: the bracket is then (span / 513) / 33^3 ~ 5e-8 of the
    // Gershgorin span, the resolution of FP32 itself
    for (int it = 0; it < 3 && has0; ++it) {
      const float x0 = lo_0 + (hi_0 - lo_0) * (float)(lane + 1) * (1.f / 33.f);
      if (has1) {
        const float x1 = lo_1 + (hi_1 - lo_1) * (float)(lane + 1) * (1.f / 33.f);
        int c0, c1;
        sturm2(de, groups4, x0, x1, c0, c1);
        narrow(c0, k - j0, x0, lo_0, hi_0);
        narrow(c1, k - j1, x1, lo_1, hi_1);
      } else {
        narrow(sturm(de, groups4, x0), k - j0, x0, lo_0, hi_0);
      }
    }
    if (lane == 0 && has0) lam[j0] = 0.5f * (lo_0 + hi_0) * down;
    if (lane == 0 && has1) lam[j1] = 0.5f * (lo_1 + hi_1) * down;
  }

  // ---------------------------------------------------------------- 3
  // Two rounds of one inverse-iteration solve per vector followed by an
  // orthonormalisation of all r vectors (a subspace iteration): for nearly
  // equal eigenvalues the solves pull every vector towards the same
  // eigenvector, and orthonormalising after each single solve keeps the
  // remainders inside the cluster's invariant subspace.
  const float tiny = FLT_EPSILON * tnorm + pivmin;
  float* cur = sm + L.X;                  // [r][ldx]
  float* nxt = sm + L.X2;                 // [r][ldx]
  // start vector 1 + 0.01 h(j, i), h pseudo-random in [-1, 1) and different
  // for every vector: equal shifts (a cluster below FP32 resolution) must
  // not produce equal vectors
  for (int j = ty; j < r; j += NW)
    for (int i = lane; i < ldx; i += 32) {
      cur[(size_t)j * ldx + i] = (i < k) ? fmaf(0.01f, hash_uniform(0xE16ull + (uint64_t)j, (uint64_t)i), 1.f) : 0.f;
      nxt[(size_t)j * ldx + i] = 0.f;
    }
  __syncthreads();
  for (int round = 0; round < 2; ++round) {
    if (tid < r) {
      float4* w = reinterpret_cast<float4*>(Wk + (size_t)tid * L.ldw);
      uint32_t* ex = exb + tid * 21;
      if (round == 0) tri_lu(d, e, k, L.kp, lam[tid], tiny, w, ex);
      const float mx = tri_lu_solve(w, ex, L.kp, cur + (size_t)tid * ldx);
      red[tid] = mx > 0.f ? 1.f / mx : 0.f;
    }
    if (tid == 0) *sflag = 0;
    __syncthreads();
    for (int j = ty; j < r; j += NW)
      for (int i = lane; i < k; i += 32) cur[(size_t)j * ldx + i] *= red[j];
    // the factors are dead after the last solve: stage the reflectors for
    // step 5 in their place while step 4 runs
    if (round == 1) {
      const int n4 = k * k / 4;
      for (int x = tid; x < n4; x += NT) cp_async16(Vs + 4 * x, Vg + 4 * x);
      for (int x = 4 * n4 + tid; x < k * k; x += NT) cp_async4(Vs + x, Vg + x, true);
      if (tid < 32) Vs[k * k + tid] = 0.f;
    }
    __syncthreads();

  // ---------------------------------------------------------------- 4
    // one Cholesky QR pass keeps the vectors apart before the second solve;
    // two make the final ones orthonormal to working accuracy
    for (int pass = 0; pass < (round == 0 ? 1 : 2); ++pass) {
      // upper triangle of the Gram in 4 x 4 tiles, a warp each
      const int nb = (r + 3) / 4;
      for (int t = ty; t < nb * (nb + 1) / 2; t += NW) {
        int tb = 0;
        while ((tb + 1) * (tb + 2) / 2 <= t) ++tb;
        const int ta = t - tb * (tb + 1) / 2;
        const float* ra[4];
        const float* rb[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {     // rows past r repeat the last one; their sums are not used
          ra[u] = cur + (size_t)min(4 * ta + u, r - 1) * ldx;
          rb[u] = cur + (size_t)min(4 * tb + u, r - 1) * ldx;
        }
        warp_dots4<KT>(ra, rb, 0, [&](int u, int v, float s) { G[(4 * ta + u) * 33 + 4 * tb + v] = s; });
      }
      __syncthreads();
      if (round == 1 && pass == 1) {
        // after one Cholesky QR the Gram is usually within rounding of the
        // identity: then X (1.5 I - 0.5 G) (first-order polar correction,
        // orthogonality error O(|G - I|^2), same span) replaces the second
        float dev = 0.f;
        for (int x = tid; x < r * r; x += NT) {
          const int a = x / r, b = x % r;
          if (b >= a) dev = fmaxf(dev, fabsf(G[a * 33 + b] - (a == b ? 1.f : 0.f)));
        }
        dev = warp_max_f(dev);
        if (lane == 0) red[32 + ty] = dev;
        __syncthreads();
        dev = warp_max_f(lane < NW ? red[32 + lane] : 0.f);
        if (dev < 1e-4f) {                // the same decision in every thread
          for (int x = tid; x < r * r; x += NT) {
            const int a = x / r, b = x % r;
            const float g = (b >= a) ? G[a * 33 + b] : G[b * 33 + a];
            Tm[a * 33 + b] = (a == b ? 1.5f : 0.f) - 0.5f * g;
          }
          __syncthreads();
          for (int j = ty; j < r; j += NW) {
            float s[KT];
#pragma unroll
            for (int c = 0; c < KT; ++c) s[c] = 0.f;
#pragma unroll 4
            for (int a = 0; a < r; ++a) {
              const float t = Tm[a * 33 + j];
#pragma unroll
              for (int c = 0; c < KT; ++c)
                if (lane + 32 * c < k) s[c] = fmaf(cur[(size_t)a * ldx + lane + 32 * c], t, s[c]);
            }
#pragma unroll
            for (int c = 0; c < KT; ++c)
              if (lane + 32 * c < k) nxt[(size_t)j * ldx + lane + 32 * c] = s[c];
          }
          __syncthreads();
          float* tmp = cur; cur = nxt; nxt = tmp;
          continue;
        }
        __syncthreads();
      }
      if (tid < r) red[tid] = G[tid * 33 + tid];
      chol_inv_warp32_call(G, 33, r, red, Tm, 33, sflag, true);
      if (*sflag) break;                  // uniform: fall back below
      // nxt[j][i] = sum_{a <= j} cur[a][i] T[a][j]
      for (int j = ty; j < r; j += NW) {
        float s[KT];
#pragma unroll
        for (int c = 0; c < KT; ++c) s[c] = 0.f;
#pragma unroll 4
        for (int a = 0; a <= j; ++a) {
          const float t = Tm[a * 33 + j];
#pragma unroll
          for (int c = 0; c < KT; ++c)
            if (lane + 32 * c < k) s[c] = fmaf(cur[(size_t)a * ldx + lane + 32 * c], t, s[c]);
        }
#pragma unroll
        for (int c = 0; c < KT; ++c)
          if (lane + 32 * c < k) nxt[(size_t)j * ldx + lane + 32 * c] = s[c];
      }
      __syncthreads();
      float* tmp = cur; cur = nxt; nxt = tmp;
    }
    if (*sflag) {
      // Gram-Schmidt twice in descending eigenvalue order (a Cholesky pass
      // that was applied leaves the span of each leading set unchanged)
      for (int j = 0, attempt = 0; j < r;) {
        float* xj = cur + (size_t)j * ldx;
        float p0 = 0.f;
        for (int i = tid; i < k; i += NT) p0 = fmaf(xj[i], xj[i], p0);
        const float n0 = sqrtf(block_sum(p0, red));
        __syncthreads();
        for (int pass = 0; pass < 2 && j > 0; ++pass) {
          for (int i2 = ty; i2 < j; i2 += NW) {
            const float* xi = cur + (size_t)i2 * ldx;
            float pp = 0.f;
            for (int i = lane; i < k; i += 32) pp = fmaf(xi[i], xj[i], pp);
            pp = warp_sum(pp);
            if (lane == 0) G[i2] = pp;
          }
          __syncthreads();
          for (int i = tid; i < k; i += NT) {
            float s0 = xj[i];
            for (int i2 = 0; i2 < j; ++i2) s0 = fmaf(-G[i2], cur[(size_t)i2 * ldx + i], s0);
            xj[i] = s0;
          }
          __syncthreads();
        }
        float pp = 0.f;
        for (int i = tid; i < k; i += NT) pp = fmaf(xj[i], xj[i], pp);
        const float nrm = sqrtf(block_sum(pp, red));
        __syncthreads();
        if (!(nrm > 1e-4f * n0) && attempt < 3) {
          // numerically inside the span of the earlier vectors (a cluster
          // below FP32 resolution): any direction orthogonal to them serves,
          // take a pseudo-random one through the same projections
          for (int i = tid; i < k; i += NT)
            xj[i] = hash_uniform(0x65A0ull + 64ull * (uint64_t)attempt + (uint64_t)j, (uint64_t)i);
          __syncthreads();
          ++attempt;
          continue;
        }
        const float inv = nrm > 0.f ? 1.f / nrm : 0.f;
        for (int i = tid; i < k; i += NT) xj[i] *= inv;
        __syncthreads();
        ++j;
        attempt = 0;
      }
    }
    __syncthreads();
  }

  // ---------------------------------------------------------------- 5
  // x <- P_0 P_1 ... P_{k-3} x for the r vectors, ER_GB reflectors at a time
  // from the last.  For the reflectors of a group in the order of their
  // application (q = 0 the highest index), c_q = tau_q (v_q^T x - sum_{p < q}
  // (v_q^T v_p) c_p) and x -= sum_q c_q v_q, so c = S D with D = [v_q^T x] and
  // a triangular S that depends on the reflectors alone: all S first, a warp
  // per group, then three small products per group for all vectors at once.
  // v_h is zero at indices <= h (and entirely where tau_h = 0), so a group
  // starts at its lowest reflector.
  cp_async_wait_all();
  __syncthreads();
  {
    constexpr int GB = ER_GB, LS = GB + 1;
    float* Sg = sm + L.S;                 // [groups][GB][LS]
    float* Dm = sm + L.D;                 // [GB][36]
    float* Cm = sm + L.C;                 // [GB][36]
    const int ng = L.groups;
    auto top = [&](int g) { return k - 3 - GB * g; };       // highest reflector of group g
    auto size = [&](int g) { return min(GB, top(g) + 1); };
    // Reads of a reflector's last chunk run past its k entries into the next
    // reflector: the vectors are zero there, and the reflectors' own products
    // mask one side.
    // inner products of each group's reflectors, rows in application order
    // (row q is reflector top - q; past the group, the zero row k - 1)
    constexpr int NTL = (GB / 4) * (GB / 4 + 1) / 2;
    for (int t = ty; t < ng * NTL; t += NW) {
      const int g = t / NTL, tl = t % NTL;
      int ta = 0;
      while ((ta + 1) * (ta + 2) / 2 <= tl) ++ta;
      const int tb = tl - ta * (ta + 1) / 2;              // p <= q
      const int h = top(g), n = size(g);
      float* S = Sg + (size_t)g * GB * LS;
      float acc[16];
#pragma unroll
      for (int x = 0; x < 16; ++x) acc[x] = 0.f;
      const int c0 = (h - n + 2) >> 5;
#pragma unroll
      for (int c = 0; c < KT; ++c)
        if (c >= c0) {
          const int i = 32 * c + lane;
          float x[4], y[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            x[u] = Vs[(size_t)((4 * ta + u < n) ? h - 4 * ta - u : k - 1) * k + i];
            y[u] = Vs[(size_t)((4 * tb + u < n) ? h - 4 * tb - u : k - 1) * k + i];
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) x[u] = (i < k) ? x[u] : 0.f;
#pragma unroll
          for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v < 4; ++v) acc[4 * u + v] = fmaf(x[u], y[v], acc[4 * u + v]);
        }
      const float tot = lane_transpose_sum<16>(acc);
      if (!(lane & 1)) S[(4 * ta + (lane >> 3)) * LS + 4 * tb + ((lane >> 1) & 3)] = tot;
    }
    __syncthreads();
    // S by forward substitution, lane = column: S[q][c] = tau_q ([q == c] -
    // sum_{c <= p < q} g_qp S[p][c])
    for (int g = ty; g < ng; g += NW) {
      float* S = Sg + (size_t)g * GB * LS;
      const int h = top(g), n = size(g);
      float col[GB];
#pragma unroll
      for (int q = 0; q < GB; ++q) {
        float s0 = (q == lane) ? 1.f : 0.f, s1 = 0.f;
#pragma unroll
        for (int p = 0; p < q; ++p) {
          const float gp = (q < n) ? S[q * LS + p] : 0.f;
          if (p & 1) s1 = fmaf(-gp, col[p], s1);
          else s0 = fmaf(-gp, col[p], s0);
        }
        col[q] = (q < n) ? tau[h - q] * (s0 + s1) : 0.f;
      }
      __syncwarp();
      if (lane < GB) {
#pragma unroll
        for (int q = 0; q < GB; ++q) S[q * LS + lane] = col[q];
      }
    }
    __syncthreads();
    const int nv = (r + 3) / 4;
    for (int g = 0; g < ng; ++g) {
      const int h = top(g), n = size(g), i0 = (h - n + 2) & ~31;
      const float* S = Sg + (size_t)g * GB * LS;
      for (int t = ty; t < (GB / 4) * nv; t += NW) {
        const int ta = t / nv, tb = t % nv;
        const float* ra[4];
        const float* rb[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          ra[u] = Vs + (size_t)((4 * ta + u < n) ? h - 4 * ta - u : k - 1) * k;
          rb[u] = cur + (size_t)min(4 * tb + u, r - 1) * ldx;
        }
        warp_dots4<KT>(ra, rb, i0 >> 5, [&](int u, int v, float s) { Dm[(4 * ta + u) * 36 + 4 * tb + v] = s; });
      }
      __syncthreads();
      for (int x = tid; x < GB * 32; x += NT) {
        const int q = x >> 5, j = x & 31;
        if (j < 4 * nv) {
          float s0 = 0.f, s1 = 0.f;
#pragma unroll
          for (int p = 0; p < GB; p += 2) {
            s0 = fmaf(S[q * LS + p], Dm[p * 36 + j], s0);
            s1 = fmaf(S[q * LS + p + 1], Dm[(p + 1) * 36 + j], s1);
          }
          Cm[q * 36 + j] = s0 + s1;
        }
      }
      __syncthreads();
      const int nc = (k - i0 + 31) >> 5;
      for (int t = ty; t < nv * nc; t += NW) {
        const int tj = t / nc, i = i0 + 32 * (t % nc) + lane;
        if (i < k) {
          float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int q = 0; q < GB; ++q) {    // rows of Cm past the group are zero
            const float v = Vs[(size_t)max(h - q, 0) * k + i];
            const float4 c = *reinterpret_cast<const float4*>(Cm + q * 36 + 4 * tj);
            acc[0] = fmaf(v, c.x, acc[0]); acc[1] = fmaf(v, c.y, acc[1]);
            acc[2] = fmaf(v, c.z, acc[2]); acc[3] = fmaf(v, c.w, acc[3]);
          }
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (4 * tj + u < r) cur[(size_t)(4 * tj + u) * ldx + i] -= acc[u];
        }
      }
      __syncthreads();
    }
    for (int x = tid; x < k * r; x += NT) {
      const int i = x / r, j = x % r;
      V[(size_t)i * ldv + j] = cur[(size_t)j * ldx + i];
    }
    if (evals)
      for (int j = tid; j < r; j += NT) evals[j] = lam[j];
  }
}

// ------------------------------------------------------------ launcher
static int er_kt(int k) { return (k + 31) / 32; }

bool eig_reg_ok(int k, int r) {
  if (k < 1 || r < 1 || r > 32 || r > k || k > 32 * ER_KTMAX) return false;
  // dynamic shared memory plus the kernel's static arrays (the Cholesky's
  // 8,448 bytes, 12 KB reserved) within the 227 KB a CTA may use
  return er_layout(32 * er_kt(k), k, r).total * 4 + 12 * 1024 <= 227 * 1024;
}

template <int KT>
static cudaError_t launch_kt(const float* H, int64_t ldh, int k, int r, float* V, int ldv, float* evals,
                             float* scratch, cudaStream_t st) {
  // 16-byte aligned, for the reflectors' copy
  float* Vg = reinterpret_cast<float*>((reinterpret_cast<uintptr_t>(scratch) + 15) & ~uintptr_t(15));
  float* tau = Vg + (size_t)k * k;
  float* d = tau + k;
  float* e = d + k;
  k_eig_tridiag8<KT, ER_TRI_WARPS><<<1, ER_TRI_WARPS * 32, 0, st>>>(H, ldh, k, Vg, tau, d, e);
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) return err;
  const size_t smem = er_layout(32 * KT, k, r).total * 4;
  err = raise_smem_limit(k_eig_vectors<KT>);
  if (err != cudaSuccess) return err;
  k_eig_vectors<KT><<<1, 512, smem, st>>>(Vg, tau, d, e, k, r, V, ldv, evals);
  return cudaGetLastError();
}

// scratch: k * k + 3 k + 4 floats (device)
cudaError_t launch_eig_reg(const float* H, int64_t ldh, int k, int r, float* V, int ldv, float* evals,
                           float* scratch, cudaStream_t st) {
  if (!eig_reg_ok(k, r)) return cudaErrorInvalidValue;
  ProfScope prof("eig_top", st, 0, 0);
  note_launch("eig_top", 2);
  switch (er_kt(k)) {
    case 1: return launch_kt<1>(H, ldh, k, r, V, ldv, evals, scratch, st);
    case 2: return launch_kt<2>(H, ldh, k, r, V, ldv, evals, scratch, st);
    case 3: return launch_kt<3>(H, ldh, k, r, V, ldv, evals, scratch, st);
    case 4: return launch_kt<4>(H, ldh, k, r, V, ldv, evals, scratch, st);
    default: return launch_kt<5>(H, ldh, k, r, V, ldv, evals, scratch, st);
  }
}

}  // namespace ttr
