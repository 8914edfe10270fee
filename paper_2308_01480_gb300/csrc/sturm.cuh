// Eigenvalue counts of a symmetric tridiagonal matrix (step 2 of eig_reg.cu).
#pragma once

namespace ttr {
namespace {

// Row (d_i, e_{i-1}^2) of de.  Where x is an eigenvalue of a leading block and
// the next off-diagonal is zero, two minors in a row would be zero and every
// later one with them; so e^2 is kept at 2^-60 at least.  Zeros then stand
// alone (their sign bit does not matter: the minors beside them have opposite
// signs), and T moves by 2^-30 of its norm, below the 2^-24 that the bisection
// resolves.
constexpr float kSturmE2Min = 8.67361738e-19f;   // 2^-60
__device__ __forceinline__ float2 sturm_row(float d, float e) { return make_float2(d, fmaxf(e * e, kSturmE2Min)); }

// Number of eigenvalues of the scaled T below x: sign changes of the leading
// principal minors p_i = (d_i - x) p_{i-1} - e_{i-1}^2 p_{i-2} (Givens 1953),
// de[i] = (d_i, e_{i-1}^2), |T| < 2.  One multiply-add a row is on the chain
// (the ratios p_i / p_{i-1} would put a reciprocal and a comparison there);
// every four rows the pair is rescaled by a power of two.  Rows past the last
// are padded by (16, 0), which changes no sign, up to 1 + 4 groups rows.
// k = 150: 75 to 100 cycles a row as ratios, about 55 (two counts a warp).
struct SturmPair {
  float p0, p1;
  unsigned m;        // signs of the last p's, newest in bit 0
  int c;
  __device__ __forceinline__ void start(float2 t, float x) {
    p0 = 1.f;
    p1 = t.x - x;
    m = __float_as_uint(p1) >> 31;
    c = (int)m;
  }
  __device__ __forceinline__ void step(float d, float e2, float x) {
    const float pn = fmaf(d - x, p1, -(e2 * p0));
    m = __funnelshift_l(__float_as_uint(pn), m, 1);
    p0 = p1;
    p1 = pn;
  }
  // after every four steps
  __device__ __forceinline__ void settle() {
    c += __popc((m ^ (m >> 1)) & 15u);
    const float f0 = fmaxf(fabsf(p0), fabsf(p1));
    const float f = __uint_as_float(0x7f000000u - (__float_as_uint(f0) & 0x7f800000u));
    p0 *= f;
    p1 = (f0 == 0.f) ? copysignf(1.f, p1) : p1 * f;     // both underflowed: go on from the last sign
  }
};

// Rows 1 .. 4 groups are read as pairs: de + 1 is 16-byte aligned.
__device__ __forceinline__ int sturm(const float2* de, int groups, float x) {
  SturmPair s;
  s.start(de[0], x);
  const float4* q = reinterpret_cast<const float4*>(de + 1);
#pragma unroll 2
  for (int g = 0; g < groups; ++g) {
    const float4 a = q[2 * g], b = q[2 * g + 1];
    s.step(a.x, a.y, x);
    s.step(a.z, a.w, x);
    s.step(b.x, b.y, x);
    s.step(b.z, b.w, x);
    s.settle();
  }
  return s.c;
}

// Two counts (at x0 and x1) in one pass, so that the two chains overlap.
__device__ __forceinline__ void sturm2(const float2* de, int groups, float x0, float x1, int& c0, int& c1) {
  SturmPair s0, s1;
  s0.start(de[0], x0);
  s1.start(de[0], x1);
  const float4* q = reinterpret_cast<const float4*>(de + 1);
  for (int g = 0; g < groups; ++g) {
    const float4 a = q[2 * g], b = q[2 * g + 1];
    s0.step(a.x, a.y, x0); s1.step(a.x, a.y, x1);
    s0.step(a.z, a.w, x0); s1.step(a.z, a.w, x1);
    s0.step(b.x, b.y, x0); s1.step(b.x, b.y, x1);
    s0.step(b.z, b.w, x0); s1.step(b.z, b.w, x1);
    s0.settle();
    s1.settle();
  }
  c0 = s0.c;
  c1 = s1.c;
}

}  // namespace
}  // namespace ttr
