// GeLU and its derivative in the epilogues of the bf16 products, on packed pairs of fp32 values and without branches.  (The fp32 products
// take gelu_fwd and gelu_bwd of internal.h.)
#pragma once
#include <stdint.h>
#include "tc_ptx.cuh"

namespace ecmoe {

namespace {

// z within [-Z, Z]; NaN stays NaN (fminf and fmaxf answer the other operand), so that a derivative taken there is NaN too
__device__ __forceinline__ float clamp_nan(float z, float Z) {
  float r; asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(z), "f"(-Z));
  asm("min.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(r), "f"(Z));
  return r;
}

// Phi(z) = (1 + erf(z / sqrt 2)) / 2 for two values at once, without special-function instructions:
// erf(u) = u Q(t) with t = 2 u^2 / U^2 - 1 in [-1, 1], U = 3.4, u clamped to [-U, U] (erf(3.4) = 1 - 1.5e-6), and Q
// the degree-11 polynomial that interpolates erf(u) / u at the Chebyshev nodes in t (fitted for this file; the
// coefficients are those of the powers of t, all below 1 in size, so Horner's rule is stable in fp32).
// |error of Phi| < 1.6e-6 in fp32, three orders below bf16 resolution.
__device__ __forceinline__ unsigned long long norm_cdf2(unsigned long long z) {
  constexpr float U = 3.4f;
  const unsigned long long u = mul2(z, pk2(0.70710678118654752f, 0.70710678118654752f));
  const unsigned long long uc = pk2(fminf(fmaxf(lo2(u), -U), U), fminf(fmaxf(hi2(u), -U), U));
  const unsigned long long t = fma2(mul2(uc, uc), pk2(2.f / (U * U), 2.f / (U * U)), pk2(-1.f, -1.f));
  constexpr float c[12] = {4.156643398e-01f, -2.060884763e-01f, 1.495694051e-01f, -1.149434119e-01f, 8.608386700e-02f,
                           -6.136962761e-02f, 4.273188249e-02f, -2.607233935e-02f, 1.084438127e-02f, -5.875344802e-03f,
                           6.353731497e-03f, -2.781673617e-03f};
  unsigned long long acc = pk2(c[11], c[11]);
#pragma unroll
  for (int i = 10; i >= 0; --i) acc = fma2(acc, t, pk2(c[i], c[i]));
  return fma2(mul2(uc, acc), pk2(0.5f, 0.5f), pk2(0.5f, 0.5f));
}
// Of two values: 1 / (1 + 2^y), the logistic function of -y log 2; 0 where 2^y overflows
__device__ __forceinline__ unsigned long long logistic2(unsigned long long y) {
  float e[2], r[2];
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e[0]) : "f"(lo2(y))); asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e[1]) : "f"(hi2(y)));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r[0]) : "f"(1.f + e[0])); asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r[1]) : "f"(1.f + e[1]));
  return pk2(r[0], r[1]);
}
// The tanh form's (1 + tanh(u)) / 2 is the logistic function of 2 u, u = sqrt(2 / pi) (z + 0.044715 z^3): two special-function
// instructions and no branches where tanhf has both, |error| 1e-7 and small against the value in the tail too.
// 6080 x 1000 x 2072, ten experts: GEMM-1 55.4 -> 51.2 us, dZ 65.5 -> 49.1.
constexpr float kTanhA = 0.7978845608028654f, kTanhB = 0.044715f, kLog2E = 1.4426950408889634f;
__device__ __forceinline__ unsigned long long tanh_gate2(unsigned long long z, unsigned long long zz) {
  constexpr float c0 = -2.f * kTanhA * kLog2E, c1 = c0 * kTanhB;
  return logistic2(mul2(z, fma2(zz, pk2(c1, c1), pk2(c0, c0))));
}
// GeLU of a pair, in place.  VARIANT 0: z Phi(z); 1: the tanh form.
template <int VARIANT>
__device__ __forceinline__ void gelu_fwd2(float z0, float z1, float& h0, float& h1) {
  const unsigned long long z = pk2(z0, z1), h = mul2(z, VARIANT == 0 ? norm_cdf2(z) : tanh_gate2(z, mul2(z, z)));
  h0 = lo2(h); h1 = hi2(h);
}
// GeLU'(z) of a pair.  VARIANT 0: Phi(z) + z phi(z), phi the normal density.  Less 1/2 it is odd: z Q(t), t = 2 z^2 / Z^2 - 1, Z = 5.5 (z
// clamped to [-Z, Z]: GeLU'(5.5) = 1 + 5.7e-7), Q the degree-15 polynomial through the Chebyshev nodes in t, fitted like norm_cdf2's.
// |error| < 5e-7 in fp32, where norm_cdf2 and an exponential had 1.6e-6 and took half as many instructions again (dZ of
// 8192 x 768 x 3072, 32 experts: 127 -> 118 us).
template <int VARIANT>
__device__ __forceinline__ void gelu_bwd2(float z0, float z1, float& g0, float& g1) {
  unsigned long long g;
  if constexpr (VARIANT == 0) {
    constexpr float Z = 5.5f;
    const unsigned long long z = pk2(clamp_nan(z0, Z), clamp_nan(z1, Z));
    const unsigned long long t = fma2(mul2(z, z), pk2(2.f / (Z * Z), 2.f / (Z * Z)), pk2(-1.f, -1.f));
    constexpr float c[16] = {1.287591376e-01f, -6.573985250e-02f, 5.367434234e-02f, -5.373902109e-02f, 6.012413464e-02f, -6.868787701e-02f,
                             7.575927955e-02f, -7.385357749e-02f, 5.931453062e-02f, -5.048873522e-02f, 5.172561041e-02f, -3.163604518e-02f,
                             2.391405735e-03f, -3.607926043e-03f, 1.264834743e-02f, -5.734611948e-03f};
    unsigned long long acc = pk2(c[15], c[15]);
#pragma unroll
    for (int i = 14; i >= 0; --i) acc = fma2(acc, t, pk2(c[i], c[i]));
    g = fma2(z, acc, pk2(0.5f, 0.5f));
  } else {
    const unsigned long long z = pk2(z0, z1), zz = mul2(z, z), s = tanh_gate2(z, zz);
    constexpr float w0 = 2.f * kTanhA, w1 = 3.f * kTanhB * w0;          // of d(2 u) / dz
    g = fma2(mul2(mul2(z, s), fma2(s, pk2(-1.f, -1.f), pk2(1.f, 1.f))), fma2(zz, pk2(w1, w1), pk2(w0, w0)), s);
  }
  g0 = lo2(g); g1 = hi2(g);
}

}  // namespace

}  // namespace ecmoe
