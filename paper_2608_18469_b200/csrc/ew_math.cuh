// Elementwise math shared by the elementwise kernels, the GEMM epilogues and the persistent dual-list
// kernel, so that all of them produce the same bits.
#pragma once
#include <stdint.h>

namespace erase {

// Exact-erf GELU on bf16 data (the result is rounded to bf16 by the caller).  With t = min(|u|, 6) and
//   R(t) = Phi(-t) exp(t^2/2)      (smooth: falls from 0.5 to 0.066 on [0, 6]),
//   gelu(u)  = max(u, 0) - t exp(-u^2/2) R(t)
//   gelu'(u) = r for u < 0, 1 - r for u >= 0,   r = exp(-u^2/2) (R(t) - t/sqrt(2 pi)).
// R and R - t/sqrt(2 pi) are polynomials in x = t/3 - 1 on [-1, 1], fitted for the smallest largest error of
// exp(-t^2/2) R (a linear program over a Chebyshev basis); evaluated in fp32 on every bf16 argument the error of
// the value is 2.5e-7, of the derivative 2.3e-7 (2.6e-7 both on fp32 arguments), as large as fp32 rounding itself and
// three orders below bf16 resolution.  Beyond |u| = 6 only the factors t and R(t) stay where they are while the
// exponential of the true argument falls on: below -6 the value is off by 3e-12 at most and the derivative by 4e-10,
// and both go to zero (with the exponential clamped too they would stay at -6e-9 and -4e-8: a unit that is
// far off would still pass a gradient back).  An infinity gives its limits, a NaN stays a NaN.
// What bounds this code is instruction issue in a GEMM epilogue, whose few warps share the SM with the tensor
// core: one special-function instruction per element (ex2) instead of the two of a rational form in
// 1/(1 + p|u|), and the polynomial runs on packed pairs (fma.rn.f32x2: two fp32 FMAs per issue slot), about 11
// issue slots per element against 20.
constexpr int GELU_NV = 13, GELU_ND = 12;
#define ERASE_GELU_VALUE_COEF {-0.121514406f, 0.103172934f, -0.0825883924f, 0.0624255716f, -0.0424559082f, 0.0360049661f, -0.0258772451f, -0.00638427118f, -0.0134245794f, 0.0305226626f, 0.0148703471f, -0.00816017831f, -0.0114281104f}
#define ERASE_GELU_DERIV_COEF {-1.07531861f, -1.30003944f, 0.0829805067f, -0.0589785751f, 0.0494564107f, -0.0417208265f, -0.00814567257f, -0.0161115608f, 0.0528829511f, 0.0233364257f, -0.0163927669f, -0.0210231259f}

__device__ __forceinline__ float ex2_fast(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rcp_fast(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float min_nan(float a, float b) {   // NaN if either is
  float r;
  asm("min.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}

typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack_f2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack_f2(f32x2 v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ f32x2 fma_f2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f32x2 add_f2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 mul_f2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// P independent pairs side by side: a polynomial is a serial chain, and an epilogue has only two warps per
// scheduler to hide it with, so the pairs' chains are interleaved term by term.
// t = min(|u|, 6), x = t/3 - 1, e = exp(-u^2/2)
template <int P>
__device__ __forceinline__ void gelu_parts(const float* u, f32x2* t, f32x2* x, f32x2* e) {
  f32x2 a[P];
#pragma unroll
  for (int p = 0; p < P; p++) t[p] = pack_f2(min_nan(fabsf(u[2 * p]), 6.f), min_nan(fabsf(u[2 * p + 1]), 6.f));
#pragma unroll
  for (int p = 0; p < P; p++) a[p] = mul_f2(pack_f2(u[2 * p], u[2 * p + 1]), pack_f2(-0.72134752f, -0.72134752f));
#pragma unroll
  for (int p = 0; p < P; p++) a[p] = mul_f2(a[p], pack_f2(u[2 * p], u[2 * p + 1]));       // -u^2/2 in log2 units
#pragma unroll
  for (int p = 0; p < P; p++) x[p] = fma_f2(t[p], pack_f2(0.333333343f, 0.333333343f), pack_f2(-1.f, -1.f));
#pragma unroll
  for (int p = 0; p < P; p++) {
    float a0, a1;
    unpack_f2(a[p], a0, a1);
    e[p] = pack_f2(ex2_fast(a0), ex2_fast(a1));
  }
}
template <int P, int N>
__device__ __forceinline__ void poly(const float (&c)[N], const f32x2* x, f32x2* r) {
#pragma unroll
  for (int p = 0; p < P; p++) r[p] = fma_f2(pack_f2(c[N - 1], c[N - 1]), x[p], pack_f2(c[N - 2], c[N - 2]));
#pragma unroll
  for (int k = N - 3; k >= 0; k--)
#pragma unroll
    for (int p = 0; p < P; p++) r[p] = fma_f2(r[p], x[p], pack_f2(c[k], c[k]));
}
// v <- gelu(v) for N values, in place
template <int N>
__device__ __forceinline__ void gelu_bf16_n(float* v) {
  constexpr int P = N / 2;
  constexpr float c[GELU_NV] = ERASE_GELU_VALUE_COEF;   // coefficients of -R
  f32x2 t[P], x[P], e[P], r[P];
  gelu_parts<P>(v, t, x, e);
#pragma unroll
  for (int p = 0; p < P; p++) e[p] = mul_f2(t[p], e[p]);
  poly<P>(c, x, r);
#pragma unroll
  for (int p = 0; p < P; p++) {
    const f32x2 g = fma_f2(e[p], r[p], pack_f2(fmaxf(v[2 * p], 0.f), fmaxf(v[2 * p + 1], 0.f)));
    unpack_f2(g, v[2 * p], v[2 * p + 1]);
  }
}
// d <- d * gelu'(u) for N values, in place
template <int N>
__device__ __forceinline__ void dgelu_bf16_n(const float* u, float* d) {
  constexpr int P = N / 2;
  constexpr float c[GELU_ND] = ERASE_GELU_DERIV_COEF;
  f32x2 t[P], x[P], e[P], r[P];
  gelu_parts<P>(u, t, x, e);
  poly<P>(c, x, r);
#pragma unroll
  for (int p = 0; p < P; p++) {
    float r0, r1;
    unpack_f2(mul_f2(e[p], r[p]), r0, r1);
    d[2 * p] *= u[2 * p] < 0.f ? r0 : 1.f - r0;
    d[2 * p + 1] *= u[2 * p + 1] < 0.f ? r1 : 1.f - r1;
  }
}
// y <- gelu(u) and g <- gelu'(u) for N values.  Both follow from Phi(-t) = exp(-t^2/2) (b1 s + .. + b5 s^5),
// s = 1/(1 + p t): the form of Abramowitz and Stegun 7.1.26, with p and b fitted as above (largest error of max(1, t) Phi);
// t as above.  On every bf16 argument the value is off by 2.5e-7 at most, the derivative by 2.4e-7.  In an elementwise kernel
// the FMA pipe is what the polynomials above would fill (12 FMAs, where five and a second special function do here).
template <int N>
__device__ __forceinline__ void gelu_both_bf16_n(const float* u, float* y, float* g) {
  constexpr int P = N / 2;
  f32x2 t[P], e[P], q[P], s[P];
#pragma unroll
  for (int p = 0; p < P; p++) t[p] = pack_f2(min_nan(fabsf(u[2 * p]), 6.f), min_nan(fabsf(u[2 * p + 1]), 6.f));
#pragma unroll
  for (int p = 0; p < P; p++) {
    const f32x2 v = pack_f2(u[2 * p], u[2 * p + 1]);
    float a0, a1;
    unpack_f2(mul_f2(mul_f2(v, pack_f2(-0.72134752f, -0.72134752f)), v), a0, a1);
    e[p] = pack_f2(ex2_fast(a0), ex2_fast(a1));
  }
#pragma unroll
  for (int p = 0; p < P; p++) {
    float a0, a1;
    unpack_f2(fma_f2(t[p], pack_f2(0.3325f, 0.3325f), pack_f2(1.f, 1.f)), a0, a1);
    s[p] = pack_f2(rcp_fast(a0), rcp_fast(a1));
  }
  constexpr float b[5] = {0.123695001f, 0.199656487f, -0.0793629587f, 0.365162402f, -0.109150954f};
#pragma unroll
  for (int p = 0; p < P; p++) q[p] = fma_f2(s[p], pack_f2(b[4], b[4]), pack_f2(b[3], b[3]));
#pragma unroll
  for (int k = 2; k >= 0; k--)
#pragma unroll
    for (int p = 0; p < P; p++) q[p] = fma_f2(q[p], s[p], pack_f2(b[k], b[k]));
#pragma unroll
  for (int p = 0; p < P; p++) q[p] = mul_f2(mul_f2(q[p], s[p]), e[p]);           // Phi(-t)
#pragma unroll
  for (int p = 0; p < P; p++) {
    float q0, q1, t0, t1, d0, d1;
    unpack_f2(q[p], q0, q1);
    unpack_f2(t[p], t0, t1);
    y[2 * p] = fmaf(-t0, q0, fmaxf(u[2 * p], 0.f));
    y[2 * p + 1] = fmaf(-t1, q1, fmaxf(u[2 * p + 1], 0.f));
    unpack_f2(fma_f2(mul_f2(t[p], e[p]), pack_f2(-0.39894228f, -0.39894228f), q[p]), d0, d1);
    g[2 * p] = u[2 * p] < 0.f ? d0 : 1.f - d0;
    g[2 * p + 1] = u[2 * p + 1] < 0.f ? d1 : 1.f - d1;
  }
}

}  // namespace erase
