// Hand-written CUDA kernels (plain SIMT) of the ERASE step library: the general GEMM used for
// fp32 models and for shapes the tensor-core path does not take, and every non-GEMM operation
// of the step (LayerNorm, causal attention, losses, gathers, dot interaction, optimizer).
// Reductions are fixed-partition / fixed-order: no floating-point atomics anywhere.
#include "kernels.cuh"
#include "launch.cuh"
#include "ew_math.cuh"

#include <stdlib.h>

#include <algorithm>
#include <atomic>
#include <type_traits>

#include <cuda.h>
#include <cuda_bf16.h>
#include <math.h>

namespace erase {

typedef __nv_bfloat16 bf16_t;

template <typename T> __device__ __forceinline__ float ldf(const T* p);
template <> __device__ __forceinline__ float ldf<float>(const float* p) { return *p; }
template <> __device__ __forceinline__ float ldf<bf16_t>(const bf16_t* p) { return __bfloat162float(*p); }
template <typename T> __device__ __forceinline__ void stf(T* p, float v);
template <> __device__ __forceinline__ void stf<float>(float* p, float v) { *p = v; }
template <> __device__ __forceinline__ void stf<bf16_t>(bf16_t* p, float v) { *p = __float2bfloat16_rn(v); }
// four consecutive values (p 16-byte aligned for float, 8-byte for bf16)
__device__ __forceinline__ void store4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ void store4(bf16_t* p, float4 v) {
  __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
  uint2 q;
  q.x = *reinterpret_cast<uint32_t*>(&lo);
  q.y = *reinterpret_cast<uint32_t*>(&hi);
  *reinterpret_cast<uint2*>(p) = q;
}

__device__ __forceinline__ float act_apply(int act, float v) {
  if (act == ACT_RELU) return v > 0.f ? v : 0.f;
  if (act == ACT_GELU) return v * 0.5f * (1.f + erff(v * 0.70710678118654752f));
  return v;
}
// derivative of the activation; GELU takes the pre-activation, ReLU accepts either the
// pre-activation or the output (same sign test; 0 at exactly 0).
__device__ __forceinline__ float act_deriv(int act, float u) {
  if (act == ACT_RELU) return u > 0.f ? 1.f : 0.f;
  if (act == ACT_GELU) {
    float cdf = 0.5f * (1.f + erff(u * 0.70710678118654752f));
    float pdf = 0.39894228040143268f * expf(-0.5f * u * u);
    return cdf + u * pdf;
  }
  return 1.f;
}

// GELU / GELU' of a 16-byte vector in place; bf16 data takes the cheaper form of ew_math.cuh
__device__ __forceinline__ void gelu_vec(float (&v)[4]) {
#pragma unroll
  for (int j = 0; j < 4; j++) v[j] = act_apply(ACT_GELU, v[j]);
}
__device__ __forceinline__ void gelu_vec(float (&v)[8]) { gelu_bf16_n<8>(v); }
__device__ __forceinline__ void dgelu_vec(const float (&u)[4], float (&d)[4]) {
#pragma unroll
  for (int j = 0; j < 4; j++) d[j] *= act_deriv(ACT_GELU, u[j]);
}
__device__ __forceinline__ void dgelu_vec(const float (&u)[8], float (&d)[8]) { dgelu_bf16_n<8>(u, d); }

// y <- gelu(u), g <- gelu'(u) for eight values; data of type T
template <typename T>
__device__ __forceinline__ void act_both(const float (&u)[8], float (&y)[8], float (&g)[8]) {
  if (sizeof(T) == 2) {
    gelu_both_bf16_n<8>(u, y, g);
  } else {
#pragma unroll
    for (int j = 0; j < 8; j++) { y[j] = act_apply(ACT_GELU, u[j]); g[j] = act_deriv(ACT_GELU, u[j]); }
  }
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

static inline unsigned cdiv(long long a, long long b) { return (unsigned)((a + b - 1) / b); }

// ------------------------------------------------------------------------------------------
// general GEMM on the FMA pipe: TS x TS output tiles (TS = 32: one to four groups of 128 threads with 2 x 4 outputs, TS = 64:
// 256 threads with 4 x 4), K in chunks of 32 through two shared-memory buffers (one per group where there are several), the next
// chunk's loads in flight while a chunk is multiplied.  It serves fp32 models, GEMVs and bf16 shapes that TMA cannot describe.  On the sizes of the fp32
// models (256 rows, widths 64..256) the latency of a CTA's chain of chunks bounds it, hence small tiles over
// more SMs, long chunks and the prefetch; the order of the sum over k follows from the shape alone (with groups of
// threads along it, the sums of their shares are added in turn).
// (64 x 64 x 16 tiles without the prefetch took 23, 20 and 15 us for the forward, weight-gradient and dgrad GEMMs of
// a 256-row block of widths 64 and 256, now 11, 9 and 10.5 between events; with the weight gradients' partials added
// in the block's batched reduction the whole step went from 120 to 56 us.)
// Both operands are staged [k][m] so that a thread reads its rows and columns as vectors; column m of row k sits
// at m ^ (4 * (k/4 mod 8)), which makes the transposing stores of a K-major operand free of bank conflicts.
// ------------------------------------------------------------------------------------------
// four consecutive elements starting at p, of which `valid` exist (vec: p is aligned for one vector load)
__device__ __forceinline__ float4 ld4_guard(const float* p, int valid, bool vec) {
  if (vec && valid >= 4) return *reinterpret_cast<const float4*>(p);
  return make_float4(valid > 0 ? p[0] : 0.f, valid > 1 ? p[1] : 0.f, valid > 2 ? p[2] : 0.f, valid > 3 ? p[3] : 0.f);
}
__device__ __forceinline__ float4 ld4_guard(const bf16_t* p, int valid, bool vec) {
  if (vec && valid >= 4) {
    const uint2 q = *reinterpret_cast<const uint2*>(p);
    return make_float4(__uint_as_float(q.x << 16), __uint_as_float(q.x & 0xffff0000u), __uint_as_float(q.y << 16), __uint_as_float(q.y & 0xffff0000u));
  }
  return make_float4(valid > 0 ? ldf(p) : 0.f, valid > 1 ? ldf(p + 1) : 0.f, valid > 2 ? ldf(p + 2) : 0.f, valid > 3 ? ldf(p + 3) : 0.f);
}

// One operand's share of a chunk: two groups of four elements per thread, contiguous along K (KM) or along M.
template <typename T, bool KM, int TS, int NT>
struct SimtOperand {
  static constexpr int LD = TS + 4;
  float4 q[2];
  __device__ __forceinline__ void load(const T* P, long long s_m, long long s_k, int m0, int M, int k0, int kend, bool vec) {
#pragma unroll
    for (int g = 0; g < 2; g++) {
      const int e = threadIdx.x % NT + g * NT;
      const int m = KM ? m0 + (e >> 3) : m0 + (e % (TS / 4)) * 4, k = KM ? k0 + (e & 7) * 4 : k0 + e / (TS / 4);
      const int valid = KM ? (m < M ? kend - k : 0) : (k < kend ? M - m : 0);
      q[g] = ld4_guard(valid > 0 ? P + (long long)m * s_m + (long long)k * s_k : P, valid, vec);
    }
  }
  __device__ __forceinline__ void store(float* sm) const {
#pragma unroll
    for (int g = 0; g < 2; g++) {
      const int e = threadIdx.x % NT + g * NT;
      if (KM) {
        const int m = e >> 3, k = (e & 7) * 4, at = m ^ ((e & 7) << 2);
        sm[k * LD + at] = q[g].x;
        sm[(k + 1) * LD + at] = q[g].y;
        sm[(k + 2) * LD + at] = q[g].z;
        sm[(k + 3) * LD + at] = q[g].w;
      } else {
        const int m = (e % (TS / 4)) * 4, k = e / (TS / 4);
        *reinterpret_cast<float4*>(sm + k * LD + (m ^ (((k >> 2) & 7) << 2))) = q[g];
      }
    }
  }
};

// The epilogue of one output; alpha, bias, pre-activation, activation, multiplier, residual, derivative, product -- in this order
template <typename T>
__device__ __forceinline__ void simt_finish(const GemmArgs& g, int split, int m, int n, float v) {
  if (m >= g.M || n >= g.N) return;
  const Epilogue& e = g.epi;
  if (g.splits > 1) {
    g.ws[(long long)split * g.M * g.N + (long long)m * g.N + n] = v;
    return;
  }
  v *= e.alpha;
  if (e.bias) v += e.bias[n];
  const long long ia = (long long)m * e.ld_aux + n;
  if (e.pre_out) stf((T*)e.pre_out + ia, v);
  v = act_apply(e.act, v);
  if (e.mul) v *= ldf((const T*)e.mul + ia);
  if (e.res) v += ldf((const T*)e.res + ia);
  if (e.dact != ACT_NONE) v *= act_deriv(e.dact, ldf((const T*)e.dact_src + ia));
  if (e.post_mul) {
    const float w = v * ldf((const T*)e.post_mul + ia);
    if (e.post_out) stf((T*)e.post_out + ia, w);
    else v = w;
  }
  const long long ic = (long long)m * g.ldc + n;
  if (g.c_f32) ((float*)g.C)[ic] = v; else stf((T*)g.C + ic, v);
}

// KG > 1 (32 x 32 tiles): KG groups of 128 threads take contiguous shares of the CTA's contraction, whose chunks are then
// in flight side by side, and their sums are added in the order of the groups.  Where the grid leaves SMs idle anyway, the
// chain of chunks is what a GEMM takes: 256 x 64 x 256 between events 12.7 us with one group, 11.0 with four (two-block MLP step
// 47 -> 40 us).
template <typename T, bool AK, bool BK, int TS, int KG>
__global__ void __launch_bounds__(TS == 32 ? 128 * KG : 256) gemm_simt_kernel(GemmArgs g, bool avec, bool bvec) {
  pdl_wait();
  static_assert(KG == 1 || TS == 32, "groups share 32 x 32 tiles");
  constexpr int NT = TS == 32 ? 128 : 256, KC = 32, LD = TS + 4, RM = TS == 32 ? 2 : 4, BUFS = KG == 1 ? 2 : KG;
  __shared__ __align__(16) float As[BUFS][KC * LD];
  __shared__ __align__(16) float Bs[BUFS][KC * LD];
  const int tid = threadIdx.x % NT, kg = threadIdx.x / NT, tx = tid % (TS / 4), ty = tid / (TS / 4);
  const int m0 = blockIdx.y * TS, n0 = blockIdx.x * TS, split = blockIdx.z;
  const int kchunk = (((g.K + g.splits - 1) / g.splits) + 15) / 16 * 16;
  const int sbeg = split * kchunk, send = min(g.K, sbeg + kchunk);
  const int share = KG == 1 ? send - sbeg : ((send - sbeg + KG - 1) / KG + 3) / 4 * 4;      // (all groups go through the same number of chunks)
  const int kbeg = sbeg + kg * share, kend = min(send, kbeg + share);
  const T* A = (const T*)g.A;
  const T* B = (const T*)g.B;
  float acc[RM][4];
#pragma unroll
  for (int i = 0; i < RM; i++)
#pragma unroll
    for (int j = 0; j < 4; j++) acc[i][j] = 0.f;

  SimtOperand<T, AK, TS, NT> a;
  SimtOperand<T, BK, TS, NT> b;
  if (share > 0) {
    a.load(A, g.sa_m, g.sa_k, m0, g.M, kbeg, kend, avec);
    b.load(B, g.sb_n, g.sb_k, n0, g.N, kbeg, kend, bvec);
  }
  int buf = KG == 1 ? 0 : kg;
  for (int k = 0; k < share; k += KC) {
    a.store(As[buf]);
    b.store(Bs[buf]);
    __syncthreads();       // (KG == 1, two buffers: the next chunk's stores meet no reader of this one)
    if (k + KC < share) {
      a.load(A, g.sa_m, g.sa_k, m0, g.M, kbeg + k + KC, kend, avec);
      b.load(B, g.sb_n, g.sb_k, n0, g.N, kbeg + k + KC, kend, bvec);
    }
#pragma unroll
    for (int kk = 0; kk < KC; kk++) {
      const int swz = ((kk >> 2) & 7) << 2;
      float av[RM];
#pragma unroll
      for (int i = 0; i < RM; i += 2) {
        const float2 t = *reinterpret_cast<const float2*>(&As[buf][kk * LD + ((ty * RM + i) ^ swz)]);
        av[i] = t.x; av[i + 1] = t.y;
      }
      const float4 b4 = *reinterpret_cast<const float4*>(&Bs[buf][kk * LD + ((tx * 4) ^ swz)]);
      const float bv[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
      for (int i = 0; i < RM; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
    }
    if (KG == 1) buf ^= 1;
    else __syncthreads();
  }

  if (KG > 1) {
    float* part = &As[0][0];       // [group][row][column]: KG * 1024 floats
#pragma unroll
    for (int i = 0; i < RM; i++)
      *reinterpret_cast<float4*>(part + kg * 1024 + (ty * RM + i) * 32 + tx * 4) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
    __syncthreads();
#pragma unroll
    for (int o = 0; o < 8 / KG; o++) {
      const int i = threadIdx.x + o * 128 * KG;
      float v = part[i];
#pragma unroll
      for (int k = 1; k < KG; k++) v += part[k * 1024 + i];
      simt_finish<T>(g, split, m0 + (i >> 5), n0 + (i & 31), v);
    }
    return;
  }
#pragma unroll
  for (int i = 0; i < RM; i++)
#pragma unroll
    for (int j = 0; j < 4; j++) simt_finish<T>(g, split, m0 + ty * RM + i, n0 + tx * 4 + j, acc[i][j]);
}

template <typename T, int TS, int KG>
static void gemm_simt_ts(const GemmArgs& g, cudaStream_t s) {
  dim3 grid(cdiv(g.N, TS), cdiv(g.M, TS), g.splits);
  constexpr int NT = TS == 32 ? 128 * KG : 256;
  auto al = [](const void* p, long long ld) { return ld % 4 == 0 && (reinterpret_cast<uintptr_t>(p) & (4 * sizeof(T) - 1)) == 0; };
  const bool ak = g.sa_k == 1, bk = g.sb_k == 1, av = al(g.A, ak ? g.sa_m : g.sa_k), bv = al(g.B, bk ? g.sb_n : g.sb_k);
  if (ak && bk) pdl_launch(gemm_simt_kernel<T, true, true, TS, KG>, grid, NT, 0, s, g, av, bv);
  else if (ak && !bk) pdl_launch(gemm_simt_kernel<T, true, false, TS, KG>, grid, NT, 0, s, g, av, bv);
  else if (!ak && bk) pdl_launch(gemm_simt_kernel<T, false, true, TS, KG>, grid, NT, 0, s, g, av, bv);
  else pdl_launch(gemm_simt_kernel<T, false, false, TS, KG>, grid, NT, 0, s, g, av, bv);
}

template <typename T>
static cudaError_t gemm_simt_t(const GemmArgs& g, cudaStream_t s) {
  // 64 x 64 tiles (half the shared-memory reads per FMA) once they fill the 148 SMs, 32 x 32 below
  if ((long long)cdiv(g.N, 64) * cdiv(g.M, 64) * g.splits >= 148) {
    gemm_simt_ts<T, 64, 1>(g, s);
    return cudaGetLastError();
  }
  // groups of threads along the contraction while their CTAs fit side by side (four per SM), each with a chunk or more
  const long long ctas = (long long)cdiv(g.N, 32) * cdiv(g.M, 32) * g.splits;
  const int k = (g.K + g.splits - 1) / g.splits;
  if (ctas <= 296 && k >= 128) gemm_simt_ts<T, 32, 4>(g, s);
  else if (ctas <= 592 && k >= 64) gemm_simt_ts<T, 32, 2>(g, s);
  else gemm_simt_ts<T, 32, 1>(g, s);
  return cudaGetLastError();
}

cudaError_t gemm_simt(const GemmArgs& g, bool bf16, cudaStream_t s) {
  if (g.M <= 0 || g.N <= 0) return cudaSuccess;
  return bf16 ? gemm_simt_t<bf16_t>(g, s) : gemm_simt_t<float>(g, s);
}

// one thread writes the GPU's nanosecond clock: a phase boundary that can be captured into a graph
__global__ void stamp_kernel(unsigned long long* slot) {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  *slot = t;
}
cudaError_t stamp_time(unsigned long long* slot, cudaStream_t s) {
  stamp_kernel<<<1, 1, 0, s>>>(slot);
  return cudaGetLastError();
}

template <bool BF16_OUT>
__global__ void splitk_reduce_kernel(const float* ws, int splits, long long mn, int N,
                                     void* __restrict__ out, long long ldo) {
  pdl_wait();
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= mn) return;
  float a = 0.f;
  for (int s = 0; s < splits; s++) a += ws[(long long)s * mn + i];
  const long long o = (i / N) * ldo + (i % N);
  if (BF16_OUT) ((bf16_t*)out)[o] = __float2bfloat16_rn(a);
  else ((float*)out)[o] = a;
}

// four adjacent columns per thread (N, ldo multiples of 4); the partials of up to four splits are in flight at once
template <bool BF16_OUT>
__device__ __forceinline__ void splitk_reduce_v4_body(const float4* ws, int splits, long long mn4, int N4,
                                                      void* __restrict__ out, long long ldo, long long i) {
  if (i >= mn4) return;
  float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int s0 = 0; s0 < splits; s0 += 4) {
    float4 v[4];
#pragma unroll
    for (int u = 0; u < 4; u++) v[u] = s0 + u < splits ? __ldcs(ws + (long long)(s0 + u) * mn4 + i) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int u = 0; u < 4; u++)
      if (s0 + u < splits) { a.x += v[u].x; a.y += v[u].y; a.z += v[u].z; a.w += v[u].w; }
  }
  const long long o = (i / N4) * ldo + (i % N4) * 4;
  if (BF16_OUT) {
    __nv_bfloat162 lo = __floats2bfloat162_rn(a.x, a.y), hi = __floats2bfloat162_rn(a.z, a.w);
    uint2 q;
    q.x = *reinterpret_cast<uint32_t*>(&lo);
    q.y = *reinterpret_cast<uint32_t*>(&hi);
    *reinterpret_cast<uint2*>((bf16_t*)out + o) = q;
  } else {
    *reinterpret_cast<float4*>((float*)out + o) = a;
  }
}
template <bool BF16_OUT>
__global__ void splitk_reduce_v4_kernel(const float4* ws, int splits, long long mn4, int N4,
                                        void* __restrict__ out, long long ldo) {
  pdl_wait();
  splitk_reduce_v4_body<BF16_OUT>(ws, splits, mn4, N4, out, ldo, (long long)blockIdx.x * blockDim.x + threadIdx.x);
}

cudaError_t splitk_reduce(const float* ws, int splits, long long mn, int N, void* out, long long ldo,
                          cudaStream_t s, bool out_bf16) {
  if (mn <= 0) return cudaSuccess;
  const bool vec = N % 4 == 0 && ldo % 4 == 0 && (reinterpret_cast<uintptr_t>(ws) & 15) == 0 &&
                   (reinterpret_cast<uintptr_t>(out) & 15) == 0;
  if (vec) {
    const long long mn4 = mn / 4;
    if (out_bf16) pdl_launch(splitk_reduce_v4_kernel<true>, cdiv(mn4, 256), 256, 0, s, (const float4*)ws, splits, mn4, N / 4, out, ldo);
    else pdl_launch(splitk_reduce_v4_kernel<false>, cdiv(mn4, 256), 256, 0, s, (const float4*)ws, splits, mn4, N / 4, out, ldo);
  } else {
    if (out_bf16) pdl_launch(splitk_reduce_kernel<true>, cdiv(mn, 256), 256, 0, s, ws, splits, mn, N, out, ldo);
    else pdl_launch(splitk_reduce_kernel<false>, cdiv(mn, 256), 256, 0, s, ws, splits, mn, N, out, ldo);
  }
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------
// column sums (bias gradients, head weight gradient of the BCE head)
// A CTA sums a strip of 64 columns over one chunk of the rows (a thread owns two adjacent
// columns: one 4-byte load per bf16 pair, 128 bytes per warp and row); the chunk partials go to
// ws and the last CTA of a strip to finish (atomic ticket) adds them in chunk order, so the
// result does not depend on which CTA that is.  The ticket counter is left at zero again.
// ------------------------------------------------------------------------------------------
int colsum_chunks(int rows, int cols) {
  int strips = (cols + 255) / 256;   // as wide as bf16 uses them: four CTAs per SM (two: 32768 x 4096 73 us, now 60)
  int want = (592 + strips - 1) / strips;
  int maxc = rows / 64;
  if (maxc < 1) maxc = 1;
  if (want > maxc) want = maxc;
  if (want < 1) want = 1;
  return want;
}

template <typename T> __device__ __forceinline__ float2 ld2(const T* p, bool vec);
template <> __device__ __forceinline__ float2 ld2<float>(const float* p, bool vec) {
  if (vec) return *reinterpret_cast<const float2*>(p);
  return make_float2(p[0], p[1]);
}
template <> __device__ __forceinline__ float2 ld2<bf16_t>(const bf16_t* p, bool vec) {
  if (vec) return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(p));
  return make_float2(__bfloat162float(p[0]), __bfloat162float(p[1]));
}

// sum_{k < chunks} p[k*stride] added in the order k = 0, 1, ..; eight loads are issued before the
// first add so that the final pass costs one memory latency per eight partials, not per partial.
__device__ __forceinline__ float ordered_sum(const float* p, long long stride, int chunks) {
  float t = 0.f;
  for (int k0 = 0; k0 < chunks; k0 += 8) {
    float v[8];
#pragma unroll
    for (int u = 0; u < 8; u++) v[u] = k0 + u < chunks ? __ldcg(p + (long long)(k0 + u) * stride) : 0.f;
#pragma unroll
    for (int u = 0; u < 8; u++) if (k0 + u < chunks) t += v[u];
  }
  return t;
}

// Shared tail of the two-stage reductions: returns true in the CTA that arrives last on `ticket`.
__device__ __forceinline__ bool last_cta(int* ticket, int expected) {
  __shared__ int s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = atomicAdd(ticket, 1);
    s_last = (t == expected - 1);
    if (s_last) *ticket = 0;
  }
  __syncthreads();
  if (s_last) __threadfence();
  return s_last != 0;
}

template <typename T> struct VecOf;
template <> struct VecOf<float> { static constexpr int N = 4; };
template <> struct VecOf<bf16_t> { static constexpr int N = 8; };

// 16 bytes = VecOf<T>::N consecutive elements -> floats
template <typename T> __device__ __forceinline__ void ld_vec(const T* p, float* out);
template <> __device__ __forceinline__ void ld_vec<float>(const float* p, float* out) {
  const float4 q = *reinterpret_cast<const float4*>(p);
  out[0] = q.x; out[1] = q.y; out[2] = q.z; out[3] = q.w;
}
template <> __device__ __forceinline__ void ld_vec<bf16_t>(const bf16_t* p, float* out) {
  const uint4 q = *reinterpret_cast<const uint4*>(p);
  const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
  for (int j = 0; j < 4; j++) {
    out[2 * j] = __uint_as_float(w[j] << 16);
    out[2 * j + 1] = __uint_as_float(w[j] & 0xffff0000u);
  }
}

__device__ __forceinline__ void st_vec(float* p, const float (&v)[4]) { *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]); }
__device__ __forceinline__ void st_vec(bf16_t* p, const float (&v)[8]) {
  uint32_t w[4];
#pragma unroll
  for (int j = 0; j < 4; j++) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
    w[j] = *reinterpret_cast<const uint32_t*>(&h);
  }
  *reinterpret_cast<uint4*>(p) = make_uint4(w[0], w[1], w[2], w[3]);
}
// the same for a row's last, partial vector (or an unaligned matrix): n valid elements, zeros behind
template <typename T, bool ALIGNED>
__device__ __forceinline__ void ld_vec_n(const T* p, int n, float (&v)[VecOf<T>::N]) {
  if (ALIGNED) {
    ld_vec<T>(p, v);
  } else {
#pragma unroll
    for (int j = 0; j < VecOf<T>::N; j++) v[j] = j < n ? ldf(p + j) : 0.f;
  }
}
// four elements as loaded, not yet converted (what a loop keeps in flight)
template <typename T> struct Raw4 { float4 q = {0.f, 0.f, 0.f, 0.f}; };
template <> struct Raw4<bf16_t> { uint2 q = {0u, 0u}; };
template <typename T, bool ALIGNED>
__device__ __forceinline__ void ld_raw4(const T* p, int n, Raw4<T>& r) {
  if (ALIGNED) {
    r = *reinterpret_cast<const Raw4<T>*>(p);
  } else {
    T* e = reinterpret_cast<T*>(&r);
#pragma unroll
    for (int j = 0; j < 4; j++)
      if (j < n) e[j] = p[j];
  }
}
__device__ __forceinline__ void unpack_raw4(const Raw4<float>& r, float* v) { v[0] = r.q.x; v[1] = r.q.y; v[2] = r.q.z; v[3] = r.q.w; }
__device__ __forceinline__ void unpack_raw4(const Raw4<bf16_t>& r, float* v) {
  v[0] = __uint_as_float(r.q.x << 16); v[1] = __uint_as_float(r.q.x & 0xffff0000u);
  v[2] = __uint_as_float(r.q.y << 16); v[3] = __uint_as_float(r.q.y & 0xffff0000u);
}
template <typename T, bool ALIGNED>
__device__ __forceinline__ void st_vec_n(T* p, int n, const float (&v)[VecOf<T>::N]) {
  if (ALIGNED) {
    st_vec(p, v);
  } else {
#pragma unroll
    for (int j = 0; j < VecOf<T>::N; j++)
      if (j < n) stf(p + j, v[j]);
  }
}

// A CTA sums a strip of 32*VEC columns over one chunk of rows: a thread owns VEC adjacent
// columns (one 16-byte load per row) and every 8th row, four rows in flight.
// bx = column strip, by = row chunk of this CTA (the grid of the plain kernel, or what the batched
// kernel derived from its job table).
template <typename T>
__device__ __forceinline__ void colsum_body(const T* X, long long ldx, int rows,
                                            int cols, const float* scale,
                                            float* __restrict__ ws, float* __restrict__ out, int chunks,
                                            int dact, const float* colscale, int* tickets, int bx, int by,
                                            float* smem) {   // 8 * 32*VEC floats
  constexpr int VEC = VecOf<T>::N;
  constexpr int SW = 32 * VEC;  // strip width
  float (*sm)[SW] = reinterpret_cast<float (*)[SW]>(smem);
  const int cx = threadIdx.x & 31, ry = threadIdx.x >> 5;
  const int c = bx * SW + cx * VEC;
  const int per = (rows + chunks - 1) / chunks;
  const int rb = by * per, re = min(rows, rb + per);
  const bool vec = X && (c + VEC <= cols) && (ldx % VEC == 0) && ((reinterpret_cast<uintptr_t>(X) & 15) == 0);
  float a[VEC];
#pragma unroll
  for (int j = 0; j < VEC; j++) a[j] = 0.f;
  if (c < cols) {
    if (vec) {
      int r = rb + ry;
      for (; r + 24 < re; r += 32) {
        float v[4][VEC];
#pragma unroll
        for (int u = 0; u < 4; u++) ld_vec<T>(X + (long long)(r + 8 * u) * ldx + c, v[u]);
#pragma unroll
        for (int u = 0; u < 4; u++) {
          const float sc = scale ? scale[r + 8 * u] : 1.f;
#pragma unroll
          for (int j = 0; j < VEC; j++) {
            float t = v[u][j];
            if (dact != ACT_NONE) t = act_deriv(dact, t);
            a[j] = fmaf(t, sc, a[j]);
          }
        }
      }
      for (; r < re; r += 8) {
        float v[VEC];
        ld_vec<T>(X + (long long)r * ldx + c, v);
        const float sc = scale ? scale[r] : 1.f;
#pragma unroll
        for (int j = 0; j < VEC; j++) {
          float t = v[j];
          if (dact != ACT_NONE) t = act_deriv(dact, t);
          a[j] = fmaf(t, sc, a[j]);
        }
      }
    } else {
      for (int r = rb + ry; r < re; r += 8) {
        const float sc = scale ? scale[r] : 1.f;
#pragma unroll
        for (int j = 0; j < VEC; j++) {
          if (c + j < cols) {
            float t = X ? ldf(X + (long long)r * ldx + c + j) : 1.f;
            if (dact != ACT_NONE) t = act_deriv(dact, t);
            a[j] = fmaf(t, sc, a[j]);
          }
        }
      }
    }
  }
#pragma unroll
  for (int j = 0; j < VEC; j++) sm[ry][cx * VEC + j] = a[j];
  __syncthreads();
  float* dst = chunks == 1 ? out : ws + (long long)by * cols;
  for (int i = threadIdx.x; i < SW; i += 256) {
    const int cc = bx * SW + i;
    if (cc < cols) {
      float t = 0.f;
#pragma unroll
      for (int k = 0; k < 8; k++) t += sm[k][i];
      if (chunks == 1 && colscale) t *= colscale[cc];
      dst[cc] = t;
    }
  }
  if (chunks == 1) return;
  if (!last_cta(tickets + bx, chunks)) return;
  for (int i = threadIdx.x; i < SW; i += 256) {
    const int cc = bx * SW + i;
    if (cc < cols) {
      float t = ordered_sum(ws + cc, cols, chunks);
      if (colscale) t *= colscale[cc];
      out[cc] = t;
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(256) colsum_kernel(const T* X, long long ldx, int rows,
                                                     int cols, const float* scale,
                                                     float* __restrict__ ws, float* __restrict__ out, int chunks,
                                                     int dact, const float* colscale, int* tickets) {
  pdl_wait();
  __shared__ float smem[8 * 32 * VecOf<T>::N];
  colsum_body<T>(X, ldx, rows, cols, scale, ws, out, chunks, dact, colscale, tickets, blockIdx.x, blockIdx.y, smem);
}

cudaError_t colsum(const void* X, bool x_bf16, long long ldx, int rows, int cols, const float* scale,
                   float* ws, int chunks, int* tickets, float* out, cudaStream_t s, int dact, const float* colscale) {
  if (x_bf16) {
    dim3 grid(cdiv(cols, 256), chunks);
    pdl_launch(colsum_kernel<bf16_t>, grid, 256, 0, s, (const bf16_t*)X, ldx, rows, cols, scale, ws, out, chunks, dact, colscale, tickets);
  } else {
    dim3 grid(cdiv(cols, 128), chunks);
    pdl_launch(colsum_kernel<float>, grid, 256, 0, s, (const float*)X, ldx, rows, cols, scale, ws, out, chunks, dact, colscale, tickets);
  }
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------
// LayerNorm
// ------------------------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(256) layernorm_fwd_kernel(const T* x, const float* gain,
                                                            const float* shift, T* __restrict__ y, T* __restrict__ xhat,
                                                            float* __restrict__ mean, float* __restrict__ rstd,
                                                            int rows, int d) {
  pdl_wait();
  int row = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (row >= rows) return;
  const T* xr = x + (long long)row * d;
  float s = 0.f;
  for (int c = lane; c < d; c += 32) s += ldf(xr + c);
  float mu = warp_sum(s) / d;
  float q = 0.f;
  for (int c = lane; c < d; c += 32) { float t = ldf(xr + c) - mu; q += t * t; }
  float r = rsqrtf(warp_sum(q) / d + 1e-5f);
  for (int c = lane; c < d; c += 32) {
    const float n = (ldf(xr + c) - mu) * r;
    stf(y + (long long)row * d + c, n * gain[c] + shift[c]);
    if (xhat) stf(xhat + (long long)row * d + c, n);
  }
  if (mean && lane == 0) { mean[row] = mu; rstd[row] = r; }
}

// bf16 rows of d <= 256*VPL columns, d % 8 == 0: a lane keeps up to VPL 16-byte pieces of its row in registers, so the
// row is read once (the generic kernel above walks over it three times, two bytes per lane and load: 1407 x 320 between
// events 9.6 us, here 7.1; its dx 12.1, here 8.6).
template <int VPL>
__global__ void __launch_bounds__(256) layernorm_fwd_vec_kernel(const bf16_t* x, const float* gain,
                                                                const float* shift, bf16_t* __restrict__ y, bf16_t* __restrict__ xhat,
                                                                float* __restrict__ mean, float* __restrict__ rstd,
                                                                int rows, int d) {
  pdl_wait();
  const int row = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (row >= rows) return;
  const bf16_t* xr = x + (long long)row * d;
  float v[VPL][8];
  float s = 0.f;
#pragma unroll
  for (int k = 0; k < VPL; k++) {
    if ((k * 32 + lane) * 8 >= d) continue;
    ld_vec<bf16_t>(xr + (k * 32 + lane) * 8, v[k]);
#pragma unroll
    for (int j = 0; j < 8; j++) s += v[k][j];
  }
  const float mu = warp_sum(s) / d;
  float q = 0.f;
#pragma unroll
  for (int k = 0; k < VPL; k++) {
    if ((k * 32 + lane) * 8 >= d) continue;
#pragma unroll
    for (int j = 0; j < 8; j++) { const float t = v[k][j] - mu; q = fmaf(t, t, q); }
  }
  const float r = rsqrtf(warp_sum(q) / d + 1e-5f);
#pragma unroll
  for (int k = 0; k < VPL; k++) {
    const int c = (k * 32 + lane) * 8;
    if (c >= d) continue;
    const float4 g0 = *reinterpret_cast<const float4*>(gain + c), g1 = *reinterpret_cast<const float4*>(gain + c + 4);
    const float4 b0 = *reinterpret_cast<const float4*>(shift + c), b1 = *reinterpret_cast<const float4*>(shift + c + 4);
    const float gg[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
    const float bb[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
    float n[8], o[8];
#pragma unroll
    for (int j = 0; j < 8; j++) { n[j] = (v[k][j] - mu) * r; o[j] = n[j] * gg[j] + bb[j]; }
    st_vec(y + (long long)row * d + c, o);
    if (xhat) st_vec(xhat + (long long)row * d + c, n);
  }
  if (mean && lane == 0) { mean[row] = mu; rstd[row] = r; }
}

cudaError_t layernorm_fwd(const void* x, const float* gain, const float* shift, void* y, void* xhat, float* mean,
                          float* rstd, int rows, int d, bool bf16, cudaStream_t s) {
  const bool al = ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(y) | reinterpret_cast<uintptr_t>(xhat) |
                    reinterpret_cast<uintptr_t>(gain) | reinterpret_cast<uintptr_t>(shift)) & 15) == 0;
  const unsigned grid = cdiv(rows, 8);
  if (bf16) {
    auto go = [&](auto kernel) {
      pdl_launch(kernel, grid, 256, 0, s, (const bf16_t*)x, gain, shift, (bf16_t*)y, (bf16_t*)xhat, mean, rstd, rows, d);
    };
    if (!al || d % 8 != 0 || d > 1024) go(layernorm_fwd_kernel<bf16_t>);
    else if (d <= 256) go(layernorm_fwd_vec_kernel<1>);
    else if (d <= 512) go(layernorm_fwd_vec_kernel<2>);
    else if (d <= 768) go(layernorm_fwd_vec_kernel<3>);
    else go(layernorm_fwd_vec_kernel<4>);
  } else {
    pdl_launch(layernorm_fwd_kernel<float>, grid, 256, 0, s, (const float*)x, gain, shift, (float*)y, (float*)xhat, mean, rstd, rows, d);
  }
  return cudaGetLastError();
}

template <typename T>
__global__ void __launch_bounds__(256) layernorm_bwd_dx_kernel(const T* dy, const T* x,
                                                               const float* gain,
                                                               const float* mean,
                                                               const float* rstd, const T* add,
                                                               T* dx, int rows, int d) {
  pdl_wait();
  int row = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (row >= rows) return;
  long long o = (long long)row * d;
  float mu = mean[row], r = rstd[row];
  float s1 = 0.f, s2 = 0.f;
  for (int c = lane; c < d; c += 32) {
    float g = ldf(dy + o + c) * gain[c];
    float xh = (ldf(x + o + c) - mu) * r;
    s1 += g;
    s2 += g * xh;
  }
  s1 = warp_sum(s1) / d;
  s2 = warp_sum(s2) / d;
  for (int c = lane; c < d; c += 32) {
    float g = ldf(dy + o + c) * gain[c];
    float xh = (ldf(x + o + c) - mu) * r;
    float v = r * (g - s1 - xh * s2);
    if (add) v += ldf(add + o + c);
    stf(dx + o + c, v);
  }
}

// bf16 rows of d <= 256*VPL columns, d % 8 == 0: dy and x are read once (16-byte pieces kept in registers).  A warp takes
// every 8th of its CTA's `per` rows and, with `part`, adds dy xhat and dy to sums of its own in shared memory; their totals
// over the warps are the CTA's partial sums of the gain's and shift's gradients, part[cta][2][d].  (As a reduction of their own,
// which read dy and x again and had its last CTA add up to 98 partials, they took 14 us per block at 4096 x 256 and 4096 x 512, 22
// at 8192 x 768.)
template <int VPL>
__global__ void __launch_bounds__(256) layernorm_bwd_dx_vec_kernel(const bf16_t* dy, const bf16_t* x,
                                                                   const float* gain,
                                                                   const float* mean,
                                                                   const float* rstd, const bf16_t* add,
                                                                   bf16_t* dx, float* __restrict__ part, int rows, int d, int per) {
  pdl_wait();
  extern __shared__ __align__(16) float ln_sums[];      // [8 warps][2][d], with part
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* mine = ln_sums + warp * 2 * d;
  const int r0 = blockIdx.x * per, r1 = min(rows, r0 + per);
  for (int row = r0 + warp; row < r1; row += 8) {
    const long long o = (long long)row * d;
    const float mu = mean[row], r = rstd[row];
    float g[VPL][8], xh[VPL][8];
    float s1 = 0.f, s2 = 0.f;
#pragma unroll
    for (int k = 0; k < VPL; k++) {
      const int c = (k * 32 + lane) * 8;
      if (c >= d) continue;
      ld_vec<bf16_t>(dy + o + c, g[k]);
      ld_vec<bf16_t>(x + o + c, xh[k]);
      const float4 g0 = *reinterpret_cast<const float4*>(gain + c), g1 = *reinterpret_cast<const float4*>(gain + c + 4);
      const float gg[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
#pragma unroll
      for (int j = 0; j < 8; j++) xh[k][j] = (xh[k][j] - mu) * r;
      if (part) {
        float4* sg = reinterpret_cast<float4*>(mine + c);
        float4* sb = reinterpret_cast<float4*>(mine + d + c);
        const bool first = row < r0 + 8;
#pragma unroll
        for (int h = 0; h < 2; h++) {
          const float* y = g[k] + 4 * h;
          const float* n = xh[k] + 4 * h;
          float4 ag = first ? make_float4(0.f, 0.f, 0.f, 0.f) : sg[h], ab = first ? ag : sb[h];
          ag.x = fmaf(y[0], n[0], ag.x); ag.y = fmaf(y[1], n[1], ag.y); ag.z = fmaf(y[2], n[2], ag.z); ag.w = fmaf(y[3], n[3], ag.w);
          ab.x += y[0]; ab.y += y[1]; ab.z += y[2]; ab.w += y[3];
          sg[h] = ag;
          sb[h] = ab;
        }
      }
#pragma unroll
      for (int j = 0; j < 8; j++) {
        g[k][j] *= gg[j];
        s1 += g[k][j];
        s2 += g[k][j] * xh[k][j];
      }
    }
    s1 = warp_sum(s1) / d;
    s2 = warp_sum(s2) / d;
#pragma unroll
    for (int k = 0; k < VPL; k++) {
      const int c = (k * 32 + lane) * 8;
      if (c >= d) continue;
      float v[8], a[8];
      if (add) ld_vec<bf16_t>(add + o + c, a);
#pragma unroll
      for (int j = 0; j < 8; j++) {
        v[j] = r * (g[k][j] - s1 - xh[k][j] * s2);
        if (add) v[j] += a[j];
      }
      st_vec(dx + o + c, v);
    }
  }
  if (!part) return;
  if (r0 + warp >= r1)          // a warp without rows
    for (int c = lane; c < 2 * d; c += 32) mine[c] = 0.f;
  __syncthreads();
  for (int c = threadIdx.x; c < 2 * d; c += 256) {
    float t = 0.f;
#pragma unroll
    for (int k = 0; k < 8; k++) t += ln_sums[k * 2 * d + c];
    part[(long long)blockIdx.x * 2 * d + c] = t;
  }
}

// Whole turns of 8 rows, about two CTAs per SM; rows of up to 768 columns leave partial sums (48 KB of shared memory).
static int layernorm_bwd_rows(int rows) { return std::max(1, (rows + 8 * 296 - 1) / (8 * 296)) * 8; }
int layernorm_bwd_parts(int rows, int d, bool bf16) { return bf16 && d % 8 == 0 && d <= 768 ? (int)cdiv(rows, layernorm_bwd_rows(rows)) : 0; }
cudaError_t layernorm_bwd_dx(const void* dy, const void* x, const float* gain, const float* mean,
                             const float* rstd, const void* add, void* dx, float* part, int rows, int d, bool bf16,
                             cudaStream_t s) {
  const bool al = ((reinterpret_cast<uintptr_t>(dy) | reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(gain) |
                    reinterpret_cast<uintptr_t>(add) | reinterpret_cast<uintptr_t>(dx)) & 15) == 0;
  if (bf16 && al && d % 8 == 0 && d <= 1024) {
    const int per = part ? layernorm_bwd_rows(rows) : 8;
    auto go = [&](auto kernel) {
      pdl_launch(kernel, cdiv(rows, per), 256, part ? (size_t)16 * d * sizeof(float) : 0, s, (const bf16_t*)dy, (const bf16_t*)x, gain, mean, rstd,
                 (const bf16_t*)add, (bf16_t*)dx, part, rows, d, per);
    };
    if (d <= 256) go(layernorm_bwd_dx_vec_kernel<1>);
    else if (d <= 512) go(layernorm_bwd_dx_vec_kernel<2>);
    else if (d <= 768) go(layernorm_bwd_dx_vec_kernel<3>);
    else go(layernorm_bwd_dx_vec_kernel<4>);
    return cudaGetLastError();
  }
  if (part) return cudaErrorInvalidValue;      // (buffers of the model are aligned)
  if (bf16) pdl_launch(layernorm_bwd_dx_kernel<bf16_t>, cdiv(rows, 8), 256, 0, s, (const bf16_t*)dy, (const bf16_t*)x, gain, mean, rstd, (const bf16_t*)add, (bf16_t*)dx, rows, d);
  else pdl_launch(layernorm_bwd_dx_kernel<float>, cdiv(rows, 8), 256, 0, s, (const float*)dy, (const float*)x, gain, mean, rstd, (const float*)add, (float*)dx, rows, d);
  return cudaGetLastError();
}

// dgain / dshift partial sums: a CTA takes a strip of 32*VEC columns and one chunk of rows, a thread
// VEC adjacent columns (16-byte loads of dy and x) and every 8th row, four rows in flight.
template <typename T>
__device__ __forceinline__ void layernorm_param_grad_body(const T* dy, const T* x,
                                                          const float* mean,
                                                          const float* rstd,
                                                          float* __restrict__ ws, float* __restrict__ dgain,
                                                          float* __restrict__ dshift, int rows, int d, int chunks,
                                                          int* tickets, int bx, int by, float* smem) {   // 16 * 32*VEC floats
  constexpr int VEC = VecOf<T>::N;
  constexpr int SW = 32 * VEC;
  float (*sg)[SW] = reinterpret_cast<float (*)[SW]>(smem);
  float (*sb)[SW] = reinterpret_cast<float (*)[SW]>(smem + 8 * SW);
  const int cx = threadIdx.x & 31, ry = threadIdx.x >> 5;
  const int c = bx * SW + cx * VEC;
  const int per = (rows + chunks - 1) / chunks;
  const int rb = by * per, re = min(rows, rb + per);
  const bool vec = (c + VEC <= d) && (d % VEC == 0);
  float ag[VEC], ab[VEC];
#pragma unroll
  for (int j = 0; j < VEC; j++) ag[j] = ab[j] = 0.f;
  if (c < d) {
    if (vec) {
      int r = rb + ry;
      for (; r + 24 < re; r += 32) {
        float gy[4][VEC], xv[4][VEC], mu[4], rs[4];
#pragma unroll
        for (int u = 0; u < 4; u++) {
          ld_vec<T>(dy + (long long)(r + 8 * u) * d + c, gy[u]);
          ld_vec<T>(x + (long long)(r + 8 * u) * d + c, xv[u]);
          mu[u] = mean[r + 8 * u];
          rs[u] = rstd[r + 8 * u];
        }
#pragma unroll
        for (int u = 0; u < 4; u++)
#pragma unroll
          for (int j = 0; j < VEC; j++) {
            ag[j] = fmaf(gy[u][j], (xv[u][j] - mu[u]) * rs[u], ag[j]);
            ab[j] += gy[u][j];
          }
      }
      for (; r < re; r += 8) {
        float gy[VEC], xv[VEC];
        ld_vec<T>(dy + (long long)r * d + c, gy);
        ld_vec<T>(x + (long long)r * d + c, xv);
        const float mu = mean[r], rs = rstd[r];
#pragma unroll
        for (int j = 0; j < VEC; j++) {
          ag[j] = fmaf(gy[j], (xv[j] - mu) * rs, ag[j]);
          ab[j] += gy[j];
        }
      }
    } else {
      for (int r = rb + ry; r < re; r += 8) {
        const float mu = mean[r], rs = rstd[r];
#pragma unroll
        for (int j = 0; j < VEC; j++)
          if (c + j < d) {
            const float g = ldf(dy + (long long)r * d + c + j);
            ag[j] = fmaf(g, (ldf(x + (long long)r * d + c + j) - mu) * rs, ag[j]);
            ab[j] += g;
          }
      }
    }
  }
#pragma unroll
  for (int j = 0; j < VEC; j++) { sg[ry][cx * VEC + j] = ag[j]; sb[ry][cx * VEC + j] = ab[j]; }
  __syncthreads();
  float* pg = chunks == 1 ? dgain : ws + (long long)by * d;
  float* pb = chunks == 1 ? dshift : ws + (long long)(chunks + by) * d;
  for (int i = threadIdx.x; i < SW; i += 256) {
    const int cc = bx * SW + i;
    if (cc < d) {
      float tg = 0.f, tb = 0.f;
#pragma unroll
      for (int k = 0; k < 8; k++) { tg += sg[k][i]; tb += sb[k][i]; }
      pg[cc] = tg;
      pb[cc] = tb;
    }
  }
  if (chunks == 1) return;
  if (!last_cta(tickets + bx, chunks)) return;
  for (int i = threadIdx.x; i < SW; i += 256) {
    const int cc = bx * SW + i;
    if (cc < d) {
      dgain[cc] = ordered_sum(ws + cc, d, chunks);
      dshift[cc] = ordered_sum(ws + (long long)chunks * d + cc, d, chunks);
    }
  }
}

// A LayerNorm y = xhat g + b whose only reader is a Linear (weights W [n, d], output gradient dY), and whose input gradient
// nobody wants.  With G = dY^T xhat, formed by that Linear's weight-gradient GEMM in the place of dY^T y, and db = column sums
// of dY, everything follows from sums over the Linear's n outputs, without dY W and a pass over it and x:
//     dW[j,c] = G[j,c] g[c] + db[j] b[c],     dg[c] = sum_j W[j,c] G[j,c],     dshift[c] = sum_j W[j,c] db[j].
// (xhat is rounded where y was before; no division by g.)  G is overwritten by dW; db comes as `parts` rows of partial sums.
// A CTA takes a strip of 128 columns and LNW_ROWS rows, a thread four adjacent columns and every 8th row, four of them in
// flight; the strip's last CTA adds the partial sums in order.
// Bound by one read of G and W and one write of dW, and the latency of a launch that the block has anyway.
constexpr int LNW_ROWS = 64;
// (not inlined: its registers would spill the other jobs')
template <typename T, bool VECTOR>
__device__ __noinline__ void layernorm_from_wgrad_body(const ReduceJob& q, int bx, int by, float* smem) {      // LNW_ROWS + 2 * 8 * 128 floats
  float* G = q.io;
  const T* W = (const T*)q.X;
  const float* db = (const float*)q.X2;
  const int n = q.rows, d = q.cols, chunks = q.chunks;
  const int cx = threadIdx.x & 31, ry = threadIdx.x >> 5, c = bx * 128 + cx * 4, valid = d - c;
  const int per = (n + chunks - 1) / chunks, rb = by * per, re = min(n, rb + per);
  float4 ag = make_float4(0.f, 0.f, 0.f, 0.f), ab = ag;
  float* sdb = smem;                   // this chunk's db (per <= LNW_ROWS)
  if ((int)threadIdx.x < re - rb) {
    float t = 0.f;
    for (int i = 0; i < q.parts; i += 4) {
      float v[4];
#pragma unroll
      for (int u = 0; u < 4; u++) v[u] = i + u < q.parts ? db[(long long)(i + u) * n + rb + threadIdx.x] : 0.f;
      t += (v[0] + v[1]) + (v[2] + v[3]);
    }
    sdb[threadIdx.x] = t;
  }
  __syncthreads();
  if (valid > 0) {
    const float4 g = ld4_guard(q.a + c, valid, VECTOR), b = ld4_guard(q.b + c, valid, VECTOR);
    for (int r0 = rb + ry; r0 < re; r0 += 32) {
      float4 x[4], w[4];
      float s[4];
#pragma unroll
      for (int k = 0; k < 4; k++) {
        const int r = r0 + 8 * k;
        const bool ok = r < re;
        x[k] = ok ? ld4_guard(G + (long long)r * d + c, valid, VECTOR) : make_float4(0.f, 0.f, 0.f, 0.f);
        w[k] = ok ? ld4_guard(W + (long long)r * d + c, valid, VECTOR) : make_float4(0.f, 0.f, 0.f, 0.f);
        s[k] = ok ? sdb[r - rb] : 0.f;
      }
#pragma unroll
      for (int k = 0; k < 4; k++) {
        ag.x = fmaf(w[k].x, x[k].x, ag.x); ag.y = fmaf(w[k].y, x[k].y, ag.y); ag.z = fmaf(w[k].z, x[k].z, ag.z); ag.w = fmaf(w[k].w, x[k].w, ag.w);
        ab.x = fmaf(w[k].x, s[k], ab.x); ab.y = fmaf(w[k].y, s[k], ab.y); ab.z = fmaf(w[k].z, s[k], ab.z); ab.w = fmaf(w[k].w, s[k], ab.w);
        if (r0 + 8 * k < re) {
          const float4 o = make_float4(fmaf(x[k].x, g.x, s[k] * b.x), fmaf(x[k].y, g.y, s[k] * b.y), fmaf(x[k].z, g.z, s[k] * b.z), fmaf(x[k].w, g.w, s[k] * b.w));
          float* dst = G + (long long)(r0 + 8 * k) * d + c;
          if (VECTOR) {
            *reinterpret_cast<float4*>(dst) = o;
          } else {
            dst[0] = o.x;
            if (valid > 1) dst[1] = o.y;
            if (valid > 2) dst[2] = o.z;
            if (valid > 3) dst[3] = o.w;
          }
        }
      }
    }
  }
  float (*sm)[8][128] = reinterpret_cast<float (*)[8][128]>(smem + LNW_ROWS);
  *reinterpret_cast<float4*>(&sm[0][ry][cx * 4]) = ag;
  *reinterpret_cast<float4*>(&sm[1][ry][cx * 4]) = ab;
  __syncthreads();
  const int half = threadIdx.x >> 7, col = threadIdx.x & 127, cc = bx * 128 + col;      // 128 threads for the gain, 128 for the shift
  float* out = half ? q.out1 : q.out0;
  if (cc < d) {
    float t = 0.f;
#pragma unroll
    for (int k = 0; k < 8; k++) t += sm[half][k][col];
    if (chunks == 1) out[cc] = t;
    else q.ws[(long long)(half * chunks + by) * d + cc] = t;
  }
  if (chunks == 1 || !last_cta(q.tickets + bx, chunks)) return;
  if (cc < d) out[cc] = ordered_sum(q.ws + (long long)half * chunks * d + cc, d, chunks);
}

// Several column reductions in ONE launch: the bias gradients and LayerNorm gain/shift gradients of
// a block are each a few MB of input, so separate launches spend most of their time ramping up and
// waiting for their last CTA.  A CTA looks its job up in a table (at most a few entries).
// The table travels as a kernel argument: a CTA finds and reads its job in constant memory instead of walking a
// table in device memory with dependent loads (a 512 x 128 MLP block's five jobs: 14.7 us between events, now 11.8).
// Three CTAs to an SM (80 registers) or four (64), us between events: blocks of towers 512 and 1024 wide, whose jobs are column
// sums, 10.7 and 12.8 either way; transformer blocks of d 256, 512, 768, 1024 16.9, 16.9, 25.3, 27.1 or 17.9, 18.9, 27.2, 25.1.
constexpr int OUTER_ROWS = 32;
template <int MAX>
struct ReduceTable {
  int n;
  ReduceJob job[MAX];
};
template <int MAX>
__global__ void __launch_bounds__(256, 3) reduce_batch_kernel(const __grid_constant__ ReduceTable<MAX> table) {
  pdl_wait();
  __shared__ __align__(16) float smem[16 * 256];   // the largest need: gain and shift partials of a 256-column bf16 strip
  int j = 0;
  while (j + 1 < table.n && (int)blockIdx.x >= table.job[j + 1].cta_begin) j++;
  const ReduceJob& job = table.job[j];
  const int local = (int)blockIdx.x - job.cta_begin;
  const int bx = local % job.strips, by = local / job.strips;
  if (job.kind == 2) {   // split-K partials -> fp32 result, 1024 outputs per CTA
    splitk_reduce_v4_body<false>((const float4*)job.X, job.rows, job.mn / 4, job.cols / 4, job.out0, job.ldx,
                                 (long long)local * 256 + threadIdx.x);
    return;
  }
  if (job.kind == 5) {
    const bool vec = job.cols % 4 == 0 && ((reinterpret_cast<uintptr_t>(job.io) | reinterpret_cast<uintptr_t>(job.X) | reinterpret_cast<uintptr_t>(job.a) | reinterpret_cast<uintptr_t>(job.b)) & 15) == 0;
    if (job.x_f32) { if (vec) layernorm_from_wgrad_body<float, true>(job, bx, by, smem); else layernorm_from_wgrad_body<float, false>(job, bx, by, smem); }
    else { if (vec) layernorm_from_wgrad_body<bf16_t, true>(job, bx, by, smem); else layernorm_from_wgrad_body<bf16_t, false>(job, bx, by, smem); }
    return;
  }
  if (job.kind == 4) {   // outer product with a row that is still in partial sums: OUTER_ROWS x 256 results
    const int cg = threadIdx.x & 63, rg = threadIdx.x >> 6, c = bx % ((job.cols + 255) / 256) * 256 + cg * 4;
    const int r0 = bx / ((job.cols + 255) / 256) * OUTER_ROWS, re = min(job.rows, r0 + OUTER_ROWS), valid = job.cols - c;
    const bool vec = valid >= 4 && job.cols % 4 == 0 && ((reinterpret_cast<uintptr_t>(job.X) | reinterpret_cast<uintptr_t>(job.out0)) & 15) == 0;
    float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
    auto part = [&](int k) {
      return k < job.parts && valid > 0 ? ld4_guard((const float*)job.X + (long long)k * job.cols + c, valid, vec) : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    for (int k = rg; k < job.parts; k += 16) {         // partials rg, rg + 4, ..: four loads in flight
      const float4 a = part(k), b = part(k + 4), e = part(k + 8), f = part(k + 12);
      t.x += a.x + b.x + e.x + f.x; t.y += a.y + b.y + e.y + f.y; t.z += a.z + b.z + e.z + f.z; t.w += a.w + b.w + e.w + f.w;
    }
    float4* row = reinterpret_cast<float4*>(smem);
    row[rg * 64 + cg] = t;
    __syncthreads();
    t = row[cg];
#pragma unroll
    for (int k = 1; k < 4; k++) { const float4 a = row[k * 64 + cg]; t.x += a.x; t.y += a.y; t.z += a.z; t.w += a.w; }
    for (int r = r0 + rg; r < re; r += 4) {
      const float f = job.a[r];
      float* o = job.out0 + (long long)r * job.cols + c;
      if (vec) {
        *reinterpret_cast<float4*>(o) = make_float4(f * t.x, f * t.y, f * t.z, f * t.w);
      } else {
        if (valid > 0) o[0] = f * t.x;
        if (valid > 1) o[1] = f * t.y;
        if (valid > 2) o[2] = f * t.z;
        if (valid > 3) o[3] = f * t.w;
      }
    }
    return;
  }
  if (job.kind == 3) {   // sum of a vector, times a row of factors
    const float* x = (const float*)job.X;
    float a = 0.f;
    for (int i0 = threadIdx.x; i0 < job.rows; i0 += 8 * 256) {
      float v[8];
#pragma unroll
      for (int u = 0; u < 8; u++) v[u] = i0 + u * 256 < job.rows ? x[i0 + u * 256] : 0.f;
#pragma unroll
      for (int u = 0; u < 8; u++) a += v[u];
    }
    a = warp_sum(a);
    if ((threadIdx.x & 31) == 0) smem[threadIdx.x >> 5] = a;
    __syncthreads();
    float t = smem[0];
#pragma unroll
    for (int k = 1; k < 8; k++) t += smem[k];
    t *= job.scale;
    const int c = local * 256 + threadIdx.x;
    if (c < job.cols) job.out0[c] = job.b ? t * job.b[c] : t;
    return;
  }
  if (job.kind == 0) {
    if (job.x_f32)
      colsum_body<float>((const float*)job.X, job.ldx, job.rows, job.cols, job.a, job.ws, job.out0, job.chunks, job.dact, job.b, job.tickets, bx, by, smem);
    else
      colsum_body<bf16_t>((const bf16_t*)job.X, job.ldx, job.rows, job.cols, job.a, job.ws, job.out0, job.chunks, job.dact, job.b, job.tickets, bx, by, smem);
  } else {
    if (job.x_f32)
      layernorm_param_grad_body<float>((const float*)job.X, (const float*)job.X2, job.a, job.b, job.ws, job.out0, job.out1, job.rows, job.cols, job.chunks, job.tickets, bx, by, smem);
    else
      layernorm_param_grad_body<bf16_t>((const bf16_t*)job.X, (const bf16_t*)job.X2, job.a, job.b, job.ws, job.out0, job.out1, job.rows, job.cols, job.chunks, job.tickets, bx, by, smem);
  }
}

int reduce_job_strips(const ReduceJob& j) {
  if (j.kind == 5) return (int)cdiv(j.cols, 128);
  if (j.kind == 4) return (int)(cdiv(j.cols, 256) * cdiv(j.rows, OUTER_ROWS));
  if (j.kind == 2) return (int)cdiv(j.mn / 4, 256);
  if (j.kind == 3) return (int)cdiv(j.cols, 256);
  return (int)cdiv(j.cols, j.x_f32 ? 128 : 256);
}

int layernorm_from_wgrad_chunks(int n) { return (n + LNW_ROWS - 1) / LNW_ROWS; }

template <int MAX>
static cudaError_t reduce_batch_t(const ReduceJob* jobs, int n, int total_ctas, cudaStream_t s) {
  ReduceTable<MAX> t;
  t.n = n;
  std::copy(jobs, jobs + n, t.job);
  pdl_launch(reduce_batch_kernel<MAX>, total_ctas, 256, 0, s, t);
  return cudaGetLastError();
}
cudaError_t reduce_batch(const ReduceJob* jobs, int njobs, int total_ctas, cudaStream_t s) {
  if (njobs <= 0 || total_ctas <= 0) return cudaSuccess;
  if (njobs > REDUCE_MAX_JOBS) return cudaErrorInvalidValue;
  return njobs <= 8 ? reduce_batch_t<8>(jobs, njobs, total_ctas, s) : reduce_batch_t<REDUCE_MAX_JOBS>(jobs, njobs, total_ctas, s);
}

// ------------------------------------------------------------------------------------------
// causal attention, flash-style (no T x T matrix in memory), fp32 SIMT
// tiles of 32 queries x 32 keys; a warp owns 4 rows; lanes run over the 32 keys of a tile for
// the scores and over head columns (lane, lane+32, ..) for the accumulators.
// ------------------------------------------------------------------------------------------
#define ATT_MAXC 4  // head width <= 128

template <typename T>
__device__ __forceinline__ void att_load_tile(float* dst, int ldk, const T* src, long long ld, int r0,
                                              int T_, int dh) {
  for (int i = threadIdx.x; i < 32 * dh; i += 256) {
    int r = i / dh, c = i - r * dh;
    int t = r0 + r;
    dst[r * ldk + c] = t < T_ ? ldf(src + (long long)t * ld + c) : 0.f;
  }
}

template <typename T>
__global__ void __launch_bounds__(256) attn_fwd_kernel(const T* qkv, T* __restrict__ o,
                                                       float* __restrict__ lse, int T_, int H, int dh,
                                                       float scale) {
  pdl_wait();
  extern __shared__ float sm[];
  const int ldk = dh + 1;
  float* Qs = sm;
  float* Ks = Qs + 32 * ldk;
  float* Vs = Ks + 32 * ldk;
  const int q0 = blockIdx.x * 32, h = blockIdx.y, b = blockIdx.z;
  const int d = H * dh;
  const long long ld = 3LL * d;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const T* base = qkv + (long long)b * T_ * ld + h * dh;
  att_load_tile(Qs, ldk, base, ld, q0, T_, dh);
  float mrow[4], lrow[4], acc[4][ATT_MAXC];
#pragma unroll
  for (int r = 0; r < 4; r++) {
    mrow[r] = -INFINITY;
    lrow[r] = 0.f;
#pragma unroll
    for (int cc = 0; cc < ATT_MAXC; cc++) acc[r][cc] = 0.f;
  }
  for (int j0 = 0; j0 <= q0; j0 += 32) {
    __syncthreads();
    att_load_tile(Ks, ldk, base + d, ld, j0, T_, dh);
    att_load_tile(Vs, ldk, base + 2 * d, ld, j0, T_, dh);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 4; r++) {
      const int il = warp * 4 + r, i = q0 + il;
      if (i >= T_) continue;
      const int j = j0 + lane;
      float sc = 0.f;
      for (int c = 0; c < dh; c++) sc = fmaf(Qs[il * ldk + c], Ks[lane * ldk + c], sc);
      sc *= scale;
      const bool valid = j <= i;
      if (!valid) sc = -INFINITY;
      float mnew = fmaxf(mrow[r], warp_max(sc));
      float p = valid ? expf(sc - mnew) : 0.f;
      float corr = expf(mrow[r] - mnew);
      lrow[r] = lrow[r] * corr + warp_sum(p);
      mrow[r] = mnew;
#pragma unroll
      for (int cc = 0; cc < ATT_MAXC; cc++) acc[r][cc] *= corr;
      for (int jj = 0; jj < 32; jj++) {
        float pj = __shfl_sync(0xffffffffu, p, jj);
#pragma unroll
        for (int cc = 0; cc < ATT_MAXC; cc++) {
          int c = lane + 32 * cc;
          if (c < dh) acc[r][cc] = fmaf(pj, Vs[jj * ldk + c], acc[r][cc]);
        }
      }
    }
  }
#pragma unroll
  for (int r = 0; r < 4; r++) {
    const int i = q0 + warp * 4 + r;
    if (i >= T_) continue;
    float inv = 1.f / lrow[r];
#pragma unroll
    for (int cc = 0; cc < ATT_MAXC; cc++) {
      int c = lane + 32 * cc;
      if (c < dh) stf(o + ((long long)b * T_ + i) * d + h * dh + c, acc[r][cc] * inv);
    }
    if (lane == 0) lse[((long long)b * H + h) * T_ + i] = mrow[r] + logf(lrow[r]);
  }
}

template <typename T>
__global__ void __launch_bounds__(256) attn_delta_kernel(const T* o, const T* dout,
                                                         float* __restrict__ delta, int rows, int T_, int H,
                                                         int dh) {
  pdl_wait();
  // one warp per (row, head)
  long long w = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
  int lane = threadIdx.x & 31;
  if (w >= (long long)rows * H) return;
  int n = (int)(w / H), h = (int)(w % H);
  long long off = (long long)n * H * dh + h * dh;
  float s = 0.f;
  for (int c = lane; c < dh; c += 32) s += ldf(o + off + c) * ldf(dout + off + c);
  s = warp_sum(s);
  if (lane == 0) {
    int b = n / T_, t = n % T_;
    delta[((long long)b * H + h) * T_ + t] = s;
  }
}

// dK, dV for a tile of 32 keys: loop over the query tiles at or after it.
template <typename T>
__global__ void __launch_bounds__(256) attn_bwd_kv_kernel(const T* qkv, const T* dout,
                                                          const float* lse,
                                                          const float* delta, T* __restrict__ dqkv,
                                                          int T_, int H, int dh, float scale) {
  pdl_wait();
  extern __shared__ float sm[];
  const int ldk = dh + 1;
  float* Ks = sm;
  float* Vs = Ks + 32 * ldk;
  float* Qs = Vs + 32 * ldk;
  float* Ds = Qs + 32 * ldk;
  float* Ls = Ds + 32 * ldk;  // [32] lse
  float* Es = Ls + 32;        // [32] delta
  const int k0 = blockIdx.x * 32, h = blockIdx.y, b = blockIdx.z;
  const int d = H * dh;
  const long long ld = 3LL * d;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const T* base = qkv + (long long)b * T_ * ld + h * dh;
  const T* dob = dout + (long long)b * T_ * d + h * dh;
  att_load_tile(Ks, ldk, base + d, ld, k0, T_, dh);
  att_load_tile(Vs, ldk, base + 2 * d, ld, k0, T_, dh);
  float dk[4][ATT_MAXC], dv[4][ATT_MAXC];
#pragma unroll
  for (int r = 0; r < 4; r++)
#pragma unroll
    for (int cc = 0; cc < ATT_MAXC; cc++) dk[r][cc] = dv[r][cc] = 0.f;
  for (int i0 = k0; i0 < T_; i0 += 32) {
    __syncthreads();
    att_load_tile(Qs, ldk, base, ld, i0, T_, dh);
    att_load_tile(Ds, ldk, dob, (long long)d, i0, T_, dh);
    if (threadIdx.x < 32) {
      int i = i0 + threadIdx.x;
      Ls[threadIdx.x] = i < T_ ? lse[((long long)b * H + h) * T_ + i] : 0.f;
      Es[threadIdx.x] = i < T_ ? delta[((long long)b * H + h) * T_ + i] : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 4; r++) {
      const int jl = warp * 4 + r, j = k0 + jl;
      if (j >= T_) continue;
      const int i = i0 + lane;
      float sc = 0.f, dp = 0.f;
      for (int c = 0; c < dh; c++) {
        sc = fmaf(Qs[lane * ldk + c], Ks[jl * ldk + c], sc);
        dp = fmaf(Ds[lane * ldk + c], Vs[jl * ldk + c], dp);
      }
      const bool valid = i < T_ && j <= i;
      float p = valid ? expf(sc * scale - Ls[lane]) : 0.f;
      float ds = p * (dp - Es[lane]);
      for (int ii = 0; ii < 32; ii++) {
        float pi = __shfl_sync(0xffffffffu, p, ii);
        float di = __shfl_sync(0xffffffffu, ds, ii);
#pragma unroll
        for (int cc = 0; cc < ATT_MAXC; cc++) {
          int c = lane + 32 * cc;
          if (c < dh) {
            dv[r][cc] = fmaf(pi, Ds[ii * ldk + c], dv[r][cc]);
            dk[r][cc] = fmaf(di, Qs[ii * ldk + c], dk[r][cc]);
          }
        }
      }
    }
  }
#pragma unroll
  for (int r = 0; r < 4; r++) {
    const int j = k0 + warp * 4 + r;
    if (j >= T_) continue;
    T* row = dqkv + ((long long)b * T_ + j) * ld + h * dh;
#pragma unroll
    for (int cc = 0; cc < ATT_MAXC; cc++) {
      int c = lane + 32 * cc;
      if (c < dh) {
        stf(row + d + c, dk[r][cc] * scale);
        stf(row + 2 * d + c, dv[r][cc]);
      }
    }
  }
}

// dQ for a tile of 32 queries: loop over the key tiles at or before it.
template <typename T>
__global__ void __launch_bounds__(256) attn_bwd_q_kernel(const T* qkv, const T* dout,
                                                         const float* lse,
                                                         const float* delta, T* __restrict__ dqkv,
                                                         int T_, int H, int dh, float scale) {
  pdl_wait();
  extern __shared__ float sm[];
  const int ldk = dh + 1;
  float* Qs = sm;
  float* Ds = Qs + 32 * ldk;
  float* Ks = Ds + 32 * ldk;
  float* Vs = Ks + 32 * ldk;
  const int q0 = blockIdx.x * 32, h = blockIdx.y, b = blockIdx.z;
  const int d = H * dh;
  const long long ld = 3LL * d;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const T* base = qkv + (long long)b * T_ * ld + h * dh;
  const T* dob = dout + (long long)b * T_ * d + h * dh;
  att_load_tile(Qs, ldk, base, ld, q0, T_, dh);
  att_load_tile(Ds, ldk, dob, (long long)d, q0, T_, dh);
  float dq[4][ATT_MAXC], lrow[4], erow[4];
#pragma unroll
  for (int r = 0; r < 4; r++) {
    int i = q0 + warp * 4 + r;
    lrow[r] = i < T_ ? lse[((long long)b * H + h) * T_ + i] : 0.f;
    erow[r] = i < T_ ? delta[((long long)b * H + h) * T_ + i] : 0.f;
#pragma unroll
    for (int cc = 0; cc < ATT_MAXC; cc++) dq[r][cc] = 0.f;
  }
  for (int j0 = 0; j0 <= q0; j0 += 32) {
    __syncthreads();
    att_load_tile(Ks, ldk, base + d, ld, j0, T_, dh);
    att_load_tile(Vs, ldk, base + 2 * d, ld, j0, T_, dh);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 4; r++) {
      const int il = warp * 4 + r, i = q0 + il;
      if (i >= T_) continue;
      const int j = j0 + lane;
      float sc = 0.f, dp = 0.f;
      for (int c = 0; c < dh; c++) {
        sc = fmaf(Qs[il * ldk + c], Ks[lane * ldk + c], sc);
        dp = fmaf(Ds[il * ldk + c], Vs[lane * ldk + c], dp);
      }
      float p = j <= i ? expf(sc * scale - lrow[r]) : 0.f;
      float ds = p * (dp - erow[r]);
      for (int jj = 0; jj < 32; jj++) {
        float dj = __shfl_sync(0xffffffffu, ds, jj);
#pragma unroll
        for (int cc = 0; cc < ATT_MAXC; cc++) {
          int c = lane + 32 * cc;
          if (c < dh) dq[r][cc] = fmaf(dj, Ks[jj * ldk + c], dq[r][cc]);
        }
      }
    }
  }
#pragma unroll
  for (int r = 0; r < 4; r++) {
    const int i = q0 + warp * 4 + r;
    if (i >= T_) continue;
    T* row = dqkv + ((long long)b * T_ + i) * ld + h * dh;
#pragma unroll
    for (int cc = 0; cc < ATT_MAXC; cc++) {
      int c = lane + 32 * cc;
      if (c < dh) stf(row + c, dq[r][cc] * scale);
    }
  }
}

template <typename K>
static cudaError_t set_smem(K kernel, size_t bytes) {
  if (bytes <= 48 * 1024) return cudaSuccess;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <typename T>
static cudaError_t attention_fwd_t(const T* qkv, T* o, float* lse, int batch, int T_, int heads, int dh,
                                   cudaStream_t s) {
  size_t smem = (size_t)3 * 32 * (dh + 1) * sizeof(float);
  cudaError_t e = set_smem(attn_fwd_kernel<T>, smem);
  if (e != cudaSuccess) return e;
  dim3 grid(cdiv(T_, 32), heads, batch);
  pdl_launch(attn_fwd_kernel<T>, grid, 256, smem, s, qkv, o, lse, T_, heads, dh, 1.f / sqrtf((float)dh));
  return cudaGetLastError();
}

// 0: fp32 SIMT / mma.sync kernels only; 1 (default): tcgen05 kernels where they apply
static int attention_tc_mode() { return getenv("ERASE_ATTN_TC") ? atoi(getenv("ERASE_ATTN_TC")) : 1; }

cudaError_t attention_fwd(const void* qkv, void* o, float* lse, int batch, int T_, int heads, int dh,
                          bool bf16, cudaStream_t s, int* status) {
  if (dh > 32 * ATT_MAXC) return cudaErrorInvalidValue;
  if (bf16 && attention_tc_mode() && attention_tc_supported(dh, heads * dh, qkv, o))
    return attention_fwd_tc(qkv, o, lse, batch, T_, heads, status, s);
  if (bf16 && attention_mma_supported(dh, heads * dh)) return attention_fwd_mma(qkv, o, lse, batch, T_, heads, s);
  return bf16 ? attention_fwd_t<bf16_t>((const bf16_t*)qkv, (bf16_t*)o, lse, batch, T_, heads, dh, s)
              : attention_fwd_t<float>((const float*)qkv, (float*)o, lse, batch, T_, heads, dh, s);
}

template <typename T>
static cudaError_t attention_bwd_t(const T* qkv, const T* o, const T* dout, const float* lse, float* delta,
                                   T* dqkv, int batch, int T_, int heads, int dh, cudaStream_t s) {
  int rows = batch * T_;
  pdl_launch(attn_delta_kernel<T>, cdiv((long long)rows * heads, 8), 256, 0, s, o, dout, delta, rows, T_, heads, dh);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  size_t smem = ((size_t)4 * 32 * (dh + 1) + 64) * sizeof(float);
  if ((e = set_smem(attn_bwd_kv_kernel<T>, smem)) != cudaSuccess) return e;
  if ((e = set_smem(attn_bwd_q_kernel<T>, smem)) != cudaSuccess) return e;
  dim3 grid(cdiv(T_, 32), heads, batch);
  float scale = 1.f / sqrtf((float)dh);
  pdl_launch(attn_bwd_kv_kernel<T>, grid, 256, smem, s, qkv, dout, lse, delta, dqkv, T_, heads, dh, scale);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  pdl_launch(attn_bwd_q_kernel<T>, grid, 256, smem, s, qkv, dout, lse, delta, dqkv, T_, heads, dh, scale);
  return cudaGetLastError();
}

cudaError_t attention_bwd(const void* qkv, const void* o, const void* dout, const float* lse, float* delta,
                          void* dqkv, int batch, int T_, int heads, int dh, bool bf16, cudaStream_t s, int* status) {
  if (dh > 32 * ATT_MAXC) return cudaErrorInvalidValue;
  if (bf16 && attention_tc_mode() && attention_tc_supported(dh, heads * dh, qkv, dout) && ((reinterpret_cast<uintptr_t>(dqkv) | reinterpret_cast<uintptr_t>(o)) & 15) == 0) {
    return attention_bwd_tc(qkv, o, dout, lse, delta, dqkv, batch, T_, heads, status, s);
  }
  if (bf16 && attention_mma_supported(dh, heads * dh)) return attention_bwd_mma(qkv, o, dout, lse, delta, dqkv, batch, T_, heads, s);
  return bf16 ? attention_bwd_t<bf16_t>((const bf16_t*)qkv, (const bf16_t*)o, (const bf16_t*)dout, lse, delta, (bf16_t*)dqkv, batch, T_, heads, dh, s)
              : attention_bwd_t<float>((const float*)qkv, (const float*)o, (const float*)dout, lse, delta, (float*)dqkv, batch, T_, heads, dh, s);
}

// ------------------------------------------------------------------------------------------
// losses
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ float block_reduce_256(float v, float* sm, bool is_max) {
  int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  v = is_max ? warp_max(v) : warp_sum(v);
  __syncthreads();
  if (lane == 0) sm[warp] = v;
  __syncthreads();
  float r = sm[0];
#pragma unroll
  for (int i = 1; i < 8; i++) r = is_max ? fmaxf(r, sm[i]) : r + sm[i];
  return r;
}

template <typename T>
__global__ void __launch_bounds__(256) softmax_ce_kernel(T* __restrict__ logits, const int32_t* ids,
                                                         int T_, float* __restrict__ rowloss, int V,
                                                         float inv_rows) {
  pdl_wait();
  __shared__ float sm[8];
  const int row = blockIdx.x;
  T* p = logits + (long long)row * V;
  // an id out of range was reported by the input staging; here it must only not be used as an index
  const int tgt = min(max(ids[(long long)(row / T_) * (T_ + 1) + (row % T_) + 1], 0), V - 1);
  const float lt = ldf(p + tgt);
  float mx = -INFINITY;
  for (int v = threadIdx.x; v < V; v += 256) mx = fmaxf(mx, ldf(p + v));
  mx = block_reduce_256(mx, sm, true);
  float se = 0.f;
  for (int v = threadIdx.x; v < V; v += 256) se += expf(ldf(p + v) - mx);
  se = block_reduce_256(se, sm, false);
  const float lse = mx + logf(se);
  __syncthreads();  // lt was read by every thread before any store below
  for (int v = threadIdx.x; v < V; v += 256) {
    float g = expf(ldf(p + v) - lse) - (v == tgt ? 1.f : 0.f);
    stf(p + v, g * inv_rows);
  }
  if (threadIdx.x == 0) rowloss[row] = lse - lt;
}

// bf16 rows kept in registers: one 16-byte load and one 16-byte store per 8 logits, nothing re-read.
// A thread owns vectors tid, tid+THREADS, ...; VPT of them (V <= THREADS*8*VPT, V % 8 == 0).
template <int THREADS, int VPT>
__global__ void __launch_bounds__(THREADS) softmax_ce_reg_kernel(bf16_t* __restrict__ logits,
                                                                  const int32_t* ids, int T_,
                                                                  float* __restrict__ rowloss, int V, float inv_rows) {
  pdl_wait();
  __shared__ float sm[THREADS / 32];
  const int row = blockIdx.x, nvec = V >> 3;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint4* p = reinterpret_cast<uint4*>(logits + (long long)row * V);
  const int tgt = ids[(long long)(row / T_) * (T_ + 1) + (row % T_) + 1];
  const float L2E = 1.4426950408889634f;
  float x[VPT][8];
  float mx = -INFINITY, lt = 0.f;
#pragma unroll
  for (int k = 0; k < VPT; k++) {
    const int i = threadIdx.x + k * THREADS;
    if (i < nvec) {
      const uint4 q = p[i];
      const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
      for (int j = 0; j < 4; j++) {
        x[k][2 * j] = __uint_as_float(w[j] << 16);
        x[k][2 * j + 1] = __uint_as_float(w[j] & 0xffff0000u);
      }
#pragma unroll
      for (int j = 0; j < 8; j++) {
        mx = fmaxf(mx, x[k][j]);
        if (i * 8 + j == tgt) lt = x[k][j];
      }
    } else {
#pragma unroll
      for (int j = 0; j < 8; j++) x[k][j] = -INFINITY;
    }
  }
  auto block_reduce = [&](float v, bool is_max) {
    v = is_max ? warp_max(v) : warp_sum(v);
    __syncthreads();
    if (lane == 0) sm[warp] = v;
    __syncthreads();
    float r = sm[0];
    for (int i = 1; i < THREADS / 32; i++) r = is_max ? fmaxf(r, sm[i]) : r + sm[i];
    return r;
  };
  mx = block_reduce(mx, true);
  float se = 0.f;
#pragma unroll
  for (int k = 0; k < VPT; k++)
#pragma unroll
    for (int j = 0; j < 8; j++) {
      x[k][j] = exp2f((x[k][j] - mx) * L2E);     // keep exp(x - max): the probabilities are this over the sum
      se += x[k][j];
    }
  se = block_reduce(se, false);
  const float lse = mx + logf(se);
  const float inv_se = 1.f / se;
#pragma unroll
  for (int k = 0; k < VPT; k++) {
    const int i = threadIdx.x + k * THREADS;
    if (i < nvec) {
      float g[8];
#pragma unroll
      for (int j = 0; j < 8; j++) g[j] = (x[k][j] * inv_se - (i * 8 + j == tgt ? 1.f : 0.f)) * inv_rows;
      uint4 q;
      __nv_bfloat162 h;
      h = __floats2bfloat162_rn(g[0], g[1]); q.x = *reinterpret_cast<uint32_t*>(&h);
      h = __floats2bfloat162_rn(g[2], g[3]); q.y = *reinterpret_cast<uint32_t*>(&h);
      h = __floats2bfloat162_rn(g[4], g[5]); q.z = *reinterpret_cast<uint32_t*>(&h);
      h = __floats2bfloat162_rn(g[6], g[7]); q.w = *reinterpret_cast<uint32_t*>(&h);
      p[i] = q;
    }
  }
  if ((tgt >> 3) % THREADS == threadIdx.x) rowloss[row] = lse - lt;   // the thread that holds the target logit
}

// Long rows (vocabularies beyond 16 Ki): the row is kept PACKED (bf16 pairs) in registers so
// that two 512-thread CTAs fit on an SM and their load / reduce / store phases overlap; the
// exponentials of the first pass overwrite the logits in place (as bf16) and the second pass only
// scales them, so each element costs one exp.
template <int THREADS, int VPT>
__global__ void __launch_bounds__(THREADS, 2) softmax_ce_packed_kernel(bf16_t* __restrict__ logits,
                                                                       const int32_t* ids, int T_,
                                                                       float* __restrict__ rowloss, int V,
                                                                       float inv_rows) {
  pdl_wait();
  __shared__ float sm[THREADS / 32];
  const int row = blockIdx.x, nvec = V >> 3;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint4* p = reinterpret_cast<uint4*>(logits + (long long)row * V);
  const int tgt = ids[(long long)(row / T_) * (T_ + 1) + (row % T_) + 1];
  const float L2E = 1.4426950408889634f;
  uint32_t w[VPT][4];
  float mx = -INFINITY, lt = 0.f;
#pragma unroll
  for (int k = 0; k < VPT; k++) {
    const int i = threadIdx.x + k * THREADS;
    if (i < nvec) {
      const uint4 q = p[i];
      w[k][0] = q.x; w[k][1] = q.y; w[k][2] = q.z; w[k][3] = q.w;
#pragma unroll
      for (int j = 0; j < 4; j++) {
        const float lo = __uint_as_float(w[k][j] << 16), hi = __uint_as_float(w[k][j] & 0xffff0000u);
        mx = fmaxf(mx, fmaxf(lo, hi));
        if (i * 8 + 2 * j == tgt) lt = lo;
        if (i * 8 + 2 * j + 1 == tgt) lt = hi;
      }
    } else {
#pragma unroll
      for (int j = 0; j < 4; j++) w[k][j] = 0xff80ff80u;   // two bf16 -inf
    }
  }
  auto block_reduce = [&](float v, bool is_max) {
    v = is_max ? warp_max(v) : warp_sum(v);
    __syncthreads();
    if (lane == 0) sm[warp] = v;
    __syncthreads();
    float r = sm[0];
    for (int i = 1; i < THREADS / 32; i++) r = is_max ? fmaxf(r, sm[i]) : r + sm[i];
    return r;
  };
  mx = block_reduce(mx, true);
  float se = 0.f;
#pragma unroll
  for (int k = 0; k < VPT; k++)
#pragma unroll
    for (int j = 0; j < 4; j++) {
      const float lo = exp2f((__uint_as_float(w[k][j] << 16) - mx) * L2E);
      const float hi = exp2f((__uint_as_float(w[k][j] & 0xffff0000u) - mx) * L2E);
      se += lo + hi;                                       // the sum uses the unrounded exponentials
      __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
      w[k][j] = *reinterpret_cast<uint32_t*>(&h);
    }
  se = block_reduce(se, false);
  const float lse = mx + logf(se);
  const float scale = inv_rows / se;
#pragma unroll
  for (int k = 0; k < VPT; k++) {
    const int i = threadIdx.x + k * THREADS;
    if (i < nvec) {
      uint32_t o[4];
#pragma unroll
      for (int j = 0; j < 4; j++) {
        float lo = __uint_as_float(w[k][j] << 16) * scale, hi = __uint_as_float(w[k][j] & 0xffff0000u) * scale;
        if (i * 8 + 2 * j == tgt) lo -= inv_rows;
        if (i * 8 + 2 * j + 1 == tgt) hi -= inv_rows;
        __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
        o[j] = *reinterpret_cast<uint32_t*>(&h);
      }
      p[i] = make_uint4(o[0], o[1], o[2], o[3]);
    }
  }
  if ((tgt >> 3) % THREADS == threadIdx.x) rowloss[row] = lse - lt;
}

// Persistent variant that also produces the head's bias gradient.  A CTA walks over rows
// blockIdx.x, blockIdx.x + gridDim.x, ...; the next row streams into a shared-memory buffer
// (cp.async) while the current one, held packed in registers, goes through max / exp-sum / scale,
// so the memory system stays busy through the reductions; every thread adds the gradients it
// writes (unrounded, fp32) to column sums it alone owns in shared memory, and the CTA leaves one
// row of partial sums per CTA: colpart[gridDim.x][V].  Their ordered sum over the CTAs is the bias
// gradient -- without reading the rows x V gradient matrix a second time.
// Dynamic shared memory: V*2 bytes (row buffer) + V*4 bytes (column sums).
template <int THREADS, int VPT>
__global__ void __launch_bounds__(THREADS) softmax_ce_fused_kernel(bf16_t* __restrict__ logits,
                                                                    const int32_t* ids, int T_,
                                                                    float* __restrict__ rowloss, float* __restrict__ colpart,
                                                                    int rows, int V, float inv_rows) {
  pdl_wait();
  extern __shared__ __align__(16) uint8_t dyn[];
  __shared__ float sm[THREADS / 32];
  uint4* buf = reinterpret_cast<uint4*>(dyn);
  float* acc = reinterpret_cast<float*>(dyn + (size_t)V * 2);
  const int nvec = V >> 3;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const float L2E = 1.4426950408889634f;
  for (int i = threadIdx.x; i < V; i += THREADS) acc[i] = 0.f;
  auto fetch = [&](int row) {
    const uint4* src = reinterpret_cast<const uint4*>(logits + (long long)row * V);
#pragma unroll
    for (int k = 0; k < VPT; k++) {
      const int i = threadIdx.x + k * THREADS;
      if (i < nvec)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(buf + i)), "l"(src + i) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  auto block_reduce = [&](float v, bool is_max) {
    v = is_max ? warp_max(v) : warp_sum(v);
    __syncthreads();
    if (lane == 0) sm[warp] = v;
    __syncthreads();
    float r = sm[0];
    for (int i = 1; i < THREADS / 32; i++) r = is_max ? fmaxf(r, sm[i]) : r + sm[i];
    return r;
  };
  int row = blockIdx.x;
  if (row < rows) fetch(row);
  for (; row < rows; row += gridDim.x) {
    uint4* p = reinterpret_cast<uint4*>(logits + (long long)row * V);
    const int tgt = ids[(long long)(row / T_) * (T_ + 1) + (row % T_) + 1];
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    uint32_t w[VPT][4];
    float mx = -INFINITY, lt = 0.f;
#pragma unroll
    for (int k = 0; k < VPT; k++) {
      const int i = threadIdx.x + k * THREADS;
      if (i < nvec) {
        const uint4 q = buf[i];
        w[k][0] = q.x; w[k][1] = q.y; w[k][2] = q.z; w[k][3] = q.w;
#pragma unroll
        for (int j = 0; j < 4; j++) {
          const float lo = __uint_as_float(w[k][j] << 16), hi = __uint_as_float(w[k][j] & 0xffff0000u);
          mx = fmaxf(mx, fmaxf(lo, hi));
          if (i * 8 + 2 * j == tgt) lt = lo;
          if (i * 8 + 2 * j + 1 == tgt) lt = hi;
        }
      } else {
#pragma unroll
        for (int j = 0; j < 4; j++) w[k][j] = 0xff80ff80u;   // two bf16 -inf
      }
    }
    mx = block_reduce(mx, true);                 // its first barrier also says: every thread has read buf
    if (row + (int)gridDim.x < rows) fetch(row + gridDim.x);
    float se = 0.f;
#pragma unroll
    for (int k = 0; k < VPT; k++)
#pragma unroll
      for (int j = 0; j < 4; j++) {
        const float lo = exp2f((__uint_as_float(w[k][j] << 16) - mx) * L2E);
        const float hi = exp2f((__uint_as_float(w[k][j] & 0xffff0000u) - mx) * L2E);
        se += lo + hi;                                       // the sum uses the unrounded exponentials
        __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
        w[k][j] = *reinterpret_cast<uint32_t*>(&h);
      }
    se = block_reduce(se, false);
    const float lse = mx + logf(se);
    const float scale = inv_rows / se;
#pragma unroll
    for (int k = 0; k < VPT; k++) {
      const int i = threadIdx.x + k * THREADS;
      if (i < nvec) {
        uint32_t o[4];
        float g[8];
#pragma unroll
        for (int j = 0; j < 4; j++) {
          float lo = __uint_as_float(w[k][j] << 16) * scale, hi = __uint_as_float(w[k][j] & 0xffff0000u) * scale;
          if (i * 8 + 2 * j == tgt) lo -= inv_rows;
          if (i * 8 + 2 * j + 1 == tgt) hi -= inv_rows;
          g[2 * j] = lo; g[2 * j + 1] = hi;
          __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
          o[j] = *reinterpret_cast<uint32_t*>(&h);
        }
        p[i] = make_uint4(o[0], o[1], o[2], o[3]);
        float4* a4 = reinterpret_cast<float4*>(acc + i * 8);   // columns i*8 .. i*8+7 belong to this thread alone
        float4 a0 = a4[0], a1 = a4[1];
        a0.x += g[0]; a0.y += g[1]; a0.z += g[2]; a0.w += g[3];
        a1.x += g[4]; a1.y += g[5]; a1.z += g[6]; a1.w += g[7];
        a4[0] = a0; a4[1] = a1;
      }
    }
    if ((tgt >> 3) % THREADS == threadIdx.x) rowloss[row] = lse - lt;
  }
  // this CTA's column sums (zeros if it had no row)
  float4* dst = reinterpret_cast<float4*>(colpart + (long long)blockIdx.x * V);
#pragma unroll
  for (int k = 0; k < VPT; k++) {
    const int i = threadIdx.x + k * THREADS;
    if (i < nvec) {
      const float4* a4 = reinterpret_cast<const float4*>(acc + i * 8);
      dst[2 * i] = a4[0];
      dst[2 * i + 1] = a4[1];
    }
  }
}

int softmax_ce_fused_ctas(int rows) { return rows < 296 ? rows : 296; }

bool softmax_ce_fused_supported(int V, bool bf16, const void* logits) {
  return bf16 && V % 8 == 0 && V / 8 <= 512 * 16 && (size_t)V * 6 <= 200 * 1024 && (reinterpret_cast<uintptr_t>(logits) & 15) == 0;
}

template <int THREADS, int VPT>
static cudaError_t softmax_ce_fused_launch(bf16_t* lg, const int32_t* ids, int T_, float* rowloss, float* colpart, int rows, int V,
                                           float inv_rows, cudaStream_t s) {
  const size_t smem = (size_t)V * 6;
  static size_t attr = 0;
  if (smem > 40 * 1024 && smem > attr) {   // dynamic + static shared memory beyond the 48 KB default
    cudaError_t e = cudaFuncSetAttribute(softmax_ce_fused_kernel<THREADS, VPT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    attr = smem;
  }
  pdl_launch(softmax_ce_fused_kernel<THREADS, VPT>, softmax_ce_fused_ctas(rows), THREADS, smem, s, lg, ids, T_, rowloss, colpart, rows, V, inv_rows);
  return cudaGetLastError();
}

cudaError_t softmax_ce_fused(void* logits, const int32_t* ids, int T_, float* rowloss, float* colpart, int rows, int V,
                             float inv_rows, cudaStream_t s) {
  const int nvec = V / 8;
  bf16_t* lg = (bf16_t*)logits;
  if (nvec <= 256 * 2) return softmax_ce_fused_launch<256, 2>(lg, ids, T_, rowloss, colpart, rows, V, inv_rows, s);
  if (nvec <= 256 * 4) return softmax_ce_fused_launch<256, 4>(lg, ids, T_, rowloss, colpart, rows, V, inv_rows, s);
  if (nvec <= 512 * 4) return softmax_ce_fused_launch<512, 4>(lg, ids, T_, rowloss, colpart, rows, V, inv_rows, s);
  if (nvec <= 512 * 8) return softmax_ce_fused_launch<512, 8>(lg, ids, T_, rowloss, colpart, rows, V, inv_rows, s);
  return softmax_ce_fused_launch<512, 16>(lg, ids, T_, rowloss, colpart, rows, V, inv_rows, s);
}

cudaError_t softmax_ce_inplace(void* logits, const int32_t* ids, int T_, float* rowloss, int rows, int V,
                               float inv_rows, bool bf16, cudaStream_t s) {
  if (bf16 && V % 8 == 0 && (reinterpret_cast<uintptr_t>(logits) & 15) == 0) {
    const int nvec = V / 8;
    bf16_t* lg = (bf16_t*)logits;
    if (nvec <= 256 * 2) { pdl_launch(softmax_ce_reg_kernel<256, 2>, rows, 256, 0, s, lg, ids, T_, rowloss, V, inv_rows); return cudaGetLastError(); }
    if (nvec <= 256 * 4) { pdl_launch(softmax_ce_reg_kernel<256, 4>, rows, 256, 0, s, lg, ids, T_, rowloss, V, inv_rows); return cudaGetLastError(); }
    if (nvec <= 512 * 4) { pdl_launch(softmax_ce_packed_kernel<512, 4>, rows, 512, 0, s, lg, ids, T_, rowloss, V, inv_rows); return cudaGetLastError(); }
    if (nvec <= 512 * 8) { pdl_launch(softmax_ce_packed_kernel<512, 8>, rows, 512, 0, s, lg, ids, T_, rowloss, V, inv_rows); return cudaGetLastError(); }
    if (nvec <= 512 * 16) { pdl_launch(softmax_ce_packed_kernel<512, 16>, rows, 512, 0, s, lg, ids, T_, rowloss, V, inv_rows); return cudaGetLastError(); }
  }
  if (bf16) pdl_launch(softmax_ce_kernel<bf16_t>, rows, 256, 0, s, (bf16_t*)logits, ids, T_, rowloss, V, inv_rows);
  else pdl_launch(softmax_ce_kernel<float>, rows, 256, 0, s, (float*)logits, ids, T_, rowloss, V, inv_rows);
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------
// Softmax cross-entropy head without a pass over the logits (bf16 models, tensor-core head GEMM).
//
// With a per-row reference c_n known BEFORE the head GEMM, the GEMM's epilogue stores
// P[n,v] = exp(l[n,v] - c_n) (bf16) instead of the logit and leaves fp32 partial sums of the
// unrounded exponentials.  Then, with S_n = sum_v exp(l[n,v] - c_n):
//     lse_n = c_n + log S_n,      loss_n = lse_n - l[n,t_n],
//     dl[n,v] = (softmax - onehot)/N = r_n * (P[n,v] - S_n [v = t_n]),     r_n = 1 / (S_n N).
// The finalize kernel therefore patches ONE element per row, P[n,t_n] <- P[n,t_n] - S_n, and from
// then on the gradient of the logits is r (.) P: the backward GEMMs consume P directly,
//     dW_h = P^T (r (.) z),     dz_n = r_n (P W_h)_n,     db_h = sum_n r_n P[n,:].
// c_n is the target's own logit (z_n . W_h[t_n] + b_h[t_n], a gather and a dot product): it is at
// most the row maximum, and it is far enough below it to endanger the exponent range only when the
// token's loss exceeds ~69 nats.  Such rows (S_n >= 1e30 or not finite) are recomputed exactly by the finalize
// kernel, with c_n = the true row maximum.
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ float dot8_bf16(uint4 a, uint4 b) {
  const uint32_t x[4] = {a.x, a.y, a.z, a.w}, y[4] = {b.x, b.y, b.z, b.w};
  float acc = 0.f;
#pragma unroll
  for (int j = 0; j < 4; j++) {
    acc = fmaf(__uint_as_float(x[j] << 16), __uint_as_float(y[j] << 16), acc);
    acc = fmaf(__uint_as_float(x[j] & 0xffff0000u), __uint_as_float(y[j] & 0xffff0000u), acc);
  }
  return acc;
}

// One warp per row: tgt[n] (clamped into the vocabulary; a bad id was already reported by the
// input staging), ref[n] = lt[n] = z_n . W[t_n] + b[t_n].  d % 8 == 0.
__global__ void __launch_bounds__(256) ce_target_logit_kernel(const bf16_t* z, const bf16_t* W,
                                                              const float* bias, const int32_t* ids,
                                                              int T_, int rows, int d, int V, int* __restrict__ tgt,
                                                              float* __restrict__ ref, float* __restrict__ lt) {
  pdl_wait();
  const int lane = threadIdx.x & 31;
  for (int n = blockIdx.x * 8 + (threadIdx.x >> 5); n < rows; n += gridDim.x * 8) {
    const int t = min(max(ids[(long long)(n / T_) * (T_ + 1) + (n % T_) + 1], 0), V - 1);
    const uint4* zr = reinterpret_cast<const uint4*>(z + (long long)n * d);
    const uint4* wr = reinterpret_cast<const uint4*>(W + (long long)t * d);
    float acc = 0.f;
    for (int i = lane; i < (d >> 3); i += 32) acc += dot8_bf16(zr[i], wr[i]);
    acc = warp_sum(acc);
    if (lane == 0) {
      const float l = acc + bias[t];
      tgt[n] = t;
      ref[n] = l;
      lt[n] = l;
    }
  }
}

__device__ __forceinline__ void scale_row_bf16(const bf16_t* z, bf16_t* __restrict__ zs, int d, float r, int lane) {
  const uint4* src = reinterpret_cast<const uint4*>(z);
  uint4* dst = reinterpret_cast<uint4*>(zs);
  for (int i = lane; i < (d >> 3); i += 32) {
    const uint4 q = src[i];
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
    uint32_t o[4];
#pragma unroll
    for (int j = 0; j < 4; j++) {
      __nv_bfloat162 h = __floats2bfloat162_rn(__uint_as_float(w[j] << 16) * r, __uint_as_float(w[j] & 0xffff0000u) * r);
      o[j] = *reinterpret_cast<uint32_t*>(&h);
    }
    dst[i] = make_uint4(o[0], o[1], o[2], o[3]);
  }
}

// The 16 columns behind a scaled row of d (its stride may be larger, nothing reads further): the row scale as a sum of three bf16 values (all 24 bits of
// it), then zeros.  The weight-gradient GEMM multiplies P^T with them too, and the first three products add up to the
// head's bias gradient sum_n r_n P[n,:].  (With the leading part alone, 804 rows x 5008 logits: bias gradient 2.3e-3 off
// the float64 one, where the separate column sum with the fp32 scale gives 1.7e-3.)
__device__ __forceinline__ void scale_row_tail(bf16_t* __restrict__ zs_row, int d, int ldzs, float r, int lane) {
  if (ldzs >= d + 16 && lane < 2) {
    uint32_t part[3];
#pragma unroll
    for (int k = 0; k < 3; k++) {
      const __nv_bfloat16 b = __float2bfloat16_rn(r);
      part[k] = lane == 0 ? (uint32_t)(*reinterpret_cast<const unsigned short*>(&b)) : 0u;
      r -= __bfloat162float(b);
    }
    reinterpret_cast<uint4*>(zs_row + d)[lane] = make_uint4(part[0] | part[1] << 16, part[2], 0u, 0u);
  }
}

// The row's patched element P[n,t_n] = e_t - S is by far its largest and rounded to bf16 like the others.  The row scale
// takes that rounding up, so that their product, the gradient's one-hot part, stays exact and the rounding goes to the
// other elements, which share the same sum (their random roundings are as large).  804 rows x 5008 logits, bias gradient
// 1.7e-3 off the float64 one without it.
__device__ __forceinline__ float target_scale(float r, float t, bf16_t stored) {
  const float s = __bfloat162float(stored);
  return s != 0.f ? r * (t / s) : r;
}

// A row whose sum left the safe range, by the whole CTA: the logits are recomputed from z_n and the head's operands (twice:
// maximum, then exponentials), P[n,:] is rewritten relative to the true maximum, and loss_n, r_n and the scaled copy of z_n
// follow.
__device__ __noinline__ void ce_fixup_row(int n, float* red, const int* tgt, const bf16_t* z, const bf16_t* W, const float* bias,
                                          bf16_t* __restrict__ P, int ldp, float* __restrict__ ref, const float* lt, bf16_t* __restrict__ zs,
                                          float* __restrict__ rowloss, float* __restrict__ rowscale, int d, int ldzs, int V, float inv_rows) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint4* zr = reinterpret_cast<const uint4*>(z + (long long)n * d);
  auto logit = [&](int v) {
    const uint4* wr = reinterpret_cast<const uint4*>(W + (long long)v * d);
    float acc = 0.f;
    for (int k = lane; k < (d >> 3); k += 32) acc += dot8_bf16(zr[k], wr[k]);
    return warp_sum(acc) + bias[v];
  };
  float mx = -INFINITY;
  for (int v = warp; v < V; v += 8) mx = fmaxf(mx, logit(v));
  __syncthreads();
  if (lane == 0) red[warp] = mx;
  __syncthreads();
  mx = red[0];
#pragma unroll
  for (int w = 1; w < 8; w++) mx = fmaxf(mx, red[w]);
  float S = 0.f;
  for (int v = warp; v < V; v += 8) {
    const float e = expf(logit(v) - mx);
    S += e;
    if (lane == 0) P[(long long)n * ldp + v] = __float2bfloat16_rn(e);
  }
  __syncthreads();
  if (lane == 0) red[warp] = S;
  __syncthreads();
  S = red[0];
#pragma unroll
  for (int w = 1; w < 8; w++) S += red[w];
  const float t = expf(lt[n] - mx) - S;
  const bf16_t tb = __float2bfloat16_rn(t);
  const float r = target_scale(inv_rows / S, t, tb);
  if (threadIdx.x == 0) {      // (the barrier above ordered every warp's writes of P before this patch)
    ref[n] = mx;
    rowloss[n] = mx + logf(S) - lt[n];
    rowscale[n] = r;
    P[(long long)n * ldp + tgt[n]] = tb;
  }
  if (warp == 0) {
    scale_row_bf16(z + (long long)n * d, zs + (long long)n * ldzs, d, r, lane);
    scale_row_tail(zs + (long long)n * ldzs, d, ldzs, r, lane);
  }
  __syncthreads();
}

// One warp per row: S_n from the GEMM's partial sums (lanes stride over the groups, then a fixed
// shuffle tree), loss_n, r_n, the patch P[n,t_n] -= S_n, the scaled copy r_n z_n for the
// weight-gradient GEMM; then the CTA recomputes those of its rows whose sum left the safe range, normally none.  (By a
// launch of its own behind this one: 2 us and a launch gap in every block's backward, and 32 CTAs for any number of rows.)
__global__ void __launch_bounds__(256) ce_finalize_kernel(const float* psum, int groups, const int* status, float* __restrict__ ref,
                                                          const float* lt, const int* tgt,
                                                          bf16_t* __restrict__ P, int ldp, const bf16_t* z, const bf16_t* W, const float* bias,
                                                          bf16_t* __restrict__ zs, float* __restrict__ rowloss,
                                                          float* __restrict__ rowscale, int rows, int d,
                                                          int ldzs, int V, float inv_rows) {
  pdl_wait();
  __shared__ float red[8];
  __shared__ int unsafe[8], dead;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int n0 = blockIdx.x * 8; n0 < rows; n0 += gridDim.x * 8) {
    const int n = n0 + warp;
    bool ok = true;
    if (n < rows) {
      const float* ps = psum + (long long)n * groups;
      float S = 0.f;
      for (int g = lane; g < groups; g += 32) S += ps[g];
      S = warp_sum(S);
      ok = S < 1e30f && S > 0.f;      // false for inf and NaN too
      const float t = expf(lt[n] - ref[n]) - S;       // the one-hot part of the gradient
      const bf16_t tb = __float2bfloat16_rn(t);
      const float r = ok ? target_scale(inv_rows / S, t, tb) : 0.f;
      if (lane == 0) {
        rowloss[n] = ok ? ref[n] + logf(S) - lt[n] : 0.f;
        rowscale[n] = r;
        if (ok) P[(long long)n * ldp + tgt[n]] = tb;
      }
      scale_row_bf16(z + (long long)n * d, zs + (long long)n * ldzs, d, r, lane);
      scale_row_tail(zs + (long long)n * ldzs, d, ldzs, r, lane);
    }
    if (!__syncthreads_or(!ok)) continue;
    if (lane == 0) unsafe[warp] = ok ? 0 : 1;
    if (threadIdx.x == 0) dead = status && *status != 0;      // the step is already void (an expired wait, a bad id): its sums mean nothing
    __syncthreads();
    if (dead) return;
    for (int w = 0; w < 8; w++)
      if (unsafe[w]) ce_fixup_row(n0 + w, red, tgt, z, W, bias, P, ldp, ref, lt, zs, rowloss, rowscale, d, ldzs, V, inv_rows);
    __syncthreads();
  }
}

// dz[n,c] = r_n * sum_s part[s][n,c]   (partials of P W_h in split order; rounded to bf16 once)
__global__ void __launch_bounds__(256) ce_dz_finish_kernel(const float4* part, int splits, long long mn4, int d4,
                                                           const float* rowscale, bf16_t* __restrict__ dz) {
  pdl_wait();
  const long long i = (long long)blockIdx.x * 256 + threadIdx.x;
  if (i >= mn4) return;
  const int n = (int)(i / d4);
  float4 a = part[i];
  for (int s = 1; s < splits; s++) {
    const float4 b = part[(long long)s * mn4 + i];
    a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w;
  }
  const float r = rowscale[n];
  store4(dz + i * 4, make_float4(a.x * r, a.y * r, a.z * r, a.w * r));
}

cudaError_t ce_target_logit(const void* z, const void* W, const float* bias, const int32_t* ids, int T_, int rows, int d, int V,
                            int* tgt, float* ref, float* lt, cudaStream_t s) {
  const int grid = (int)std::min<long long>(cdiv(rows, 8), 148 * 8);
  pdl_launch(ce_target_logit_kernel, grid, 256, 0, s, (const bf16_t*)z, (const bf16_t*)W, bias, ids, T_, rows, d, V, tgt, ref, lt);
  return cudaGetLastError();
}
cudaError_t ce_finalize(const float* psum, int groups, const int* status, float* ref, const float* lt, const int* tgt, void* P, int ldp, const void* z,
                        const void* W, const float* bias, void* zs, int ldzs, float* rowloss, float* rowscale, int rows, int d, int V,
                        float inv_rows, cudaStream_t s) {
  const int grid = (int)std::min<long long>(cdiv(rows, 8), 148 * 8);
  pdl_launch(ce_finalize_kernel, grid, 256, 0, s, psum, groups, status, ref, lt, tgt, (bf16_t*)P, ldp, (const bf16_t*)z, (const bf16_t*)W, bias,
             (bf16_t*)zs, rowloss, rowscale, rows, d, ldzs, V, inv_rows);
  return cudaGetLastError();
}
cudaError_t ce_dz_finish(const float* part, int splits, int rows, int d, const float* rowscale, void* dz, cudaStream_t s) {
  const long long mn4 = (long long)rows * d / 4;
  pdl_launch(ce_dz_finish_kernel, cdiv(mn4, 256), 256, 0, s, (const float4*)part, splits, mn4, d / 4, rowscale, (bf16_t*)dz);
  return cudaGetLastError();
}

// BCE head, forward and backward in one pass over z: s = z.w + b, row loss, ds = (sigmoid(s) - y)/rows,
// dz = ds w (times act'(src) when the block ends in an activation) and this CTA's partial sums of the
// parameter gradients.  A CTA takes R <= BCE_ROWS rows: its warps first form the dot products (four rows of a
// warp side by side, so the loads of four rows are in flight), then walk over strips of 32*VEC columns, each
// warp every 8th row, re-reading the rows out of L1/L2.  Nothing in a step reads the loss or the parameter
// gradients before the optimizer, so only their partials are left here, one row per CTA; the block's batched
// reduction adds them in a fixed order.
// Bound by one read of z and one write of dz (and launch latency on small matrices).  It stands for a forward
// pass, a one-CTA loss sum, a dz pass and three column reductions that re-read z.  Between events (each adds about
// 4.5 us): 32768 x 1024 took 26 + 9 + 43 + 75 us, now 62 + 15; 4096 x 512 took 8.6 + 7 + 8.6 + 26, now 10.5 + 12.7.
// (Rows in registers, below, where they fit.)
constexpr int BCE_ROWS = 32;
// The first CTAs of the launch: partial sums of v = W^T w, the chain's share that depends on parameters only (they need
// nothing of z and run beside the head's CTAs; as a launch of its own it would stand in the chain).
template <typename T>
__device__ __forceinline__ void bce_chain_body(const BceChain& q, const float* w, int d, float* smem) {
  const int per = (d + q.chunks - 1) / q.chunks, chunk = (int)blockIdx.x / q.strips, beg = chunk * per;
  const T* W = (const T*)q.W + (long long)beg * q.hidden;
  colsum_body<T>(W, q.hidden, min(per, d - beg), q.hidden, w + beg, nullptr, q.v + (long long)chunk * q.hidden, 1, ACT_NONE, nullptr, nullptr,
                 (int)blockIdx.x % q.strips, 0, smem);
}
template <typename T, bool ALIGNED>
__global__ void __launch_bounds__(256) bce_head_kernel(const T* z, const float* w, const float* b,
                                                       const float* y, T* __restrict__ dz, int dact,
                                                       const T* src, float* __restrict__ pw, float* __restrict__ pb,
                                                       float* __restrict__ pds, float* __restrict__ ploss, int rows, int d, long long ldz, long long lddz,
                                                       int R, float inv_rows, BceChain chain) {
  pdl_wait();
  constexpr int VEC = VecOf<T>::N, SW = 32 * VEC;
  __shared__ float s_ds[BCE_ROWS], s_loss[BCE_ROWS];
  __shared__ float sm[2][8][SW];
  if ((int)blockIdx.x < chain.ctas) { bce_chain_body<T>(chain, w, d, &sm[0][0][0]); return; }
  const int part = (int)blockIdx.x - chain.ctas;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r0 = part * R, nr = min(R, rows - r0);
  for (int q0 = warp * 4; q0 < nr; q0 += 32) {
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    for (int c = lane * VEC; c < d; c += SW) {
      float wv[VEC], v[4][VEC];
#pragma unroll
      for (int k = 0; k < 4; k++)
        if (q0 + k < nr) ld_vec_n<T, ALIGNED>(z + (long long)(r0 + q0 + k) * ldz + c, d - c, v[k]);
#pragma unroll
      for (int j = 0; j < VEC; j++) wv[j] = ALIGNED || c + j < d ? w[c + j] : 0.f;
#pragma unroll
      for (int k = 0; k < 4; k++)
        if (q0 + k < nr) {
#pragma unroll
          for (int j = 0; j < VEC; j++) acc[k] = fmaf(v[k][j], wv[j], acc[k]);
        }
    }
#pragma unroll
    for (int k = 0; k < 4; k++) acc[k] = warp_sum(acc[k]);
    if (lane < 4 && q0 + lane < nr) {
      const float sv = (lane == 0 ? acc[0] : lane == 1 ? acc[1] : lane == 2 ? acc[2] : acc[3]) + b[0];
      const float yy = y[r0 + q0 + lane];
      const float e = expf(-fabsf(sv));
      s_loss[q0 + lane] = (fmaxf(sv, 0.f) - sv * yy + log1pf(e)) * inv_rows;
      const float sig = sv >= 0.f ? 1.f / (1.f + e) : e / (1.f + e);
      s_ds[q0 + lane] = (sig - yy) * inv_rows;
      if (chain.ds) chain.ds[r0 + q0 + lane] = s_ds[q0 + lane];
    }
  }
  __syncthreads();
  if (warp == 0) {
    const float l = warp_sum(lane < nr ? s_loss[lane] : 0.f), g = warp_sum(lane < nr ? s_ds[lane] : 0.f);
    if (lane == 0) { ploss[part] = l; pds[part] = g; }
  }
  for (int c0 = 0; c0 < d; c0 += SW) {
    const int c = c0 + lane * VEC;
    float aw[VEC], ab[VEC];
#pragma unroll
    for (int j = 0; j < VEC; j++) aw[j] = ab[j] = 0.f;
    if (c < d) {
      float wv[VEC];
#pragma unroll
      for (int j = 0; j < VEC; j++) wv[j] = ALIGNED || c + j < d ? w[c + j] : 0.f;
      for (int r = warp; r < nr; r += 32) {        // four rows' loads in flight, then their sums and stores
        float v[4][VEC], u[4][VEC];
#pragma unroll
        for (int k = 0; k < 4; k++)
          if (r + 8 * k < nr) {
            const long long at = (long long)(r0 + r + 8 * k) * ldz + c;
            ld_vec_n<T, ALIGNED>(z + at, d - c, v[k]);
            if (dact != ACT_NONE) ld_vec_n<T, ALIGNED>(src + at, d - c, u[k]);
          }
#pragma unroll
        for (int k = 0; k < 4; k++)
          if (r + 8 * k < nr) {
            const float dsr = s_ds[r + 8 * k];
            float o[VEC];
#pragma unroll
            for (int j = 0; j < VEC; j++) { aw[j] = fmaf(v[k][j], dsr, aw[j]); o[j] = dsr * wv[j]; }
            if (dact != ACT_NONE) {
#pragma unroll
              for (int j = 0; j < VEC; j++) {
                const float g = act_deriv(dact, u[k][j]);
                ab[j] = fmaf(g, dsr, ab[j]);
                o[j] *= g;
              }
            }
            if (dz) st_vec_n<T, ALIGNED>(dz + (long long)(r0 + r + 8 * k) * lddz + c, d - c, o);
            if (chain.prod) {
              const long long at = (long long)(r0 + r + 8 * k) * ldz + c;
              ld_vec_n<T, ALIGNED>((const T*)chain.mul + at, d - c, u[k]);
#pragma unroll
              for (int j = 0; j < VEC; j++) o[j] *= u[k][j];
              st_vec_n<T, ALIGNED>((T*)chain.prod + at, d - c, o);
            }
          }
      }
    }
#pragma unroll
    for (int j = 0; j < VEC; j++) sm[0][warp][lane * VEC + j] = aw[j];
    if (pb) {
#pragma unroll
      for (int j = 0; j < VEC; j++) sm[1][warp][lane * VEC + j] = ab[j];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < SW; i += 256) {
      if (c0 + i < d) {
        float t = 0.f;
#pragma unroll
        for (int k = 0; k < 8; k++) t += sm[0][k][i];
        pw[(long long)part * d + c0 + i] = t;
        if (pb) {
          t = 0.f;
#pragma unroll
          for (int k = 0; k < 8; k++) t += sm[1][k][i];
          pb[(long long)part * d + c0 + i] = t;
        }
      }
    }
    __syncthreads();
  }
}

// The same for bf16 rows of up to 2048 columns (16-byte aligned): a warp keeps its RW rows in registers (NV 16-byte
// pieces per lane and row) from the dot products to dz and the partial sums, so z is read once, all of a warp's loads are
// in flight together, and the CTA meets once per 256 columns.  Between events: 4096 x 512 10.6 -> 8.4 us (MLP step
// 832 -> 813), 32768 x 1024 65 -> 52, 4096 x 1680 20.8 -> 16.8.
template <int NV, int RW>
__global__ void __launch_bounds__(256) bce_head_rows_kernel(const bf16_t* z, const float* w, const float* b,
                                                            const float* y, bf16_t* __restrict__ dz, int dact,
                                                            const bf16_t* src, float* __restrict__ pw, float* __restrict__ pb,
                                                            float* __restrict__ pds, float* __restrict__ ploss, int rows, int d, long long ldz, long long lddz,
                                                            float inv_rows, BceChain chain) {
  pdl_wait();
  __shared__ float s_ds[8 * RW], s_loss[8 * RW];
  __shared__ __align__(16) float sm[2][2][8][256];        // [strip parity][weight, activation bias][warp][column]
  if ((int)blockIdx.x < chain.ctas) { bce_chain_body<bf16_t>(chain, w, d, &sm[0][0][0][0]); return; }
  const int part = (int)blockIdx.x - chain.ctas;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r0 = part * 8 * RW + warp * RW;
  uint4 q[RW][NV];
#pragma unroll
  for (int k = 0; k < RW; k++)
#pragma unroll
    for (int i = 0; i < NV; i++) {
      const int c = (i * 32 + lane) * 8;
      q[k][i] = r0 + k < rows && c < d ? *reinterpret_cast<const uint4*>(z + (long long)(r0 + k) * ldz + c) : make_uint4(0u, 0u, 0u, 0u);
    }
  auto unpack = [](uint4 p, float (&v)[8]) {
    const uint32_t x[4] = {p.x, p.y, p.z, p.w};
#pragma unroll
    for (int j = 0; j < 4; j++) { v[2 * j] = __uint_as_float(x[j] << 16); v[2 * j + 1] = __uint_as_float(x[j] & 0xffff0000u); }
  };
  auto load_w = [&](int c, float (&wv)[8]) {
    const float4 a = *reinterpret_cast<const float4*>(w + c), e = *reinterpret_cast<const float4*>(w + c + 4);
    wv[0] = a.x; wv[1] = a.y; wv[2] = a.z; wv[3] = a.w; wv[4] = e.x; wv[5] = e.y; wv[6] = e.z; wv[7] = e.w;
  };
  float acc[RW];
#pragma unroll
  for (int k = 0; k < RW; k++) acc[k] = 0.f;
#pragma unroll
  for (int i = 0; i < NV; i++) {
    const int c = (i * 32 + lane) * 8;
    if (c < d) {
      float wv[8], v[8];
      load_w(c, wv);
#pragma unroll
      for (int k = 0; k < RW; k++) {
        unpack(q[k][i], v);
#pragma unroll
        for (int j = 0; j < 8; j++) acc[k] = fmaf(v[j], wv[j], acc[k]);
      }
    }
  }
  float mine = 0.f;
#pragma unroll
  for (int k = 0; k < RW; k++) {
    acc[k] = warp_sum(acc[k]);
    if (lane == k) mine = acc[k];
  }
  float ds = 0.f, loss = 0.f;
  if (lane < RW && r0 + lane < rows) {
    const float sv = mine + b[0], yy = y[r0 + lane];
    const float e = expf(-fabsf(sv));
    loss = (fmaxf(sv, 0.f) - sv * yy + log1pf(e)) * inv_rows;
    const float sig = sv >= 0.f ? 1.f / (1.f + e) : e / (1.f + e);
    ds = (sig - yy) * inv_rows;
    if (chain.ds) chain.ds[r0 + lane] = ds;
  }
  if (lane < RW) { s_ds[warp * RW + lane] = ds; s_loss[warp * RW + lane] = loss; }
  float dsr[RW];
#pragma unroll
  for (int k = 0; k < RW; k++) dsr[k] = __shfl_sync(0xffffffffu, ds, k);
#pragma unroll
  for (int i = 0; i < NV; i++) {
    const int c = (i * 32 + lane) * 8;
    float aw[8], ab[8];
#pragma unroll
    for (int j = 0; j < 8; j++) aw[j] = ab[j] = 0.f;
    if (c < d) {
      float wv[8];
      load_w(c, wv);
#pragma unroll
      for (int k = 0; k < RW; k++) {
        float v[8], o[8];
        unpack(q[k][i], v);
#pragma unroll
        for (int j = 0; j < 8; j++) { aw[j] = fmaf(v[j], dsr[k], aw[j]); o[j] = dsr[k] * wv[j]; }
        if (dz && r0 + k < rows) {
          const long long at = (long long)(r0 + k) * ldz + c;
          if (dact != ACT_NONE) {
            float u[8];
            unpack(*reinterpret_cast<const uint4*>(src + at), u);
#pragma unroll
            for (int j = 0; j < 8; j++) {
              const float g = act_deriv(dact, u[j]);
              ab[j] = fmaf(g, dsr[k], ab[j]);
              o[j] *= g;
            }
          }
          st_vec_n<bf16_t, true>(dz + (long long)(r0 + k) * lddz + c, 8, o);
          if (chain.prod) {
            float u[8];
            unpack(*reinterpret_cast<const uint4*>((const bf16_t*)chain.mul + at), u);
#pragma unroll
            for (int j = 0; j < 8; j++) o[j] *= u[j];
            st_vec_n<bf16_t, true>((bf16_t*)chain.prod + at, 8, o);
          }
        }
      }
    }
    float (*s0)[256] = sm[i & 1][0], (*s1)[256] = sm[i & 1][1];
    *reinterpret_cast<float4*>(&s0[warp][lane * 8]) = make_float4(aw[0], aw[1], aw[2], aw[3]);
    *reinterpret_cast<float4*>(&s0[warp][lane * 8 + 4]) = make_float4(aw[4], aw[5], aw[6], aw[7]);
    if (pb) {
      *reinterpret_cast<float4*>(&s1[warp][lane * 8]) = make_float4(ab[0], ab[1], ab[2], ab[3]);
      *reinterpret_cast<float4*>(&s1[warp][lane * 8 + 4]) = make_float4(ab[4], ab[5], ab[6], ab[7]);
    }
    __syncthreads();          // (two parities: a warp writes this one again only behind the next strip's barrier)
    const int col = i * 256 + threadIdx.x;
    if (col < d) {
      float t = 0.f;
#pragma unroll
      for (int k = 0; k < 8; k++) t += s0[k][threadIdx.x];
      pw[(long long)part * d + col] = t;
      if (pb) {
        t = 0.f;
#pragma unroll
        for (int k = 0; k < 8; k++) t += s1[k][threadIdx.x];
        pb[(long long)part * d + col] = t;
      }
    }
  }
  if (warp == 0) {
    const float l = warp_sum(lane < 8 * RW ? s_loss[lane] : 0.f), g = warp_sum(lane < 8 * RW ? s_ds[lane] : 0.f);
    if (lane == 0) { ploss[part] = l; pds[part] = g; }
  }
}

// Few rows per CTA spread a small matrix over the SMs, many keep the partials small beside z: 16 until there are two CTAs
// per SM, then up to BCE_ROWS.  Rows in registers: 16 up to three CTAs of them per SM (7104 rows), then 32; over 1024
// columns always 16 (two per warp).  Head with its block's reductions, 16 / 32 rows, us between events: 512 columns
// 4096 rows 19.1 / 19.7, 6500 19.8 / 20.9, 8000 21.3 / 21.0, 12000 23.2 / 21.2; 1024 columns 4096 rows 21.2 / 23.3, 6500
// and 7104 23.3 / 23.3, 8000 25.3 / 23.3; 128 columns equal from 4096 to 9472 rows, 12000 21.2 / 19.2.
static bool bce_in_registers(int d, bool bf16) { return bf16 && d % 8 == 0 && d <= 2048; }
static int bce_head_rows(int rows, int d, bool bf16) {
  if (bce_in_registers(d, bf16)) return d > 1024 || rows <= 296 * 24 ? 16 : 32;
  return std::min(BCE_ROWS, std::max(16, (rows + 295) / 296));
}
int bce_head_parts(int rows, int d, bool bf16) { return (rows + bce_head_rows(rows, d, bf16) - 1) / bce_head_rows(rows, d, bf16); }

cudaError_t bce_head(const void* z, const float* w, const float* b, const float* y, void* dz, int dact, const void* src, float* pw,
                     float* pb, float* pds, float* ploss, int rows, int d, long long ldz, long long lddz, float inv_rows, bool bf16, cudaStream_t s,
                     const BceChain* chained) {
  BceChain chain;
  if (chained) chain = *chained;
  const int R = bce_head_rows(rows, d, bf16), grid = bce_head_parts(rows, d, bf16) + chain.ctas;
  const bool al = ((reinterpret_cast<uintptr_t>(z) | reinterpret_cast<uintptr_t>(dz) | reinterpret_cast<uintptr_t>(src) |
                    reinterpret_cast<uintptr_t>(chain.mul) | reinterpret_cast<uintptr_t>(chain.prod)) & 15) == 0 &&
                  d % (bf16 ? 8 : 4) == 0 && ldz % (bf16 ? 8 : 4) == 0 && lddz % (bf16 ? 8 : 4) == 0;
  if (bce_in_registers(d, bf16) && al && (reinterpret_cast<uintptr_t>(w) & 15) == 0) {
    auto go = [&](auto kernel) {
      pdl_launch(kernel, grid, 256, 0, s, (const bf16_t*)z, w, b, y, (bf16_t*)dz, dact, (const bf16_t*)src, pw, pb, pds, ploss, rows, d, ldz, lddz, inv_rows, chain);
    };
    const int nv = (d + 255) / 256;
    if (R == 16) { if (nv <= 1) go(bce_head_rows_kernel<1, 2>); else if (nv <= 2) go(bce_head_rows_kernel<2, 2>); else if (nv <= 4) go(bce_head_rows_kernel<4, 2>); else go(bce_head_rows_kernel<8, 2>); }
    else { if (nv <= 1) go(bce_head_rows_kernel<1, 4>); else if (nv <= 2) go(bce_head_rows_kernel<2, 4>); else go(bce_head_rows_kernel<4, 4>); }
    return cudaGetLastError();
  }
  auto go = [&](auto* t, auto kernel) {
    typedef typename std::remove_pointer<decltype(t)>::type T;
    pdl_launch(kernel, grid, 256, 0, s, (const T*)z, w, b, y, (T*)dz, dact, (const T*)src, pw, pb, pds, ploss, rows, d, ldz, lddz, R, inv_rows, chain);
  };
  if (bf16) { if (al) go((bf16_t*)nullptr, bce_head_kernel<bf16_t, true>); else go((bf16_t*)nullptr, bce_head_kernel<bf16_t, false>); }
  else { if (al) go((float*)nullptr, bce_head_kernel<float, true>); else go((float*)nullptr, bce_head_kernel<float, false>); }
  return cudaGetLastError();
}

// Backward of a Linear whose output z goes into a BCE head and nowhere else.  The loss gradient is then an outer product,
// dz[n,c] = ds[n] w[c], and so is everything the Linear's backward makes of it:
//     dz W          = ds (x) v,     v = W^T w              (in the head's launch, from the parameters alone)
//     dz^T y        = w (x) t,      t[k] = sum_n ds[n] y[n,k]
// which leaves one pass over the Linear's input y = act(src) in the place of two GEMMs over [rows, hidden]: du[n,k] =
// ds[n] v[k] act'(src[n,k]), t, and where wanted db[k] = sum_n du[n,k] for the Linear before.  ds, v and t stay in fp32, where
// the GEMMs took dz rounded to bf16.  y is recomputed from the pre-activation (GELU; not rounded as the forward stored it), so
// one matrix is read and one written.
// A CTA takes a strip of 128 columns and a chunk of rows, a thread four adjacent columns and every 8th row, and leaves its
// partial sums of t and db to the block's batched reduction (added up here, by a strip's last CTA: 512 x 512 6.3 us for the
// launch, and v with the same ticket in the head's 1.5 more).  Bound by latency at small sizes, by the bytes in flight at large
// ones: 512 x 512 2.2 us, 3001 x 2136 (ReLU) 10, 4096 x 2048 14.4, 32768 x 4096 160 (3.3 TB/s); with eight columns a thread, two
// CTAs per SM and chunks that are no whole turns 4.2, 14.5, 19.3 and 155.
constexpr int CHAIN_COLS = 128;
template <typename T, bool ALIGNED, int ACT>
__global__ void __launch_bounds__(256, 3) bce_chain_bwd_kernel(const T* src, long long ld, const float* ds, const float* v, int vparts,
                                                               T* __restrict__ du, float* __restrict__ pt, float* __restrict__ pb,
                                                               int rows, int cols, int per) {
  pdl_wait();
  __shared__ __align__(16) float sm[2][8][CHAIN_COLS];
  const int cx = threadIdx.x & 31, ry = threadIdx.x >> 5;
  const int c = blockIdx.x * CHAIN_COLS + cx * 4, valid = cols - c;
  const int rb = blockIdx.y * per, re = min(rows, rb + per);
  f32x2 vv[2], at[2], ab[2];
#pragma unroll
  for (int j = 0; j < 2; j++) at[j] = ab[j] = pack_f2(0.f, 0.f);
  if (valid > 0) {
    // Rows in turns of four.  The loads of the next turn are in flight while one is worked on, and the first ones while v is
    // added up.  Rows past the end are zeros with ds = 0.
    float d[4];
    Raw4<T> raw[4];
    auto fetch = [&](int r) {
#pragma unroll
      for (int k = 0; k < 4; k++) {
        const bool ok = r + 8 * k < re;
        d[k] = ok ? ds[r + 8 * k] : 0.f;
        raw[k] = Raw4<T>();
        if (ok) ld_raw4<T, ALIGNED>(src + (long long)(r + 8 * k) * ld + c, valid, raw[k]);
      }
    };
    int r = rb + ry;
    fetch(r);
    float4 va = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int k0 = 0; k0 < vparts; k0 += 4) {          // four partials' loads in flight
      float4 p[4];
#pragma unroll
      for (int k = 0; k < 4; k++)
        p[k] = k0 + k < vparts ? ld4_guard(v + (long long)(k0 + k) * cols + c, valid, ALIGNED) : make_float4(0.f, 0.f, 0.f, 0.f);
      va.x += (p[0].x + p[1].x) + (p[2].x + p[3].x); va.y += (p[0].y + p[1].y) + (p[2].y + p[3].y);
      va.z += (p[0].z + p[1].z) + (p[2].z + p[3].z); va.w += (p[0].w + p[1].w) + (p[2].w + p[3].w);
    }
    vv[0] = pack_f2(va.x, va.y);
    vv[1] = pack_f2(va.z, va.w);
    for (; r < re; r += 32) {
      float dk[4];
      Raw4<T> now[4];
#pragma unroll
      for (int k = 0; k < 4; k++) { now[k] = raw[k]; dk[k] = d[k]; }
      if (r + 32 < re) fetch(r + 32);
#pragma unroll
      for (int k = 0; k < 4; k += 2) {       // two rows side by side
        float u[8], y[8], g[8];
        unpack_raw4(now[k], u);
        unpack_raw4(now[k + 1], u + 4);
        if (ACT == ACT_GELU) {
          act_both<T>(u, y, g);
        } else {
#pragma unroll
          for (int j = 0; j < 8; j++) { y[j] = u[j]; g[j] = act_deriv(ACT, u[j]); }
        }
#pragma unroll
        for (int h = 0; h < 2; h++) {
          const f32x2 dd = pack_f2(dk[k + h], dk[k + h]);
          float* gh = g + 4 * h;
#pragma unroll
          for (int j = 0; j < 2; j++) {
            at[j] = fma_f2(dd, pack_f2(y[4 * h + 2 * j], y[4 * h + 2 * j + 1]), at[j]);
            const f32x2 o = mul_f2(mul_f2(dd, vv[j]), pack_f2(gh[2 * j], gh[2 * j + 1]));
            ab[j] = add_f2(ab[j], o);
            unpack_f2(o, gh[2 * j], gh[2 * j + 1]);
          }
          const int row = r + 8 * (k + h);
          if (row < re) {
            T* dst = du + (long long)row * ld + c;
            if (ALIGNED) {
              store4(dst, make_float4(gh[0], gh[1], gh[2], gh[3]));
            } else {
#pragma unroll
              for (int j = 0; j < 4; j++)
                if (j < valid) stf(dst + j, gh[j]);
            }
          }
        }
      }
    }
  }
#pragma unroll
  for (int j = 0; j < 2; j++) {
    unpack_f2(at[j], sm[0][ry][cx * 4 + 2 * j], sm[0][ry][cx * 4 + 2 * j + 1]);
    unpack_f2(ab[j], sm[1][ry][cx * 4 + 2 * j], sm[1][ry][cx * 4 + 2 * j + 1]);
  }
  __syncthreads();
  const int half = threadIdx.x >> 7, col = threadIdx.x & 127, cc = blockIdx.x * CHAIN_COLS + col;     // 128 threads for t, 128 for db
  float* out = half ? pb : pt;
  if (cc < cols && out) {
    float a = 0.f;
#pragma unroll
    for (int k = 0; k < 8; k++) a += sm[half][k][col];
    out[(long long)blockIdx.y * cols + cc] = a;
  }
}

// Rows of a CTA: whole turns of 32, as many as fill the device once (three CTAs per SM); a small matrix: one turn.
static int bce_chain_rows(int rows, int cols) {
  const int strips = (int)cdiv(cols, CHAIN_COLS), chunks = std::max(1, 444 / strips);
  return std::max(1, (int)cdiv(cdiv(rows, chunks), 32)) * 32;
}
int bce_chain_chunks(int rows, int cols) { return (int)cdiv(rows, bce_chain_rows(rows, cols)); }
cudaError_t bce_chain_bwd(const void* src, int act, long long ld, const float* ds, const float* v, int vparts, void* du, float* pt, float* pb,
                          int rows, int cols, bool bf16, cudaStream_t s) {
  const bool al = cols % 4 == 0 && ld % 4 == 0 && ((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(du)) & 15) == 0;
  const dim3 grid(cdiv(cols, CHAIN_COLS), bce_chain_chunks(rows, cols));
  auto go = [&](auto* tp, auto kernel) {
    typedef typename std::remove_pointer<decltype(tp)>::type T;
    pdl_launch(kernel, grid, 256, 0, s, (const T*)src, ld, ds, v, vparts, (T*)du, pt, pb, rows, cols, bce_chain_rows(rows, cols));
  };
  auto pick = [&](auto* tp) {
    typedef typename std::remove_pointer<decltype(tp)>::type T;
    if (act == ACT_GELU) { if (al) go(tp, bce_chain_bwd_kernel<T, true, ACT_GELU>); else go(tp, bce_chain_bwd_kernel<T, false, ACT_GELU>); }
    else if (act == ACT_RELU) { if (al) go(tp, bce_chain_bwd_kernel<T, true, ACT_RELU>); else go(tp, bce_chain_bwd_kernel<T, false, ACT_RELU>); }
    else { if (al) go(tp, bce_chain_bwd_kernel<T, true, ACT_NONE>); else go(tp, bce_chain_bwd_kernel<T, false, ACT_NONE>); }
  };
  if (bf16) pick((bf16_t*)nullptr);
  else pick((float*)nullptr);
  return cudaGetLastError();
}

// Goodness head (binary cross-entropy on G = sum_j z_j^2 with the logit G + b): one warp per row,
// the same outputs as the BCE head (row losses, ds = (sigmoid(s) - y)/rows).
template <typename T>
__global__ void __launch_bounds__(256) goodness_head_fwd_kernel(const T* z, long long ldz,
                                                                const float* b, const float* y,
                                                                float* __restrict__ rowloss, float* __restrict__ ds,
                                                                int rows, int d, float inv_rows) {
  pdl_wait();
  int row = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (row >= rows) return;
  float s = 0.f;
  for (int c = lane; c < d; c += 32) {
    const float v = ldf(z + (long long)row * ldz + c);
    s = fmaf(v, v, s);
  }
  s = warp_sum(s) + b[0];
  if (lane == 0) {
    float yy = y[row];
    float e = expf(-fabsf(s));
    rowloss[row] = fmaxf(s, 0.f) - s * yy + log1pf(e);
    float sig = s >= 0.f ? 1.f / (1.f + e) : e / (1.f + e);
    ds[row] = (sig - yy) * inv_rows;
  }
}
cudaError_t goodness_head_fwd(const void* z, long long ldz, const float* b, const float* y, float* rowloss, float* ds,
                              int rows, int d, float inv_rows, bool bf16, cudaStream_t s) {
  if (bf16) pdl_launch(goodness_head_fwd_kernel<bf16_t>, cdiv(rows, 8), 256, 0, s, (const bf16_t*)z, ldz, b, y, rowloss, ds, rows, d, inv_rows);
  else pdl_launch(goodness_head_fwd_kernel<float>, cdiv(rows, 8), 256, 0, s, (const float*)z, ldz, b, y, rowloss, ds, rows, d, inv_rows);
  return cudaGetLastError();
}

// dz = 2 ds z (times act'(src) when z = act(src) closes the block)
template <typename T>
__global__ void __launch_bounds__(256) goodness_head_dz_kernel(const float* ds, const T* z,
                                                               T* __restrict__ dz, int dact, const T* src,
                                                               long long n, int d) {
  pdl_wait();
  long long i = (long long)blockIdx.x * 256 + threadIdx.x;
  if (i >= n) return;
  float v = 2.f * ds[i / d] * ldf(z + i);
  if (dact != ACT_NONE) v *= act_deriv(dact, ldf(src + i));
  stf(dz + i, v);
}
cudaError_t goodness_head_dz(const float* ds, const void* z, void* dz, int dact, const void* src, int rows,
                             int d, bool bf16, cudaStream_t s) {
  long long n = (long long)rows * d;
  if (bf16) pdl_launch(goodness_head_dz_kernel<bf16_t>, cdiv(n, 256), 256, 0, s, ds, (const bf16_t*)z, (bf16_t*)dz, dact, (const bf16_t*)src, n, d);
  else pdl_launch(goodness_head_dz_kernel<float>, cdiv(n, 256), 256, 0, s, ds, (const float*)z, (float*)dz, dact, (const float*)src, n, d);
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------
// elementwise
// ------------------------------------------------------------------------------------------
// One 16-byte vector per thread and step (8 bf16 or 4 floats); the element tail is scalar.
// mode 0: out = a * b      mode 1: out = act(a)      mode 2: out = a * act'(b)
template <typename T>
__global__ void __launch_bounds__(256) ew_kernel(const T* a, const T* b, T* out,   // a may alias out
                                                 long long n, int mode, int act) {
  pdl_wait();
  constexpr int VEC = VecOf<T>::N;
  const long long nvec = n / VEC;
  const long long stride = (long long)gridDim.x * 256;
  for (long long i = (long long)blockIdx.x * 256 + threadIdx.x; i < nvec; i += stride) {
    float x[VEC], y[VEC];
    ld_vec<T>(a + i * VEC, x);
    if (mode != 1) ld_vec<T>(b + i * VEC, y);
    if (act == ACT_GELU && mode != 0) {     // the common case, with the cheaper normal CDF for bf16 data
      if (mode == 1) gelu_vec(x);
      else dgelu_vec(y, x);
    } else {
#pragma unroll
      for (int j = 0; j < VEC; j++)
        x[j] = mode == 0 ? x[j] * y[j] : (mode == 1 ? act_apply(act, x[j]) : x[j] * act_deriv(act, y[j]));
    }
    if (VEC == 8) {
      uint4 q;
      __nv_bfloat162 h;
      h = __floats2bfloat162_rn(x[0], x[1]); q.x = *reinterpret_cast<uint32_t*>(&h);
      h = __floats2bfloat162_rn(x[2], x[3]); q.y = *reinterpret_cast<uint32_t*>(&h);
      h = __floats2bfloat162_rn(x[4 % VEC], x[5 % VEC]); q.z = *reinterpret_cast<uint32_t*>(&h);
      h = __floats2bfloat162_rn(x[6 % VEC], x[7 % VEC]); q.w = *reinterpret_cast<uint32_t*>(&h);
      *reinterpret_cast<uint4*>(out + i * VEC) = q;
    } else {
      *reinterpret_cast<float4*>(out + i * VEC) = make_float4(x[0], x[1], x[2], x[3]);
    }
  }
  if (blockIdx.x == 0)
    for (long long i = nvec * VEC + threadIdx.x; i < n; i += 256) {
      const float xa = ldf(a + i);
      stf(out + i, mode == 0 ? xa * ldf(b + i) : (mode == 1 ? act_apply(act, xa) : xa * act_deriv(act, ldf(b + i))));
    }
}

static cudaError_t ew_launch(const void* a, const void* b, void* out, long long n, int mode, int act, bool bf16, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const bool aligned = ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b) | reinterpret_cast<uintptr_t>(out)) & 15) == 0;
  if (!aligned) return cudaErrorMisalignedAddress;   // every buffer of the library is 256-byte aligned
  const long long nvec = n / (bf16 ? 8 : 4);
  long long blocks = (nvec + 255) / 256;
  if (blocks > 148 * 16) blocks = 148 * 16;
  if (blocks < 1) blocks = 1;
  if (bf16) pdl_launch(ew_kernel<bf16_t>, (unsigned)blocks, 256, 0, s, (const bf16_t*)a, (const bf16_t*)b, (bf16_t*)out, n, mode, act);
  else pdl_launch(ew_kernel<float>, (unsigned)blocks, 256, 0, s, (const float*)a, (const float*)b, (float*)out, n, mode, act);
  return cudaGetLastError();
}
cudaError_t ew_mul(const void* a, const void* b, void* out, long long n, bool bf16, cudaStream_t s) {
  return ew_launch(a, b, out, n, 0, ACT_NONE, bf16, s);
}
cudaError_t ew_act(const void* u, void* out, int act, long long n, bool bf16, cudaStream_t s) {
  return ew_launch(u, nullptr, out, n, 1, act, bf16, s);
}
cudaError_t ew_dact(void* d, const void* src, int act, long long n, bool bf16, cudaStream_t s) {
  return ew_launch(d, src, d, n, 2, act, bf16, s);
}

// ------------------------------------------------------------------------------------------
// input staging (z_0)
// ------------------------------------------------------------------------------------------
// An id outside its table is never used as an index: the row is filled from row 0 instead and the
// model's status word is set to STATUS_BAD_ID, which the next synchronisation reports as an
// invalid argument (the step's results are void).
__device__ __forceinline__ int checked_id(int id, int rows, int* status) {
  if ((unsigned)id >= (unsigned)rows) {
    if (status) atomicExch(status, STATUS_BAD_ID);
    return 0;
  }
  return id;
}


// Token + position gather, one warp per output row: the id is read once per row, a lane moves four
// consecutive columns per step (two 16-byte loads, one 8- or 16-byte store), so a warp reads 512
// contiguous bytes of the embedding row at a time.  VEC = false is the scalar form for widths that
// are not multiples of four.
// The optimizer's step counter, advanced by one more CTA of the step's first kernel (a launch of its own takes 2 us, in front
// of the forward or of the optimizer): true in that CTA, which has nothing else to do.
__device__ __forceinline__ bool step_tick_cta(const StepTick& tk) {
  if (!tk.tick || blockIdx.x != gridDim.x - 1) return false;
  if (threadIdx.x == 0) {
    const double t = tk.tick[0] + 1.0;
    tk.tick[0] = t;
    tk.tick[1] = 1.0 - pow(tk.beta1, t);
    tk.tick[2] = 1.0 - pow(tk.beta2, t);
  }
  return true;
}
__device__ __forceinline__ int work_ctas(const StepTick& tk) { return (int)gridDim.x - (tk.tick ? 1 : 0); }

// A dense batch into the model's own buffer: rows of `row` units (16, 4 or 2 bytes), `pitch` units apart in the copy.
// (Two-block MLP of 64 / 256 columns, with the step counter's launch gone too: 40 -> 37 us; 67 MB 26 us either way.)
template <typename V>
__global__ void __launch_bounds__(256) copy_rows_kernel(const V* src, V* __restrict__ dst, long long rows, long long row, long long pitch, StepTick tk) {
  pdl_wait();
  if (step_tick_cta(tk)) return;
  const long long n = rows * row, stride = (long long)work_ctas(tk) * 1024;
  for (long long i0 = (long long)blockIdx.x * 1024 + threadIdx.x; i0 < n; i0 += stride) {
    V v[4];
#pragma unroll
    for (int k = 0; k < 4; k++)
      if (i0 + k * 256 < n) v[k] = src[i0 + k * 256];
#pragma unroll
    for (int k = 0; k < 4; k++) {
      const long long i = i0 + k * 256;
      if (i < n) dst[pitch == row ? i : i / row * pitch + i % row] = v[k];
    }
  }
}
// Can a kernel read `bytes` at p as safely as a copy would?  Memory of this device, inside one allocation.
static bool own_device_range(const void* p, size_t bytes) {
  typedef CUresult (*RangeFn)(CUdeviceptr*, size_t*, CUdeviceptr);
  static const RangeFn range = []() -> RangeFn {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuMemGetAddressRange", &f, cudaEnableDefault, &q) == cudaSuccess && q == cudaDriverEntryPointSuccess) return (RangeFn)f;
    cudaGetLastError();
    return nullptr;
  }();
  cudaPointerAttributes at;
  int dev = -1;
  if (!range || cudaPointerGetAttributes(&at, p) != cudaSuccess || cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  CUdeviceptr base = 0;
  size_t size = 0;
  return at.type == cudaMemoryTypeDevice && at.device == dev && range(&base, &size, (CUdeviceptr)p) == CUDA_SUCCESS &&
         (CUdeviceptr)p - base <= size && bytes <= size - (size_t)((CUdeviceptr)p - base);
}
cudaError_t copy_rows(const void* src, void* dst, long long rows, long long row_bytes, long long pitch_bytes, const StepTick& tk, cudaStream_t s, int* launches) {
  const unsigned long long al = reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst) | (unsigned long long)row_bytes | (unsigned long long)pitch_bytes;
  auto go = [&](auto* t, auto kernel, bool copy) {
    typedef typename std::remove_pointer<decltype(t)>::type V;
    const long long unit = sizeof(V), n = copy ? rows * (row_bytes / unit) : 0;
    const unsigned grid = (unsigned)std::min<long long>((n + 1023) / 1024, 148 * 16) + (tk.tick ? 1 : 0);
    *launches = grid > 0 ? 1 : 0;
    if (grid > 0) pdl_launch(kernel, grid, 256, 0, s, (const V*)src, (V*)dst, copy ? rows : 0LL, row_bytes / unit, pitch_bytes / unit, tk);
  };
  if (!own_device_range(src, (size_t)(rows * row_bytes))) {      // pinned host memory, a peer's, or what only the copy can refuse
    const cudaError_t e = pitch_bytes == row_bytes ? cudaMemcpyAsync(dst, src, rows * row_bytes, cudaMemcpyDeviceToDevice, s)
                                                   : cudaMemcpy2DAsync(dst, pitch_bytes, src, row_bytes, row_bytes, rows, cudaMemcpyDeviceToDevice, s);
    if (e != cudaSuccess) return e;
    go((unsigned char*)nullptr, copy_rows_kernel<unsigned char>, false);
  } else if (al % 16 == 0) go((uint4*)nullptr, copy_rows_kernel<uint4>, true);
  else if (al % 4 == 0) go((uint32_t*)nullptr, copy_rows_kernel<uint32_t>, true);
  else if (al % 2 == 0) go((unsigned short*)nullptr, copy_rows_kernel<unsigned short>, true);
  else go((unsigned char*)nullptr, copy_rows_kernel<unsigned char>, true);
  return cudaGetLastError();
}

template <typename T, bool VEC>
__global__ void __launch_bounds__(256) gather_tokens_kernel(const float* tok, const float* pos,
                                                            const int32_t* ids, T* __restrict__ z0, int T_, int d,
                                                            int rows, int vocab, int* status, StepTick tk) {
  pdl_wait();
  if (step_tick_cta(tk)) return;
  const int lane = threadIdx.x & 31;
  for (int row = blockIdx.x * 8 + (threadIdx.x >> 5); row < rows; row += work_ctas(tk) * 8) {
    const int t = row % T_, b = row / T_;
    const int id = checked_id(ids[(long long)b * (T_ + 1) + t], vocab, status);
    if (t == T_ - 1 && lane == 0) checked_id(ids[(long long)b * (T_ + 1) + T_], vocab, status);   // the last target is no input
    const float* te = tok + (long long)id * d;
    const float* pe = pos + (long long)t * d;
    T* out = z0 + (long long)row * d;
    if (VEC) {
      for (int c = lane * 4; c < d; c += 512) {      // four pairs of loads in flight, then their stores
        float4 a[4], q[4];
#pragma unroll
        for (int k = 0; k < 4; k++)
          if (c + 128 * k < d) {
            a[k] = *reinterpret_cast<const float4*>(te + c + 128 * k);
            q[k] = *reinterpret_cast<const float4*>(pe + c + 128 * k);
          }
#pragma unroll
        for (int k = 0; k < 4; k++)
          if (c + 128 * k < d) store4(out + c + 128 * k, make_float4(a[k].x + q[k].x, a[k].y + q[k].y, a[k].z + q[k].z, a[k].w + q[k].w));
      }
    } else {
      for (int c = lane; c < d; c += 32) stf(out + c, te[c] + pe[c]);
    }
  }
}
cudaError_t gather_tokens(const float* tok, const float* pos, const int32_t* ids, void* z0, int batch,
                          int T_, int d, int vocab, int* status, const StepTick& tk, bool bf16, cudaStream_t s) {
  const int rows = batch * T_;
  const bool vec = d % 4 == 0 && ((reinterpret_cast<uintptr_t>(tok) | reinterpret_cast<uintptr_t>(pos) | reinterpret_cast<uintptr_t>(z0)) & 15) == 0;
  const int grid = (int)std::min<long long>(cdiv(rows, 8), 148 * 8) + (tk.tick ? 1 : 0);
  if (bf16) {
    if (vec) pdl_launch(gather_tokens_kernel<bf16_t, true>, grid, 256, 0, s, tok, pos, ids, (bf16_t*)z0, T_, d, rows, vocab, status, tk);
    else pdl_launch(gather_tokens_kernel<bf16_t, false>, grid, 256, 0, s, tok, pos, ids, (bf16_t*)z0, T_, d, rows, vocab, status, tk);
  } else {
    if (vec) pdl_launch(gather_tokens_kernel<float, true>, grid, 256, 0, s, tok, pos, ids, (float*)z0, T_, d, rows, vocab, status, tk);
    else pdl_launch(gather_tokens_kernel<float, false>, grid, 256, 0, s, tok, pos, ids, (float*)z0, T_, d, rows, vocab, status, tk);
  }
  return cudaGetLastError();
}

// CTR gather and pack, one warp per sample: x0[n] = [table_t[ids[n,t]] for t | dense | zero pad].
// The lanes run over (table, four columns) pairs, so a table row leaves as 16-byte loads and lands
// as 8-byte (bf16) or 16-byte stores; the dense columns and the padding follow in a scalar tail.
template <typename T, bool VEC>
__global__ void __launch_bounds__(256) gather_ctr_kernel(const float* tables, long long table_stride,
                                                         const int32_t* ids, const float* dense,
                                                         T* __restrict__ x0, int batch, int ns, int e, int nd, int width,
                                                         int table_rows, int* status, StepTick tk) {
  pdl_wait();
  if (step_tick_cta(tk)) return;
  const int lane = threadIdx.x & 31;
  for (int n = blockIdx.x * 8 + (threadIdx.x >> 5); n < batch; n += work_ctas(tk) * 8) {
    T* out = x0 + (long long)n * width;
    const int32_t* idn = ids + (long long)n * ns;
    if (VEC) {
      const int vpr = e >> 2;                                  // 16-byte vectors per table row
      for (int i = lane; i < ns * vpr; i += 32) {
        const int t = i / vpr, c = (i - t * vpr) * 4;
        const int id = checked_id(idn[t], table_rows, status);
        const float4 v = *reinterpret_cast<const float4*>(tables + (long long)t * table_stride + (long long)id * e + c);
        store4(out + t * e + c, v);
      }
    } else {
      for (int i = lane; i < ns * e; i += 32) {
        const int t = i / e, c = i - t * e;
        const int id = checked_id(idn[t], table_rows, status);
        stf(out + i, tables[(long long)t * table_stride + (long long)id * e + c]);
      }
    }
    for (int c = ns * e + lane; c < width; c += 32) stf(out + c, c < ns * e + nd ? dense[(long long)n * nd + (c - ns * e)] : 0.f);
  }
}
cudaError_t gather_ctr(const float* tables, long long table_stride, const int32_t* ids, const float* dense,
                       void* x0, int batch, int ns, int e, int nd, int width, int table_rows, int* status, const StepTick& tk, bool bf16,
                       cudaStream_t s) {
  const bool vec = e % 4 == 0 && width % 4 == 0 && table_stride % 4 == 0 &&
                   ((reinterpret_cast<uintptr_t>(tables) | reinterpret_cast<uintptr_t>(x0)) & 15) == 0;
  const int grid = (int)std::min<long long>(cdiv(batch, 8), 148 * 8) + (tk.tick ? 1 : 0);
  if (bf16) {
    if (vec) pdl_launch(gather_ctr_kernel<bf16_t, true>, grid, 256, 0, s, tables, table_stride, ids, dense, (bf16_t*)x0, batch, ns, e, nd, width, table_rows, status, tk);
    else pdl_launch(gather_ctr_kernel<bf16_t, false>, grid, 256, 0, s, tables, table_stride, ids, dense, (bf16_t*)x0, batch, ns, e, nd, width, table_rows, status, tk);
  } else {
    if (vec) pdl_launch(gather_ctr_kernel<float, true>, grid, 256, 0, s, tables, table_stride, ids, dense, (float*)x0, batch, ns, e, nd, width, table_rows, status, tk);
    else pdl_launch(gather_ctr_kernel<float, false>, grid, 256, 0, s, tables, table_stride, ids, dense, (float*)x0, batch, ns, e, nd, width, table_rows, status, tk);
  }
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------
// dot interaction: one CTA of 128 threads per sample (fp32, and widths that the warp forms below do not take)
// ------------------------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(128) dot_fwd_kernel(const T* proj, const T* x0,
                                                      long long ldx0, T* __restrict__ feats, int ns, int e, int fw) {
  pdl_wait();
  extern __shared__ float sm[];  // [(ns+1)][e+1]
  const int n = blockIdx.x, nv = ns + 1, lde = e + 1;
  for (int i = threadIdx.x; i < nv * e; i += 128) {
    int j = i / e, c = i - j * e;
    sm[j * lde + c] = j == 0 ? ldf(proj + (long long)n * e + c) : ldf(x0 + (long long)n * ldx0 + (j - 1) * e + c);
  }
  __syncthreads();
  const int npair = nv * (nv - 1) / 2;
  T* f = feats + (long long)n * fw;
  for (int p = threadIdx.x; p < fw; p += 128) {
    float v = 0.f;
    if (p < npair) {
      // invert p = i(i-1)/2 + j, 0 <= j < i
      int i = (int)((1.f + sqrtf(1.f + 8.f * p)) * 0.5f);
      while (i * (i - 1) / 2 > p) i--;
      while ((i + 1) * i / 2 <= p) i++;
      int j = p - i * (i - 1) / 2;
      for (int c = 0; c < e; c++) v = fmaf(sm[i * lde + c], sm[j * lde + c], v);
    } else if (p < npair + e) {
      v = sm[p - npair];
    }
    stf(f + p, v);
  }
}
// bf16, e = 64, up to 32 vectors: a warp per sample.  The sample's vectors fill the fragments of m16n8k16 MMAs, rows of A and
// columns of B alike, so lane (g, t) loads 32 contiguous bytes of rows g, g + 8, .. (which columns of the contraction a
// fragment position means does not matter as long as A and B agree) and all 27 x 27 products are 24 MMAs; only the
// tiles that reach under the diagonal are formed.  The features leave from shared memory in 16-byte pieces.
// Bound by memory latency (17 MB at 4096 x 26).  By scalar FMAs out of shared memory 28 us.
__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
constexpr int DOT_WARPS = 4;
__global__ void __launch_bounds__(32 * DOT_WARPS) dot_fwd_mma_kernel(const bf16_t* proj, const bf16_t* x0, long long ldx0, bf16_t* __restrict__ feats, int batch, int ns, int fw) {
  pdl_wait();
  extern __shared__ __align__(16) uint4 dot_rows[];      // fw bf16 per warp
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n = blockIdx.x * DOT_WARPS + warp;
  if (n >= batch) return;
  bf16_t* row = reinterpret_cast<bf16_t*>(dot_rows) + warp * fw;
  const int nv = ns + 1, npair = nv * (nv - 1) / 2, g = lane >> 2, t = lane & 3;
  uint32_t v[4][8];        // [row group][pair of columns]
#pragma unroll
  for (int r = 0; r < 4; r++) {
    const int j = r * 8 + g;
    const uint4* src = reinterpret_cast<const uint4*>(j == 0 ? proj + (long long)n * 64 : x0 + (long long)n * ldx0 + (j - 1) * 64) + t * 2;
    const uint4 lo = j < nv ? src[0] : make_uint4(0u, 0u, 0u, 0u), hi = j < nv ? src[1] : make_uint4(0u, 0u, 0u, 0u);
    v[r][0] = lo.x; v[r][1] = lo.y; v[r][2] = lo.z; v[r][3] = lo.w;
    v[r][4] = hi.x; v[r][5] = hi.y; v[r][6] = hi.z; v[r][7] = hi.w;
  }
  if (g == 0) {            // the projection's own columns
    uint32_t* dst = reinterpret_cast<uint32_t*>(row + npair) + t * 8;
    if (npair % 2 == 0) {
#pragma unroll
      for (int k = 0; k < 8; k++) dst[k] = v[0][k];
    } else {
      unsigned short* d2 = reinterpret_cast<unsigned short*>(row + npair) + t * 16;
#pragma unroll
      for (int k = 0; k < 8; k++) { d2[2 * k] = (unsigned short)v[0][k]; d2[2 * k + 1] = (unsigned short)(v[0][k] >> 16); }
    }
  }
  for (int c = npair + 64 + lane; c < fw; c += 32) row[c] = __float2bfloat16_rn(0.f);
#pragma unroll
  for (int mt = 0; mt < 2; mt++)
#pragma unroll
    for (int nt = 0; nt < 2 * mt + 2; nt++) {
      float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int ks = 0; ks < 4; ks++) {
        const uint32_t a[4] = {v[2 * mt][2 * ks], v[2 * mt + 1][2 * ks], v[2 * mt][2 * ks + 1], v[2 * mt + 1][2 * ks + 1]};
        mma_bf16_16816(c, a, v[nt][2 * ks], v[nt][2 * ks + 1]);
      }
#pragma unroll
      for (int k = 0; k < 4; k++) {
        const int i = mt * 16 + g + (k >> 1) * 8, j = nt * 8 + t * 2 + (k & 1);
        if (j < i && i < nv) row[i * (i - 1) / 2 + j] = __float2bfloat16_rn(c[k]);
      }
    }
  __syncwarp();
  const uint4* src = reinterpret_cast<const uint4*>(row);
  uint4* dst = reinterpret_cast<uint4*>(feats + (long long)n * fw);
  for (int c = lane; c < fw / 8; c += 32) dst[c] = src[c];
}
static bool dot_by_warps(const void* small, const void* x0, long long ldx0, const void* feats, int ns, int e, int fw, bool bf16) {
  return bf16 && e == 64 && ns <= 31 && ldx0 % 8 == 0 && fw % 8 == 0 && fw >= (ns + 1) * ns / 2 + 64 &&
         ((reinterpret_cast<uintptr_t>(small) | reinterpret_cast<uintptr_t>(x0) | reinterpret_cast<uintptr_t>(feats)) & 15) == 0;
}
cudaError_t dot_fwd(const void* proj, const void* x0, long long ldx0, void* feats, int batch, int ns, int e,
                    int fw, bool bf16, cudaStream_t s) {
  if (batch > 0 && dot_by_warps(proj, x0, ldx0, feats, ns, e, fw, bf16) && (size_t)DOT_WARPS * fw * 2 <= 48 * 1024) {
    pdl_launch(dot_fwd_mma_kernel, cdiv(batch, DOT_WARPS), 32 * DOT_WARPS, (size_t)DOT_WARPS * fw * 2, s, (const bf16_t*)proj, (const bf16_t*)x0, ldx0, (bf16_t*)feats, batch, ns, fw);
    return cudaGetLastError();
  }
  size_t smem = (size_t)(ns + 1) * (e + 1) * sizeof(float);
  if (bf16) pdl_launch(dot_fwd_kernel<bf16_t>, batch, 128, smem, s, (const bf16_t*)proj, (const bf16_t*)x0, ldx0, (bf16_t*)feats, ns, e, fw);
  else pdl_launch(dot_fwd_kernel<float>, batch, 128, smem, s, (const float*)proj, (const float*)x0, ldx0, (float*)feats, ns, e, fw);
  return cudaGetLastError();
}

template <typename T>
__global__ void __launch_bounds__(128) dot_bwd_kernel(const T* dfeat, const T* x0,
                                                      long long ldx0, T* __restrict__ dproj, int ns, int e, int fw) {
  pdl_wait();
  const int n = blockIdx.x, nv = ns + 1;
  const int npair = nv * (nv - 1) / 2;
  const T* df = dfeat + (long long)n * fw;
  for (int c = threadIdx.x; c < e; c += 128) {
    float v = ldf(df + npair + c);
    for (int j = 1; j < nv; j++)
      v = fmaf(ldf(df + j * (j - 1) / 2), ldf(x0 + (long long)n * ldx0 + (j - 1) * e + c), v);
    stf(dproj + (long long)n * e + c, v);
  }
}
// The same by a warp per sample: a lane owns two columns, every vector's load is in flight at once, lane j holds the
// gradient of v_j's product with the projection.  (One chain of dependent loads per thread: 16 us at 4096 x 26.)
__global__ void __launch_bounds__(32 * DOT_WARPS) dot_bwd_warp_kernel(const bf16_t* dfeat, const bf16_t* x0, long long ldx0, bf16_t* __restrict__ dproj, int batch, int ns, int fw) {
  pdl_wait();
  const int lane = threadIdx.x & 31, n = blockIdx.x * DOT_WARPS + (threadIdx.x >> 5);
  if (n >= batch) return;
  const int npair = (ns + 1) * ns / 2;
  const bf16_t* df = dfeat + (long long)n * fw;
  const uint32_t* x = reinterpret_cast<const uint32_t*>(x0 + (long long)n * ldx0) + lane;
  uint32_t v[31];
#pragma unroll
  for (int j = 0; j < 31; j++) v[j] = j < ns ? x[j * 32] : 0u;
  const float mine = lane < ns ? ldf(df + (lane + 1) * lane / 2) : 0.f;       // pair (lane + 1, 0)
  float a = ldf(df + npair + 2 * lane), b = ldf(df + npair + 2 * lane + 1);
#pragma unroll
  for (int j = 0; j < 31; j++) {
    const float f = __shfl_sync(0xffffffffu, mine, j);
    a = fmaf(f, __uint_as_float(v[j] << 16), a);
    b = fmaf(f, __uint_as_float(v[j] & 0xffff0000u), b);
  }
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  reinterpret_cast<uint32_t*>(dproj + (long long)n * 64)[lane] = *reinterpret_cast<const uint32_t*>(&h);
}
cudaError_t dot_bwd(const void* dfeat, const void* x0, long long ldx0, void* dproj, int batch, int ns, int e,
                    int fw, bool bf16, cudaStream_t s) {
  if (batch > 0 && dot_by_warps(dproj, x0, ldx0, dfeat, ns, e, fw, bf16)) {
    pdl_launch(dot_bwd_warp_kernel, cdiv(batch, DOT_WARPS), 32 * DOT_WARPS, 0, s, (const bf16_t*)dfeat, (const bf16_t*)x0, ldx0, (bf16_t*)dproj, batch, ns, fw);
    return cudaGetLastError();
  }
  if (bf16) pdl_launch(dot_bwd_kernel<bf16_t>, batch, 128, 0, s, (const bf16_t*)dfeat, (const bf16_t*)x0, ldx0, (bf16_t*)dproj, ns, e, fw);
  else pdl_launch(dot_bwd_kernel<float>, batch, 128, 0, s, (const float*)dfeat, (const float*)x0, ldx0, (float*)dproj, ns, e, fw);
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------
// optimizer
// ------------------------------------------------------------------------------------------
// One element of SGD / Adam / AdamW; every path below applies exactly this arithmetic.
__device__ __forceinline__ void opt_element(float& th, float g, float& mm, float& vv, int kind, float lr, float b1, float b2,
                                            float eps, float wd, float bc1, float bc2) {
  if (kind == 0) {
    th -= lr * g;
  } else {
    if (kind == 2) th *= (1.f - lr * wd);
    mm = b1 * mm + (1.f - b1) * g;
    vv = b2 * vv + (1.f - b2) * g * g;
    th -= lr * (mm / bc1) / (sqrtf(vv / bc2) + eps);
  }
}

// Four consecutive parameters per thread (16-byte accesses; the arenas are 256-byte aligned and a
// block's slice starts on a multiple of 64 elements); the last, partial quad is done element-wise.
__global__ void __launch_bounds__(256) opt_update_kernel(float* __restrict__ theta, const float* grad,
                                                         float* __restrict__ m, float* __restrict__ v,
                                                         bf16_t* __restrict__ shadow, long long n, int kind, float lr,
                                                         float b1, float b2, float eps, float wd,
                                                         const double* tick, int vec) {
  pdl_wait();
  const long long q = (long long)blockIdx.x * 256 + threadIdx.x;
  const long long i = q * 4;
  if (i >= n) return;
  float bc1 = 1.f, bc2 = 1.f;
  if (kind != 0) { bc1 = (float)tick[1]; bc2 = (float)tick[2]; }
  if (vec && i + 4 <= n) {
    float4 th = reinterpret_cast<float4*>(theta)[q];
    const float4 g = reinterpret_cast<const float4*>(grad)[q];
    float4 mm = make_float4(0.f, 0.f, 0.f, 0.f), vv = mm;
    if (kind != 0) { mm = reinterpret_cast<float4*>(m)[q]; vv = reinterpret_cast<float4*>(v)[q]; }
    opt_element(th.x, g.x, mm.x, vv.x, kind, lr, b1, b2, eps, wd, bc1, bc2);
    opt_element(th.y, g.y, mm.y, vv.y, kind, lr, b1, b2, eps, wd, bc1, bc2);
    opt_element(th.z, g.z, mm.z, vv.z, kind, lr, b1, b2, eps, wd, bc1, bc2);
    opt_element(th.w, g.w, mm.w, vv.w, kind, lr, b1, b2, eps, wd, bc1, bc2);
    if (kind != 0) { reinterpret_cast<float4*>(m)[q] = mm; reinterpret_cast<float4*>(v)[q] = vv; }
    reinterpret_cast<float4*>(theta)[q] = th;
    if (shadow) {
      __nv_bfloat162 lo = __floats2bfloat162_rn(th.x, th.y), hi = __floats2bfloat162_rn(th.z, th.w);
      uint2 w;
      w.x = *reinterpret_cast<uint32_t*>(&lo);
      w.y = *reinterpret_cast<uint32_t*>(&hi);
      reinterpret_cast<uint2*>(shadow)[q] = w;
    }
    return;
  }
  for (long long k = i; k < n && k < i + 4; k++) {
    float th = theta[k], mm = 0.f, vv = 0.f;
    if (kind != 0) { mm = m[k]; vv = v[k]; }
    opt_element(th, grad[k], mm, vv, kind, lr, b1, b2, eps, wd, bc1, bc2);
    if (kind != 0) { m[k] = mm; v[k] = vv; }
    theta[k] = th;
    if (shadow) shadow[k] = __float2bfloat16_rn(th);
  }
}
cudaError_t opt_update(float* theta, const float* grad, float* m, float* v, void* shadow, long long n, int kind,
                       float lr, float beta1, float beta2, float eps, float wd, const double* tick,
                       cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  auto al = [](const void* p, uintptr_t a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0; };
  const int vec = al(theta, 16) && al(grad, 16) && (!m || al(m, 16)) && (!v || al(v, 16)) && (!shadow || al(shadow, 8));
  pdl_launch(opt_update_kernel, cdiv((n + 3) / 4, 256), 256, 0, s, theta, grad, m, v, (bf16_t*)shadow, n, kind, lr, beta1, beta2, eps, wd, tick, vec);
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------
// The undetached remainder (Section 2.2, Eq. 2): input of the main network and the embedding backward
// ------------------------------------------------------------------------------------------
// u[n, off_s .. off_s + w_s) = src_s[n, 0 .. w_s) for up to CONCAT_MAX sources: u = [z_0 | z_1 | ... | z_B]
// One warp per (row, source); 16-byte pieces where every source's width and place allow them (VECTOR), which a
// copy by single elements with a division per element cannot follow (3001 rows x 5548 columns, 67 MB read and
// written: 41 us, now 10).
template <typename T, bool VECTOR>
__global__ void __launch_bounds__(256) concat_kernel(ConcatArgs a, T* __restrict__ u, int rows) {
  pdl_wait();
  const int src = blockIdx.y, lane = threadIdx.x & 31;
  const T* p = (const T*)a.src[src];
  const int w = a.width[src], off = a.offset[src];
  for (int r = blockIdx.x * 8 + (threadIdx.x >> 5); r < rows; r += gridDim.x * 8) {
    const T* from = p + (long long)r * a.ld[src];
    T* to = u + (long long)r * a.total + off;
    if (VECTOR) {
      const int n = w / VecOf<T>::N;
      for (int i = lane; i < n; i += 128) {      // four loads in flight, then their stores
        uint4 q[4];
#pragma unroll
        for (int k = 0; k < 4; k++)
          if (i + 32 * k < n) q[k] = reinterpret_cast<const uint4*>(from)[i + 32 * k];
#pragma unroll
        for (int k = 0; k < 4; k++)
          if (i + 32 * k < n) reinterpret_cast<uint4*>(to)[i + 32 * k] = q[k];
      }
    } else {
      for (int c = lane; c < w; c += 32) to[c] = from[c];
    }
  }
}
cudaError_t concat_cols(const ConcatArgs& a, void* u, int rows, bool bf16, cudaStream_t s) {
  const int vec = bf16 ? 8 : 4;
  bool v = a.total % vec == 0 && (reinterpret_cast<uintptr_t>(u) & 15) == 0;
  for (int i = 0; i < a.n; i++)
    v = v && a.width[i] % vec == 0 && a.offset[i] % vec == 0 && a.ld[i] % vec == 0 && (reinterpret_cast<uintptr_t>(a.src[i]) & 15) == 0;
  dim3 grid((unsigned)std::min<long long>(cdiv(rows, 8), 148 * 8), a.n);
  if (bf16) {
    if (v) pdl_launch(concat_kernel<bf16_t, true>, grid, 256, 0, s, a, (bf16_t*)u, rows);
    else pdl_launch(concat_kernel<bf16_t, false>, grid, 256, 0, s, a, (bf16_t*)u, rows);
  } else {
    if (v) pdl_launch(concat_kernel<float, true>, grid, 256, 0, s, a, (float*)u, rows);
    else pdl_launch(concat_kernel<float, false>, grid, 256, 0, s, a, (float*)u, rows);
  }
  return cudaGetLastError();
}

// Embedding backward, step 1: one CTA per table sorts its (id, sample) pairs by id, so that the samples that read
// one table row are contiguous and in sample order, and numbers the distinct rows: sorted_n[t][pos] = sample at
// sorted position pos, seg_start[t][s] = first position of the s-th distinct row (seg_start[t][n_uniq] = batch),
// uniq_id[t][s] = that row, n_uniq[t].
// A stable radix sort in shared memory, `passes` digits of `bits` <= 8 bits each, lowest first: a warp owns a
// contiguous run of positions and counts its digits with match_any (one writer per counter, no atomics), a scan
// over (digit, warp) turns the counts into places, and the warps move their runs in order.  What bounds it is the
// latency of one CTA's steps: passes x 3 barriers against the n log^2 n / 2 = 78 barriers of a bitonic network on
// 4096 pairs (with step 2, 26 tables of 20000 rows and 3001 samples: 176 us before, 43 now).
__global__ void __launch_bounds__(1024) embed_sort_kernel(const int32_t* ids, int batch, int ns, int table_rows, int passes,
                                                          int bits, int* __restrict__ sorted_n, int* __restrict__ seg_start,
                                                          int* __restrict__ uniq_id, int* __restrict__ n_uniq) {
  pdl_wait();
  extern __shared__ unsigned sort_smem[];
  unsigned* key[2] = {sort_smem, sort_smem + batch};                                       // id
  unsigned short* idx[2] = {reinterpret_cast<unsigned short*>(sort_smem + 2 * batch),     // sample (batch <= 16384)
                            reinterpret_cast<unsigned short*>(sort_smem + 2 * batch) + batch};
  __shared__ unsigned short count[256 * 32];                 // [digit][warp]
  __shared__ int scan[1024];
  const int t = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int i = threadIdx.x; i < batch; i += 1024) {
    const int id = ids[(long long)i * ns + t];
    key[0][i] = (unsigned)min(max(id, 0), table_rows - 1);   // a bad id was reported by the input staging
    idx[0][i] = (unsigned short)i;
  }
  const int run = (batch + 31) / 32, beg = min(batch, warp * run), end = min(batch, beg + run);
  const unsigned mask = (1u << bits) - 1u;
  int cur = 0;
  for (int pass = 0; pass < passes; pass++, cur ^= 1) {
    const int shift = pass * bits;
    for (int i = threadIdx.x; i < 256 * 32; i += 1024) count[i] = 0;
    __syncthreads();
    for (int i0 = beg; i0 < end; i0 += 32) {
      const int i = i0 + lane;
      const unsigned active = __ballot_sync(0xffffffffu, i < end);
      if (i < end) {
        const unsigned d = (key[cur][i] >> shift) & mask;
        const unsigned same = __match_any_sync(active, d);
        if (lane == __ffs(same) - 1) count[d * 32 + warp] += (unsigned short)__popc(same);
      }
      __syncwarp();
    }
    __syncthreads();
    int c[8], sum = 0;                                       // exclusive scan over the 8192 counters, eight per thread
#pragma unroll
    for (int j = 0; j < 8; j++) { c[j] = count[threadIdx.x * 8 + j]; sum += c[j]; }
    int inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += v;
    }
    if (lane == 31) scan[warp] = inc;
    __syncthreads();
    int base = inc - sum;
    for (int w = 0; w < warp; w++) base += scan[w];
#pragma unroll
    for (int j = 0; j < 8; j++) { count[threadIdx.x * 8 + j] = (unsigned short)base; base += c[j]; }
    __syncthreads();
    for (int i0 = beg; i0 < end; i0 += 32) {
      const int i = i0 + lane;
      const unsigned active = __ballot_sync(0xffffffffu, i < end);
      if (i < end) {
        const unsigned k = key[cur][i], d = (k >> shift) & mask;
        const unsigned same = __match_any_sync(active, d);
        const int pos = count[d * 32 + warp] + __popc(same & ((1u << lane) - 1u));
        key[cur ^ 1][pos] = k;
        idx[cur ^ 1][pos] = idx[cur][i];
        __syncwarp(active);
        if (lane == __ffs(same) - 1) count[d * 32 + warp] += (unsigned short)__popc(same);
      }
      __syncwarp();
    }
    __syncthreads();
  }
  if (passes == 0) __syncthreads();
  const unsigned* keys = key[cur];
  // segment starts and their numbering: every thread owns a contiguous run of positions
  const int per = (batch + 1023) / 1024, lo = threadIdx.x * per, hi = min(batch, lo + per);
  int cnt = 0;
  for (int i = lo; i < hi; i++) cnt += (i == 0 || keys[i] != keys[i - 1]);
  scan[threadIdx.x] = cnt;
  __syncthreads();
  for (int o = 1; o < 1024; o <<= 1) {                       // inclusive scan over the 1024 counts
    const int v = threadIdx.x >= o ? scan[threadIdx.x - o] : 0;
    __syncthreads();
    scan[threadIdx.x] += v;
    __syncthreads();
  }
  int seg = scan[threadIdx.x] - cnt;
  int* sn = sorted_n + (long long)t * batch;
  int* ss = seg_start + (long long)t * (batch + 1);
  int* ui = uniq_id + (long long)t * batch;
  for (int i = lo; i < hi; i++) {
    sn[i] = idx[cur][i];
    if (i == 0 || keys[i] != keys[i - 1]) {
      ss[seg] = i;
      ui[seg] = (int)keys[i];
      seg++;
    }
  }
  if (threadIdx.x == 1023) {
    n_uniq[t] = scan[1023];
    ss[scan[1023]] = batch;
  }
}

// Step 2: grow[t][s][:] = sum over the samples of segment s of dz0[n, t*e : (t+1)*e] -- the scatter-add without
// atomics.  A warp takes one distinct row; L = e / VEC lanes hold its columns (16-byte loads) and the 32/L groups
// of lanes take every (32/L)-th sample, four loads in flight each; the groups are added in a fixed order.  The
// ids are Zipf distributed, so one row may own a seventh of the batch: segments above EMBED_LONG samples are
// shared by the CTA's eight warps, whose sums are added in warp order.
// What bounds it is the latency of the longest segment: 435 dependent steps of one warp before, 4 now.
constexpr int EMBED_LONG = 64;
template <typename T, int L>
__device__ __forceinline__ void embed_segment(const T* col, long long ld, const int* sn, int beg, int end,
                                              int lane, float (&acc)[VecOf<T>::N]) {
  constexpr int VEC = VecOf<T>::N, G = 32 / L;
  const T* p = col + (lane % L) * VEC;
#pragma unroll
  for (int j = 0; j < VEC; j++) acc[j] = 0.f;
  for (int pos = beg + lane / L; pos < end; pos += 4 * G) {
    float v[4][VEC];
#pragma unroll
    for (int u = 0; u < 4; u++) {
      if (pos + u * G < end) {
        ld_vec<T>(p + (long long)sn[pos + u * G] * ld, v[u]);
      } else {
#pragma unroll
        for (int j = 0; j < VEC; j++) v[u][j] = 0.f;
      }
    }
#pragma unroll
    for (int u = 0; u < 4; u++)
#pragma unroll
      for (int j = 0; j < VEC; j++) acc[j] += v[u][j];
  }
#pragma unroll
  for (int o = L; o < 32; o <<= 1)
#pragma unroll
    for (int j = 0; j < VEC; j++) acc[j] += __shfl_xor_sync(0xffffffffu, acc[j], o);
}
template <typename T, int L>
__global__ void __launch_bounds__(256) embed_rows_vec_kernel(const T* dz0, long long ld, int batch,
                                                             const int* sorted_n, const int* seg_start,
                                                             const int* n_uniq, float* __restrict__ grow) {
  pdl_wait();
  constexpr int VEC = VecOf<T>::N, E = L * VEC;
  __shared__ float part[8][E];
  const int t = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nu = n_uniq[t];
  const int first = blockIdx.x * 8;
  if (first >= nu) return;
  const int* sn = sorted_n + (long long)t * batch;
  const int* ss = seg_start + (long long)t * (batch + 1);
  const T* col = dz0 + t * E;
  float* out = grow + (long long)t * batch * E;
  float acc[VEC];
  if (first + warp < nu) {
    const int beg = ss[first + warp], end = ss[first + warp + 1];
    if (end - beg <= EMBED_LONG) {
      embed_segment<T, L>(col, ld, sn, beg, end, lane, acc);
      if (lane < L)
#pragma unroll
        for (int j = 0; j < VEC; j++) out[(long long)(first + warp) * E + lane * VEC + j] = acc[j];
    }
  }
  for (int s = 0; s < 8 && first + s < nu; s++) {
    const int beg = ss[first + s], end = ss[first + s + 1];
    if (end - beg <= EMBED_LONG) continue;                   // the same for every warp
    const int per = (end - beg + 7) / 8, b = min(end, beg + warp * per);
    embed_segment<T, L>(col, ld, sn, b, min(end, b + per), lane, acc);
    if (lane < L)
#pragma unroll
      for (int j = 0; j < VEC; j++) part[warp][lane * VEC + j] = acc[j];
    __syncthreads();
    for (int c = threadIdx.x; c < E; c += 256) {
      float v = 0.f;
#pragma unroll
      for (int w = 0; w < 8; w++) v += part[w][c];
      out[(long long)(first + s) * E + c] = v;
    }
    __syncthreads();
  }
}
// any embedding width: one warp per distinct row, its lanes over the columns, samples in order
template <typename T>
__global__ void __launch_bounds__(256) embed_rows_kernel(const T* dz0, long long ld, int batch, int e,
                                                         const int* sorted_n, const int* seg_start,
                                                         const int* n_uniq, float* __restrict__ grow) {
  pdl_wait();
  const int t = blockIdx.y, seg = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (seg >= n_uniq[t]) return;
  const int* sn = sorted_n + (long long)t * batch;
  const int* ss = seg_start + (long long)t * (batch + 1);
  const int beg = ss[seg], end = ss[seg + 1];
  for (int c = lane; c < e; c += 32) {
    float acc = 0.f;
    for (int pos = beg; pos < end; pos++) acc += ldf(dz0 + (long long)sn[pos] * ld + t * e + c);
    grow[((long long)t * batch + seg) * e + c] = acc;
  }
}

// Step 3: the optimizer on the touched rows only (untouched rows keep values and moments; the bias
// correction is the global one in tick[]); the same element update as the dense optimizer.
__global__ void __launch_bounds__(256) embed_update_kernel(float* __restrict__ tables, long long table_stride, float* __restrict__ m,
                                                           float* __restrict__ v, int batch, int e, const int* uniq_id,
                                                           const int* n_uniq, const float* grow, int kind,
                                                           float lr, float b1, float b2, float eps, float wd,
                                                           const double* tick) {
  pdl_wait();
  const int t = blockIdx.y, seg = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (seg >= n_uniq[t]) return;
  float bc1 = 1.f, bc2 = 1.f;
  if (kind != 0) { bc1 = (float)tick[1]; bc2 = (float)tick[2]; }
  const long long base = (long long)t * table_stride + (long long)uniq_id[(long long)t * batch + seg] * e;
  for (int c = lane; c < e; c += 32) {
    float th = tables[base + c], mm = 0.f, vv = 0.f;
    if (kind != 0) { mm = m[base + c]; vv = v[base + c]; }
    opt_element(th, grow[((long long)t * batch + seg) * e + c], mm, vv, kind, lr, b1, b2, eps, wd, bc1, bc2);
    if (kind != 0) { m[base + c] = mm; v[base + c] = vv; }
    tables[base + c] = th;
  }
}

int embed_max_batch() { return 16384; }

cudaError_t embed_sort(const int32_t* ids, int batch, int ns, int table_rows, int* sorted_n, int* seg_start, int* uniq_id, int* n_uniq,
                       cudaStream_t s) {
  int idbits = 0;
  while (idbits < 31 && (1LL << idbits) < table_rows) idbits++;
  const int passes = (idbits + 7) / 8, bits = passes ? (idbits + passes - 1) / passes : 0;
  const size_t smem = (size_t)batch * 2 * (sizeof(unsigned) + sizeof(unsigned short));
  static std::atomic<size_t> attr[64];
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) dev = 0;
  if (smem > 8 * 1024 && smem > attr[dev].load()) {      // 20 KB of counters beside it: past the default limit soon after
    cudaError_t e2 = cudaFuncSetAttribute(embed_sort_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e2 != cudaSuccess) return e2;
    attr[dev].store(smem);
  }
  pdl_launch(embed_sort_kernel, ns, 1024, smem, s, ids, batch, ns, table_rows, passes, bits, sorted_n, seg_start, uniq_id, n_uniq);
  return cudaGetLastError();
}
cudaError_t embed_backward(const void* dz0, long long ld, int batch, int ns, int e, const int* sorted_n, const int* seg_start, const int* n_uniq,
                           float* grow, bool bf16, cudaStream_t s) {
  dim3 grid(cdiv(batch, 8), ns);
  const int vec = bf16 ? 8 : 4;
  const int lanes = e % vec == 0 && ld % vec == 0 && (reinterpret_cast<uintptr_t>(dz0) & 15) == 0 ? e / vec : 0;
  auto vecs = [&](auto L) {
    if (bf16) pdl_launch(embed_rows_vec_kernel<bf16_t, decltype(L)::value>, grid, 256, 0, s, (const bf16_t*)dz0, ld, batch, sorted_n, seg_start, n_uniq, grow);
    else pdl_launch(embed_rows_vec_kernel<float, decltype(L)::value>, grid, 256, 0, s, (const float*)dz0, ld, batch, sorted_n, seg_start, n_uniq, grow);
  };
  switch (lanes) {
    case 1: vecs(std::integral_constant<int, 1>()); break;
    case 2: vecs(std::integral_constant<int, 2>()); break;
    case 4: vecs(std::integral_constant<int, 4>()); break;
    case 8: vecs(std::integral_constant<int, 8>()); break;
    case 16: vecs(std::integral_constant<int, 16>()); break;
    case 32: vecs(std::integral_constant<int, 32>()); break;
    default:
      if (bf16) pdl_launch(embed_rows_kernel<bf16_t>, grid, 256, 0, s, (const bf16_t*)dz0, ld, batch, e, sorted_n, seg_start, n_uniq, grow);
      else pdl_launch(embed_rows_kernel<float>, grid, 256, 0, s, (const float*)dz0, ld, batch, e, sorted_n, seg_start, n_uniq, grow);
  }
  return cudaGetLastError();
}

cudaError_t embed_update(float* tables, long long table_stride, float* m, float* v, int batch, int ns, int e, const int* uniq_id,
                         const int* n_uniq, const float* grow, int kind, float lr, float beta1, float beta2, float eps, float wd,
                         const double* tick, cudaStream_t s) {
  dim3 grid(cdiv(batch, 8), ns);
  pdl_launch(embed_update_kernel, grid, 256, 0, s, tables, table_stride, m, v, batch, e, uniq_id, n_uniq, grow, kind, lr, beta1, beta2, eps, wd, tick);
  return cudaGetLastError();
}

__global__ void to_bf16_kernel(const float* src, bf16_t* __restrict__ dst, long long n) {
  pdl_wait();
  long long i = (long long)blockIdx.x * 256 + threadIdx.x;
  if (i < n) dst[i] = __float2bfloat16_rn(src[i]);
}
cudaError_t to_bf16(const float* src, void* dst, long long n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  pdl_launch(to_bf16_kernel, cdiv(n, 256), 256, 0, s, src, (bf16_t*)dst, n);
  return cudaGetLastError();
}

}  // namespace erase
