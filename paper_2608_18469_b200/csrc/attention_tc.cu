// Causal flash attention on the 5th-generation tensor cores (tcgen05 / TMEM / TMA) for bf16 models
// with 64-wide heads: forward, dK/dV and dQ kernels.  No T x T matrix is ever written to memory;
// the backward recomputes the probabilities from the saved log-sum-exp.  dK/dV and dQ are separate
// kernels (one walks over query tiles, the other over key tiles), so every output element has one
// writer and a fixed summation order: no atomics, bit-reproducible.
//
// Tiles are 128 x 128 (queries x keys).  Q, K, V (and dO) tiles are fetched by TMA straight out of
// the [rows, 3 d] qkv matrix (128-byte swizzle: a head's 64 columns are one swizzle row).  Every
// product is one tcgen05.mma chain issued by one elected lane with its accumulator in tensor memory:
//     S = Q K^T        A = Q  [q, dh]   K-major      B = K [key, dh]  K-major     (M 128, N 128, K 64)
//     O = P V          A = P  [q, key]  K-major      B = V [key, dh]  MN-major    (M 128, N  64, K 128)
// and in the backward the same tiles read through the other descriptor kind (a [row, dh] tile is a
// K-major operand when the contraction runs over dh and an MN-major one when it runs over rows), so
// nothing is ever transposed in memory.  Four softmax warps own one accumulator row (TMEM lane) per
// thread: they read S with tcgen05.ld, exponentiate, and write P (bf16) into shared memory in the
// swizzled K-major layout the next MMA reads.
//
// What bounds them (ncu, 8 sequences x 12 heads x 1024): the softmax warps' own instruction and latency chain; the
// exponentials alone take 37 % of the MUFU pipe, tensor pipe 20 .. 26 %, DRAM under 15 %.  Three things shorten it: the next
// sub-tile's score MMAs are issued as soon as the scores have been read into registers, so the softmax warps do not wait
// for them; arithmetic on f32x2 pairs with the scale and reference folded into one fma; and the tile as the SLOWEST index
// of a block (attention_grid.cuh), so that the long walks of all heads start first (as the fastest index it left SMs with 28 .. 50 % of MUFU
// time, average 37 %: a quarter of the kernel was its tail).  Forward 54.8 -> 41 us, dQ 60.9 -> 45, dK/dV 81.5 -> 62.
// All waits are clock-bounded; on expiry the model's
// status word is set, the kernel still frees its tensor memory and returns.
#include <cuda.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include <atomic>

#include "gemm_tc.cuh"
#include "attention_grid.cuh"
#include "kernels.cuh"
#include "launch.cuh"
#include "tc_ptx.cuh"
#include "ew_math.cuh"

namespace erase {

namespace {

typedef __nv_bfloat16 bf16_t;
constexpr int TQ = 128;              // queries per tile
constexpr int TK = 128;              // keys per tile
constexpr int DH = 64;               // head width
constexpr uint32_t TILE_BYTES = 128 * DH * 2;     // a [128, 64] bf16 tile: 128 swizzle rows of 128 bytes
constexpr uint32_t P_BYTES = 2 * TILE_BYTES;      // a [128, 128] bf16 tile: two 64-column halves
constexpr int AT_THREADS = 160;      // warps 0..3 softmax (TMEM lane quarters 0..3), warp 4 issues TMA and MMA
constexpr float LOG2E = 1.4426950408889634f;

__device__ __forceinline__ void set_status(int* st, int code) { if (st) atomicExch(st, code); }
__device__ __forceinline__ uint32_t pack_bf(float lo, float hi) {
  __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&h);
}
__device__ __forceinline__ void sts_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
// instruction descriptor: bf16 x bf16 -> fp32, M = 128, given N and operand majors
__device__ __forceinline__ uint32_t idesc_of(int n, bool a_mn, bool b_mn) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn ? 1u : 0u) << 15) | ((b_mn ? 1u : 0u) << 16) |
         ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}
// K-major [128 rows, 64 k] tile: k step of 16 elements = 32 bytes inside the swizzled row
__device__ __forceinline__ uint64_t desc_k(uint32_t tile, int k16) { return smem_desc(tile + k16 * 32, 16, 1024); }
// MN-major [64 k rows][64 m/n] block (128-byte runs along M/N, one per k): k step of 16 = 16 rows = 2048 bytes;
// the next 64 M/N elements, if any, sit `lbo` bytes further
__device__ __forceinline__ uint64_t desc_mn(uint32_t block, int k16, uint32_t lbo) { return smem_desc(block + k16 * 2048, lbo, 1024); }

// Writes 32 consecutive values of this thread's row (bf16) into a K-major [128, 128] operand tile:
// column c lives in half c / 64; inside a half a row is 128 bytes whose 16-byte pieces are XOR-ed
// with the row (the 128-byte swizzle the descriptors and TMA assume).
__device__ __forceinline__ void store_p32(uint32_t tile, int row, int col0, const float* v) {
  const uint32_t base = tile + (uint32_t)(col0 >> 6) * TILE_BYTES + (uint32_t)row * 128u;
  const int piece0 = (col0 & 63) >> 3;
#pragma unroll
  for (int g = 0; g < 4; g++)
    sts_v4(base + (uint32_t)(((piece0 + g) ^ (row & 7)) << 4), pack_bf(v[8 * g], v[8 * g + 1]), pack_bf(v[8 * g + 2], v[8 * g + 3]),
           pack_bf(v[8 * g + 4], v[8 * g + 5]), pack_bf(v[8 * g + 6], v[8 * g + 7]));
}

struct AttnArgs {
  int T, H, batch;
  float scale;           // 1 / sqrt(dh)
  float scale_log2;      // scale * log2(e)
  bf16_t* o;             // forward output [rows, d]
  float* lse;            // [batch, H, T], natural log (written by the forward, read by the backward)
  float* delta;          // backward: [batch, H, T], sum_c dO * O (written by the dQ kernel, read by the dK/dV kernel)
  bf16_t* dqkv;          // backward output [rows, 3 d]
  int* status;
};

// ------------------------------------------------------------------------------------------------
// forward: one CTA per (query tile, head, sequence); key tiles 0 .. query tile
// ------------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(AT_THREADS, 2)
attn_fwd_tc_kernel(const __grid_constant__ CUtensorMap map_qkv, const __grid_constant__ AttnArgs p) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t base = smem_u32(smem_raw);       // the swizzled tiles need 1024-byte alignment: checked below
  const uint32_t q_s = base, k_s = base + TILE_BYTES, v_s = k_s + 2 * TILE_BYTES, p_s = v_s + 2 * TILE_BYTES;
  const uint32_t bar = p_s + P_BYTES;
  const uint32_t q_full = bar, kv_full0 = bar + 8, kv_empty0 = bar + 24, s_full = bar + 40, p_full = bar + 48, o_full = bar + 56,
                 s_free = bar + 64, tmem_slot = bar + 72;
  volatile uint32_t* tmem_slot_ptr = reinterpret_cast<volatile uint32_t*>(smem_raw + (tmem_slot - smem_u32(smem_raw)));

  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // (warp: known to be uniform)
  const AttnPlace at = attn_place(blockIdx.x, p.H, p.batch);
  const int qt = (p.T - 1) / TQ - at.tile, h = at.head, b = at.seq;      // long key ranges first
  const int d = p.H * DH;
  const int q0 = qt * TQ;
  const int nt = qt + 1;                                       // key tiles 0..qt (TQ == TK)
  int st0 = status_peek(p.status);
  if (threadIdx.x == 0 && (base & 1023u)) { set_status(p.status, 10); st0 = 10; }   // never expected: do nothing rather than misread tiles

  if (threadIdx.x == 0) {
    mbar_init(q_full, 1);
    for (int s = 0; s < 2; s++) { mbar_init(kv_full0 + 8 * s, 1); mbar_init(kv_empty0 + 8 * s, 1); }
    mbar_init(s_full, 1);
    mbar_init(p_full, 4);
    mbar_init(o_full, 1);
    mbar_init(s_free, 4);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 4) {
    if (lane == 0) asm volatile("prefetch.tensormap [%0];" ::"l"(&map_qkv) : "memory");
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tmem_slot), "r"(256u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  pdl_wait();
  const bool dead = __syncthreads_or(st0 != 0) != 0;
  tc_fence_after();
  const uint32_t tmem = *tmem_slot_ptr;
  const uint32_t tm_s = tmem, tm_o = tmem + 128;

  if (dead) {
    // the step is already void
  } else if (warp == 4) {
    // ------------------ TMA and MMA: the whole warp walks through the steps, one elected lane issues ------------------
    const int row0 = b * p.T;
    auto load_kv = [&](int j) {
      const int s = j & 1;
      if (elect_one()) {
        mbar_expect_tx(kv_full0 + 8 * s, 2 * TILE_BYTES);
        tma_load_2d(k_s + s * TILE_BYTES, &map_qkv, d + h * DH, row0 + j * TK, kv_full0 + 8 * s);
        tma_load_2d(v_s + s * TILE_BYTES, &map_qkv, 2 * d + h * DH, row0 + j * TK, kv_full0 + 8 * s);
      }
    };
    if (elect_one()) {
      mbar_expect_tx(q_full, TILE_BYTES);
      tma_load_2d(q_s, &map_qkv, h * DH, row0 + q0, q_full);
    }
    load_kv(0);
    if (nt > 1) load_kv(1);
    const uint32_t id_s = idesc_of(TK, false, false), id_o = idesc_of(DH, false, true);
    int fail = mbar_wait_warp(q_full, 0) ? 0 : 11;
    // S_j is issued as soon as S_{j-1} has been read into registers, in front of O += P_{j-1} V_{j-1}: it is ready
    // when the softmax warps come back for it
    for (int j = 0; j <= nt && fail == 0; j++) {
      const int s = j & 1;
      if (j < nt) {
        if (!mbar_wait_warp(kv_full0 + 8 * s, (j >> 1) & 1)) { fail = 12; break; }
        if (j > 0 && !mbar_wait_warp(s_free, (j - 1) & 1)) { fail = 14; break; }
        tc_fence_after();
#pragma unroll
        for (int kk = 0; kk < DH / 16; kk++) tc_mma_warp(tm_s, desc_k(q_s, kk), desc_k(k_s + s * TILE_BYTES, kk), id_s, kk > 0 ? 1u : 0u);
        tc_commit_warp<1>(s_full);
      }
      if (j > 0) {
        const int i = j - 1, si = i & 1;
        if (!mbar_wait_warp(p_full, i & 1)) { fail = 13; break; }             // P_i written (and O rescaled, if it had to be)
        tc_fence_after();
#pragma unroll
        for (int kk = 0; kk < TK / 16; kk++)
          tc_mma_warp(tm_o, desc_k(p_s + (kk >> 2) * TILE_BYTES, kk & 3), desc_mn(v_s + si * TILE_BYTES + (kk >> 2) * (TILE_BYTES / 2), kk & 3, TILE_BYTES / 2),
                      id_o, (i > 0 || kk > 0) ? 1u : 0u);
        tc_commit_warp<1>(o_full);
        tc_commit_warp<1>(kv_empty0 + 8 * si);
        if (i + 2 < nt) {                   // tile i+2 goes where tile i was, once its MMAs have read it
          if (!mbar_wait_warp(kv_empty0 + 8 * si, (i >> 1) & 1)) { fail = 15; break; }
          load_kv(i + 2);
        }
      }
    }
    if (fail) {   // give copies in flight time to land before shared memory is released
      if (lane == 0) set_status(p.status, fail);
      const long long t0 = clock64();
      while (clock64() - t0 < 2000000LL) {}
    }
    pdl_trigger();
  } else {
    // ------------------------------ softmax warps: one accumulator row per thread ------------------------------
    // A row's 128 scores are read once into registers (and S handed back at once).  The output stays in tensor memory:
    // exponentials are taken relative to a reference that follows the row maximum only when that has grown by more
    // than 2^8 since, so the accumulator is read, scaled and written back a few times per row at most; the weights
    // are then at most 256 instead of 1, which changes neither their relative rounding nor that of the sums.
    const int row = warp * 32 + lane;                 // row of the tile = TMEM lane
    const uint32_t lane_off = (uint32_t)(warp * 32) << 16;
    float m_ref = 0.f, l = 0.f;
    int fail = 0;
    for (int j = 0; j < nt; j++) {
      if (!mbar_wait_warp(s_full, j & 1)) { fail = 17; break; }
      tc_fence_after();
      uint32_t r[TK];
#pragma unroll
      for (int c = 0; c < TK / 32; c++) tc_ld32_issue(tm_s + lane_off + c * 32, r + c * 32);
#pragma unroll
      for (int c = 0; c < TK / 32; c++) tc_ld_wait(r + c * 32);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(s_free);
      if (j == nt - 1) {                              // the only tile with keys beyond some of its queries
#pragma unroll
        for (int e = 0; e < TK; e++)
          if (e > row) r[e] = 0xff800000u;            // -inf
      }
      float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
      for (int e = 0; e < TK; e += 4)
#pragma unroll
        for (int q = 0; q < 4; q++) mx[q] = fmaxf(mx[q], __uint_as_float(r[e + q]));
      const float top = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * p.scale_log2;
      if (j == 0) {
        m_ref = top;
      } else if (__any_sync(0xffffffffu, top > m_ref + 8.f)) {
        if (!mbar_wait_warp(o_full, (j - 1) & 1)) { fail = 16; break; }
        tc_fence_after();
        const float m_new = fmaxf(m_ref, top), alpha = ex2_fast(m_ref - m_new);
        uint32_t q[32];
#pragma unroll 1
        for (int c = 0; c < DH; c += 32) {
          tc_ld32(tm_o + lane_off + c, q);
#pragma unroll
          for (int e = 0; e < 32; e++) q[e] = __float_as_uint(__uint_as_float(q[e]) * alpha);
          tc_st32(tm_o + lane_off + c, q);
        }
        l *= alpha;
        m_ref = m_new;
      }
      const f32x2 sc = pack_f2(p.scale_log2, p.scale_log2), nm = pack_f2(-m_ref, -m_ref), one = pack_f2(1.f, 1.f);
      f32x2 sum0 = pack_f2(0.f, 0.f), sum1 = sum0;
#pragma unroll
      for (int e = 0; e < TK; e += 4) {
        float x0, x1, x2, x3;
        unpack_f2(fma_f2(pack_f2(__uint_as_float(r[e]), __uint_as_float(r[e + 1])), sc, nm), x0, x1);
        unpack_f2(fma_f2(pack_f2(__uint_as_float(r[e + 2]), __uint_as_float(r[e + 3])), sc, nm), x2, x3);
        x0 = ex2_fast(x0); x1 = ex2_fast(x1); x2 = ex2_fast(x2); x3 = ex2_fast(x3);
        sum0 = fma_f2(pack_f2(x0, x1), one, sum0);
        sum1 = fma_f2(pack_f2(x2, x3), one, sum1);
        r[e >> 1] = pack_bf(x0, x1);                  // the first half of r takes the packed weights
        r[(e >> 1) + 1] = pack_bf(x2, x3);
      }
      float a0, a1, a2, a3;
      unpack_f2(sum0, a0, a1);
      unpack_f2(sum1, a2, a3);
      l += (a0 + a1) + (a2 + a3);
      if (j > 0 && !mbar_wait_warp(o_full, (j - 1) & 1)) { fail = 16; break; }     // P_{j-1} has been read
#pragma unroll
      for (int g = 0; g < TK / 8; g++)
        sts_v4(p_s + (uint32_t)(g >> 3) * TILE_BYTES + (uint32_t)row * 128u + (uint32_t)(((g & 7) ^ (row & 7)) << 4), r[4 * g], r[4 * g + 1],
               r[4 * g + 2], r[4 * g + 3]);
      tc_fence_before();
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(p_full);
    }
    if (!fail && !mbar_wait_warp(o_full, (nt - 1) & 1)) fail = 16;
    if (fail) {
      if (lane == 0) set_status(p.status, fail);
    } else {
      tc_fence_after();
      const int t = q0 + row;
      const float inv = 1.f / l;
      uint32_t r[DH];
      tc_ld32_issue(tm_o + lane_off, r);
      tc_ld32_issue(tm_o + lane_off + 32, r + 32);
      tc_ld_wait(r);
      tc_ld_wait(r + 32);
      if (t < p.T) {
        bf16_t* out = p.o + ((long long)b * p.T + t) * d + h * DH;
#pragma unroll
        for (int g = 0; g < DH / 8; g++) {
          float v[8];
#pragma unroll
          for (int e = 0; e < 8; e++) v[e] = __uint_as_float(r[8 * g + e]) * inv;
          *reinterpret_cast<uint4*>(out + 8 * g) = make_uint4(pack_bf(v[0], v[1]), pack_bf(v[2], v[3]), pack_bf(v[4], v[5]), pack_bf(v[6], v[7]));
        }
        p.lse[((long long)b * p.H + h) * p.T + t] = (m_ref + log2f(l)) * 0.6931471805599453f;
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 4) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(256u) : "memory");
  }
}


// ------------------------------------------------------------------------------------------------
// backward.  Both kernels: 8 softmax warps (two per TMEM lane quarter, each takes 32 of the 64
// columns of a sub-tile) and one warp that issues TMA and MMA.  The walk goes over sub-tiles of 64
// keys (dQ kernel) or 64 queries (dK/dV kernel), so that the score, dP and gradient accumulators
// take 256 TMEM columns and two CTAs share an SM: one CTA's softmax work hides the other's MMA and
// barrier latencies.  The gradient accumulators stay in tensor memory over the whole walk (no
// rescaling is needed: the probabilities are recomputed from the final log-sum-exp).
// ------------------------------------------------------------------------------------------------
constexpr int BW_THREADS = 288;
constexpr int TW = 64;                                   // sub-tile width
constexpr uint32_t SUB_BYTES = TW * DH * 2;              // a [64, 64] bf16 sub-tile: 8 KB
constexpr int NST_Q = 3;                                 // K/V sub-tile stages of the dQ kernel
constexpr int NST_KV = 2;                                // Q/dO sub-tile stages of the dK/dV kernel

__device__ __forceinline__ void softmax_bar() { asm volatile("bar.sync 1, 256;" ::: "memory"); }

// dot product of one swizzled 128-byte row (64 bf16) of two K-major tiles
__device__ __forceinline__ float row_dot64(const uint8_t* ta, const uint8_t* tb, int row) {
  float d0 = 0.f, d1 = 0.f;
#pragma unroll
  for (int c = 0; c < 8; c++) {
    const int off = row * 128 + ((c ^ (row & 7)) << 4);
    const uint4 qa = *reinterpret_cast<const uint4*>(ta + off), qb = *reinterpret_cast<const uint4*>(tb + off);
    const uint32_t x[4] = {qa.x, qa.y, qa.z, qa.w}, y[4] = {qb.x, qb.y, qb.z, qb.w};
#pragma unroll
    for (int j = 0; j < 4; j++) {
      d0 = fmaf(__uint_as_float(x[j] << 16), __uint_as_float(y[j] << 16), d0);
      d1 = fmaf(__uint_as_float(x[j] & 0xffff0000u), __uint_as_float(y[j] & 0xffff0000u), d1);
    }
  }
  return d0 + d1;
}

// dQ (and delta): one CTA per (query tile of 128, head, sequence), key sub-tiles of 64 from 0 up to the tile's last query.
//   delta[q] = sum_c dO[q,c] O[q,c]  (from the dO and O tiles in shared memory; also written out for the dK/dV kernel)
//   S = Q K^T, dP = dO V^T (both operands K-major);  dS = P (.) (dP - delta), P = exp(S scale - lse)
//   dQ += dS K   (A = dS [q, key] K-major from shared memory, B = K [key, dh] MN-major), times scale at the end
__global__ void __launch_bounds__(BW_THREADS, 2)
attn_bwd_q_tc_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_kv,
                     const __grid_constant__ CUtensorMap map_do, const __grid_constant__ CUtensorMap map_o,
                     const __grid_constant__ AttnArgs p) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t base = smem_u32(smem_raw);
  const uint32_t q_s = base, do_s = q_s + TILE_BYTES, kv_s = do_s + TILE_BYTES, ds_s = kv_s + NST_Q * 2 * SUB_BYTES;
  const uint32_t bar = ds_s + TILE_BYTES;
  const uint32_t q_full = bar, kv_full0 = bar + 8, kv_empty0 = kv_full0 + 8 * NST_Q, sdp_full = kv_empty0 + 8 * NST_Q, ds_full = sdp_full + 8,
                 ds_free = ds_full + 8, acc_full = ds_free + 8, sdp_free = acc_full + 8, tmem_slot = sdp_free + 8;
  volatile uint32_t* tmem_slot_ptr = reinterpret_cast<volatile uint32_t*>(smem_raw + (tmem_slot - base));

  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // (warp: known to be uniform)
  const AttnPlace at = attn_place(blockIdx.x, p.H, p.batch);
  const int qt = (p.T - 1) / TQ - at.tile, h = at.head, b = at.seq;
  const int d = p.H * DH;
  const int q0 = qt * TQ;
  const int nsub = min(2 * (qt + 1), (p.T + TW - 1) / TW);    // key sub-tiles that hold a key <= the tile's last query
  int st0 = status_peek(p.status);
  if (threadIdx.x == 0 && (base & 1023u)) { set_status(p.status, 10); st0 = 10; }

  if (threadIdx.x == 0) {
    mbar_init(q_full, 1);
    for (int s = 0; s < NST_Q; s++) { mbar_init(kv_full0 + 8 * s, 1); mbar_init(kv_empty0 + 8 * s, 1); }
    mbar_init(sdp_full, 1);
    mbar_init(ds_full, 8);
    mbar_init(ds_free, 1);
    mbar_init(acc_full, 1);
    mbar_init(sdp_free, 8);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 8) {
    if (lane == 0) {
      asm volatile("prefetch.tensormap [%0];" ::"l"(&map_q) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"(&map_kv) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"(&map_do) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"(&map_o) : "memory");
    }
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tmem_slot), "r"(256u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  pdl_wait();
  const bool dead = __syncthreads_or(st0 != 0) != 0;
  tc_fence_after();
  const uint32_t tmem = *tmem_slot_ptr;
  const uint32_t tm_s = tmem, tm_dp = tmem + 64, tm_dq = tmem + 128;

  if (dead) {
  } else if (warp == 8) {
    // the whole warp walks through the steps, one elected lane issues
    const int row0 = b * p.T;
    auto load_kv = [&](int j) {
      const int s = j % NST_Q;
      const uint32_t full = kv_full0 + 8 * s, dst = kv_s + s * 2 * SUB_BYTES;
      if (elect_one()) {
        mbar_expect_tx(full, 2 * SUB_BYTES);
        tma_load_2d(dst, &map_kv, d + h * DH, row0 + j * TW, full);
        tma_load_2d(dst + SUB_BYTES, &map_kv, 2 * d + h * DH, row0 + j * TW, full);
      }
    };
    if (elect_one()) {
      mbar_expect_tx(q_full, 3 * TILE_BYTES);
      tma_load_2d(q_s, &map_q, h * DH, row0 + q0, q_full);
      tma_load_2d(do_s, &map_do, h * DH, row0 + q0, q_full);
      tma_load_2d(ds_s, &map_o, h * DH, row0 + q0, q_full);      // the O tile: read once for delta, then this buffer holds dS
    }
    for (int j = 0; j < NST_Q && j < nsub; j++) load_kv(j);
    const uint32_t id_s = idesc_of(TW, false, false), id_q = idesc_of(DH, false, true);
    int fail = mbar_wait_warp(q_full, 0) ? 0 : 21;
    // S_j and dP_j are issued as soon as those of j-1 have been read into registers, in front of dQ += dS_{j-1} K_{j-1}
    for (int j = 0; j <= nsub && fail == 0; j++) {
      if (j < nsub) {
        const int s = j % NST_Q;
        const uint32_t kj = kv_s + s * 2 * SUB_BYTES, vj = kj + SUB_BYTES;
        if (!mbar_wait_warp(kv_full0 + 8 * s, (j / NST_Q) & 1)) { fail = 22; break; }
        if (j > 0 && !mbar_wait_warp(sdp_free, (j - 1) & 1)) { fail = 29; break; }
        tc_fence_after();
#pragma unroll
        for (int kk = 0; kk < DH / 16; kk++) tc_mma_warp(tm_s, desc_k(q_s, kk), desc_k(kj, kk), id_s, kk > 0 ? 1u : 0u);
#pragma unroll
        for (int kk = 0; kk < DH / 16; kk++) tc_mma_warp(tm_dp, desc_k(do_s, kk), desc_k(vj, kk), id_s, kk > 0 ? 1u : 0u);
        tc_commit_warp<1>(sdp_full);
      }
      if (j > 0) {
        const int i = j - 1, si = i % NST_Q;
        const uint32_t ki = kv_s + si * 2 * SUB_BYTES;
        if (!mbar_wait_warp(ds_full, i & 1)) { fail = 23; break; }
        tc_fence_after();
#pragma unroll
        for (int kk = 0; kk < TW / 16; kk++) tc_mma_warp(tm_dq, desc_k(ds_s, kk), desc_mn(ki, kk, SUB_BYTES), id_q, (i > 0 || kk > 0) ? 1u : 0u);
        tc_commit_warp<1>(ds_free);
        tc_commit_warp<1>(kv_empty0 + 8 * si);
        if (i + NST_Q < nsub) {     // the freed stage takes the sub-tile NST_Q further on
          if (!mbar_wait_warp(kv_empty0 + 8 * si, (i / NST_Q) & 1)) { fail = 24; break; }
          load_kv(i + NST_Q);
        }
      }
    }
    tc_commit_warp<1>(acc_full);        // fires in any case, so that the softmax warps do not wait for their limit
    if (fail) {
      if (lane == 0) set_status(p.status, fail);
      const long long t0 = clock64();
      while (clock64() - t0 < 2000000LL) {}
    }
    pdl_trigger();
  } else {
    const int quarter = warp & 3, half = warp >> 2;
    const int row = quarter * 32 + lane;
    const uint32_t lane_off = (uint32_t)(quarter * 32) << 16;
    const int t = q0 + row;
    const bool row_ok = t < p.T;
    const long long stat = ((long long)b * p.H + h) * p.T + t;
    const float lse2 = row_ok ? p.lse[stat] * LOG2E : 0.f;
    bool ok = true;
    float dl = 0.f;
    {   // delta of this thread's row from the dO and O tiles
      bool w = mbar_wait(q_full, 0);
      if (!w) set_status(p.status, 28);
      w = __all_sync(0xffffffffu, w);
      if (w) {
        dl = row_dot64(smem_raw + (do_s - base), smem_raw + (ds_s - base), row);
        if (half == 0 && row_ok) p.delta[stat] = dl;
      } else {
        ok = false;
      }
      softmax_bar();              // every row of the O tile has been read: the buffer may now take dS
    }
    for (int j = 0; j < nsub && ok; j++) {
      bool w = mbar_wait(sdp_full, j & 1);
      if (!w) set_status(p.status, 25);
      w = __all_sync(0xffffffffu, w);
      if (!w) { ok = false; break; }
      tc_fence_after();
      const int col0 = half * 32;
      const int kcol = j * TW + col0 - q0;                      // key index minus query index = kcol + e - row
      const bool maskable = j * TW + TW - 1 > q0;              // some key of the sub-tile lies beyond some query
      uint32_t rs[32], rp[32];
      tc_ld32_issue(tm_s + lane_off + col0, rs);
      tc_ld32_issue(tm_dp + lane_off + col0, rp);
      tc_ld_wait(rs);
      tc_ld_wait(rp);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(sdp_free);
      float ds[32];
      const f32x2 sc = pack_f2(p.scale_log2, p.scale_log2), nl = pack_f2(-lse2, -lse2), nd = pack_f2(-dl, -dl), one = pack_f2(1.f, 1.f);
#pragma unroll
      for (int e = 0; e < 32; e += 2) {
        float x0, x1;
        unpack_f2(fma_f2(pack_f2(__uint_as_float(rs[e]), __uint_as_float(rs[e + 1])), sc, nl), x0, x1);
        x0 = ex2_fast(x0); x1 = ex2_fast(x1);
        const f32x2 g = fma_f2(pack_f2(__uint_as_float(rp[e]), __uint_as_float(rp[e + 1])), one, nd);
        unpack_f2(mul_f2(pack_f2(x0, x1), g), ds[e], ds[e + 1]);
      }
      if (maskable) {
#pragma unroll
        for (int e = 0; e < 32; e++)
          if (kcol + e > row) ds[e] = 0.f;
      }
      if (j > 0) {                  // the previous sub-tile's dQ MMAs must have read dS before it is overwritten
        bool f = mbar_wait(ds_free, (j - 1) & 1);
        if (!f) set_status(p.status, 26);
        f = __all_sync(0xffffffffu, f);
        if (!f) { ok = false; break; }
      }
      store_p32(ds_s, row, col0, ds);
      tc_fence_before();
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(ds_full);
    }
    if (ok) {
      bool w = mbar_wait(acc_full, 0);
      if (!w) set_status(p.status, 27);
      w = __all_sync(0xffffffffu, w);
      if (w) {
        tc_fence_after();
        uint32_t r[32];
        tc_ld32(tm_dq + lane_off + half * 32, r);
        if (row_ok) {
          bf16_t* out = p.dqkv + ((long long)b * p.T + t) * (3 * d) + h * DH + half * 32;
#pragma unroll
          for (int g = 0; g < 4; g++) {
            uint4 q;
            q.x = pack_bf(__uint_as_float(r[8 * g]) * p.scale, __uint_as_float(r[8 * g + 1]) * p.scale);
            q.y = pack_bf(__uint_as_float(r[8 * g + 2]) * p.scale, __uint_as_float(r[8 * g + 3]) * p.scale);
            q.z = pack_bf(__uint_as_float(r[8 * g + 4]) * p.scale, __uint_as_float(r[8 * g + 5]) * p.scale);
            q.w = pack_bf(__uint_as_float(r[8 * g + 6]) * p.scale, __uint_as_float(r[8 * g + 7]) * p.scale);
            *reinterpret_cast<uint4*>(out + 8 * g) = q;
          }
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 8) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(256u) : "memory");
  }
}

// dK, dV: one CTA per (key tile of 128, head, sequence), query sub-tiles of 64 from the tile's first key to the end of
// the sequence.  Everything is computed transposed, so that a softmax thread owns a KEY row:
//   S^T = K Q^T, dP^T = V dO^T (both operands K-major);  P^T = exp(S^T scale - lse[q]),  dS^T = P^T (.) (dP^T - delta[q])
//   dV += P^T dO   (A = P^T [key, q] K-major from shared memory, B = dO [q, dh] MN-major)
//   dK += dS^T Q   (A = dS^T,                                   B = Q  [q, dh] MN-major), times scale at the end
__global__ void __launch_bounds__(BW_THREADS, 2)
attn_bwd_kv_tc_kernel(const __grid_constant__ CUtensorMap map_kv, const __grid_constant__ CUtensorMap map_q,
                      const __grid_constant__ CUtensorMap map_do, const __grid_constant__ AttnArgs p) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t base = smem_u32(smem_raw);
  const uint32_t k_s = base, v_s = k_s + TILE_BYTES, qdo_s = v_s + TILE_BYTES, pt_s = qdo_s + NST_KV * 2 * SUB_BYTES, dst_s = pt_s + TILE_BYTES;
  const uint32_t vec_s = dst_s + TILE_BYTES;              // lse (log2 units) and delta of each softmax warp's queries: 8 x 2 x 32 floats
  const uint32_t bar = vec_s + 2048;
  const uint32_t kv_full = bar, qdo_full0 = bar + 8, qdo_empty0 = qdo_full0 + 8 * NST_KV, sdp_full = qdo_empty0 + 8 * NST_KV,
                 pds_full = sdp_full + 8, pds_free = pds_full + 8, acc_full = pds_free + 8, sdp_free = acc_full + 8, tmem_slot = sdp_free + 8;
  volatile uint32_t* tmem_slot_ptr = reinterpret_cast<volatile uint32_t*>(smem_raw + (tmem_slot - base));

  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // (warp: known to be uniform)
  const AttnPlace at = attn_place(blockIdx.x, p.H, p.batch);
  const int kt = at.tile, h = at.head, b = at.seq;         // key tile 0 has the longest walk and comes first
  const int d = p.H * DH;
  const int k0 = kt * TK;
  const int first = 2 * kt, n = (p.T + TW - 1) / TW - first;      // query sub-tiles first .. first+n-1 (n >= 1: k0 < T)
  int st0 = status_peek(p.status);
  if (threadIdx.x == 0 && (base & 1023u)) { set_status(p.status, 10); st0 = 10; }

  if (threadIdx.x == 0) {
    mbar_init(kv_full, 1);
    for (int s = 0; s < NST_KV; s++) { mbar_init(qdo_full0 + 8 * s, 1); mbar_init(qdo_empty0 + 8 * s, 1); }
    mbar_init(sdp_full, 1);
    mbar_init(pds_full, 8);
    mbar_init(pds_free, 1);
    mbar_init(acc_full, 1);
    mbar_init(sdp_free, 8);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 8) {
    if (lane == 0) {
      asm volatile("prefetch.tensormap [%0];" ::"l"(&map_kv) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"(&map_q) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"(&map_do) : "memory");
    }
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tmem_slot), "r"(256u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  pdl_wait();
  const bool dead = __syncthreads_or(st0 != 0) != 0;
  tc_fence_after();
  const uint32_t tmem = *tmem_slot_ptr;
  const uint32_t tm_s = tmem, tm_dp = tmem + 64, tm_dv = tmem + 128, tm_dk = tmem + 192;

  if (dead) {
  } else if (warp == 8) {
    // the whole warp walks through the steps, one elected lane issues
    const int row0 = b * p.T;
    auto load_qdo = [&](int ii) {
      const int s = ii % NST_KV;
      const uint32_t full = qdo_full0 + 8 * s, dst = qdo_s + s * 2 * SUB_BYTES;
      if (elect_one()) {
        mbar_expect_tx(full, 2 * SUB_BYTES);
        tma_load_2d(dst, &map_q, h * DH, row0 + (first + ii) * TW, full);
        tma_load_2d(dst + SUB_BYTES, &map_do, h * DH, row0 + (first + ii) * TW, full);
      }
    };
    if (elect_one()) {
      mbar_expect_tx(kv_full, 2 * TILE_BYTES);
      tma_load_2d(k_s, &map_kv, d + h * DH, row0 + k0, kv_full);
      tma_load_2d(v_s, &map_kv, 2 * d + h * DH, row0 + k0, kv_full);
    }
    for (int ii = 0; ii < NST_KV && ii < n; ii++) load_qdo(ii);
    const uint32_t id_s = idesc_of(TW, false, false), id_g = idesc_of(DH, false, true);
    int fail = mbar_wait_warp(kv_full, 0) ? 0 : 31;
    // S^T_i and dP^T_i are issued as soon as those of i-1 have been read into registers, in front of the gradients of i-1
    for (int ii = 0; ii <= n && fail == 0; ii++) {
      if (ii < n) {
        const int s = ii % NST_KV;
        const uint32_t qi = qdo_s + s * 2 * SUB_BYTES, doi = qi + SUB_BYTES;
        if (!mbar_wait_warp(qdo_full0 + 8 * s, (ii / NST_KV) & 1)) { fail = 32; break; }
        if (ii > 0 && !mbar_wait_warp(sdp_free, (ii - 1) & 1)) { fail = 38; break; }
        tc_fence_after();
#pragma unroll
        for (int kk = 0; kk < DH / 16; kk++) tc_mma_warp(tm_s, desc_k(k_s, kk), desc_k(qi, kk), id_s, kk > 0 ? 1u : 0u);
#pragma unroll
        for (int kk = 0; kk < DH / 16; kk++) tc_mma_warp(tm_dp, desc_k(v_s, kk), desc_k(doi, kk), id_s, kk > 0 ? 1u : 0u);
        tc_commit_warp<1>(sdp_full);
      }
      if (ii > 0) {
        const int i = ii - 1, si = i % NST_KV;
        const uint32_t qi = qdo_s + si * 2 * SUB_BYTES, doi = qi + SUB_BYTES;
        if (!mbar_wait_warp(pds_full, i & 1)) { fail = 33; break; }
        tc_fence_after();
#pragma unroll
        for (int kk = 0; kk < TW / 16; kk++) tc_mma_warp(tm_dv, desc_k(pt_s, kk), desc_mn(doi, kk, SUB_BYTES), id_g, (i > 0 || kk > 0) ? 1u : 0u);
#pragma unroll
        for (int kk = 0; kk < TW / 16; kk++) tc_mma_warp(tm_dk, desc_k(dst_s, kk), desc_mn(qi, kk, SUB_BYTES), id_g, (i > 0 || kk > 0) ? 1u : 0u);
        tc_commit_warp<1>(pds_free);
        tc_commit_warp<1>(qdo_empty0 + 8 * si);
        if (i + NST_KV < n) {
          if (!mbar_wait_warp(qdo_empty0 + 8 * si, (i / NST_KV) & 1)) { fail = 34; break; }
          load_qdo(i + NST_KV);
        }
      }
    }
    tc_commit_warp<1>(acc_full);
    if (fail) {
      if (lane == 0) set_status(p.status, fail);
      const long long t0 = clock64();
      while (clock64() - t0 < 2000000LL) {}
    }
    pdl_trigger();
  } else {
    const int quarter = warp & 3, half = warp >> 2;
    const int row = quarter * 32 + lane;                   // key row of the tile
    const uint32_t lane_off = (uint32_t)(quarter * 32) << 16;
    const int col0 = half * 32;
    float* vs = reinterpret_cast<float*>(smem_raw + (vec_s - base)) + warp * 64;
    bool ok = true;
    // log-sum-exp (in log2 units) and delta of the warp's 32 queries of a sub-tile, both negated; -inf marks a query
    // past the sequence.  Each lane fetches one query's pair a sub-tile ahead; the warp reads them back from its own
    // 64 floats of shared memory, so that no two warps have to meet.
    const long long stat0 = ((long long)b * p.H + h) * p.T;
    float next_l, next_d;
    auto fetch = [&](int ii) {
      const int t = (first + ii) * TW + col0 + lane;
      const bool in = ii < n && t < p.T;
      next_l = in ? -p.lse[stat0 + t] * LOG2E : -INFINITY;
      next_d = in ? -p.delta[stat0 + t] : 0.f;
    };
    fetch(0);
    for (int ii = 0; ii < n && ok; ii++) {
      const int q0 = (first + ii) * TW;
      __syncwarp();                 // the previous sub-tile's values have been read
      vs[lane] = next_l;
      vs[32 + lane] = next_d;
      __syncwarp();
      fetch(ii + 1);
      bool w = mbar_wait(sdp_full, ii & 1);
      if (!w) set_status(p.status, 35);
      w = __all_sync(0xffffffffu, w);
      if (!w) { ok = false; break; }
      tc_fence_after();
      const int qcol = q0 + col0 - k0;                      // query index minus key index = qcol + e - row
      const bool maskable = q0 < k0 + TK - 1;              // some query of the sub-tile lies before some key
      uint32_t rs[32], rp[32];
      tc_ld32_issue(tm_s + lane_off + col0, rs);
      tc_ld32_issue(tm_dp + lane_off + col0, rp);
      tc_ld_wait(rs);
      tc_ld_wait(rp);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(sdp_free);
      if (maskable) {
#pragma unroll
        for (int e = 0; e < 32; e++)
          if (qcol + e < row) rs[e] = 0xff800000u;          // -inf
      }
      // P^T and dS^T, packed in place: the first halves of rs and rp
      const f32x2 sc = pack_f2(p.scale_log2, p.scale_log2), one = pack_f2(1.f, 1.f);
#pragma unroll
      for (int e = 0; e < 32; e += 4) {
        const float4 l4 = *reinterpret_cast<const float4*>(vs + e), d4 = *reinterpret_cast<const float4*>(vs + 32 + e);
        const float lq[4] = {l4.x, l4.y, l4.z, l4.w}, dq[4] = {d4.x, d4.y, d4.z, d4.w};
#pragma unroll
        for (int q = 0; q < 4; q += 2) {
          float x0, x1, g0, g1;
          // (s scale - lse: exp2(-inf) = 0 past the sequence)
          unpack_f2(fma_f2(pack_f2(__uint_as_float(rs[e + q]), __uint_as_float(rs[e + q + 1])), sc, pack_f2(lq[q], lq[q + 1])), x0, x1);
          x0 = ex2_fast(x0); x1 = ex2_fast(x1);
          const f32x2 g = fma_f2(pack_f2(__uint_as_float(rp[e + q]), __uint_as_float(rp[e + q + 1])), one, pack_f2(dq[q], dq[q + 1]));
          unpack_f2(mul_f2(pack_f2(x0, x1), g), g0, g1);
          rs[(e + q) >> 1] = pack_bf(x0, x1);
          rp[(e + q) >> 1] = pack_bf(g0, g1);
        }
      }
      if (ii > 0) {                 // the previous sub-tile's MMAs must have read P^T and dS^T before they are overwritten
        bool f = mbar_wait(pds_free, (ii - 1) & 1);
        if (!f) set_status(p.status, 36);
        f = __all_sync(0xffffffffu, f);
        if (!f) { ok = false; break; }
      }
      const uint32_t prow = pt_s + (uint32_t)row * 128u, drow = dst_s + (uint32_t)row * 128u;
#pragma unroll
      for (int g = 0; g < 4; g++) {
        const uint32_t piece = (uint32_t)((((col0 >> 3) + g) ^ (row & 7)) << 4);
        sts_v4(prow + piece, rs[4 * g], rs[4 * g + 1], rs[4 * g + 2], rs[4 * g + 3]);
        sts_v4(drow + piece, rp[4 * g], rp[4 * g + 1], rp[4 * g + 2], rp[4 * g + 3]);
      }
      tc_fence_before();
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(pds_full);
    }
    if (ok) {
      bool w = mbar_wait(acc_full, 0);
      if (!w) set_status(p.status, 37);
      w = __all_sync(0xffffffffu, w);
      if (w) {
        tc_fence_after();
        const int t = k0 + row;
        uint32_t rv[32], rk[32];
        tc_ld32_issue(tm_dv + lane_off + half * 32, rv);
        tc_ld32_issue(tm_dk + lane_off + half * 32, rk);
        tc_ld_wait(rv);
        tc_ld_wait(rk);
        if (t < p.T) {
          bf16_t* out = p.dqkv + ((long long)b * p.T + t) * (3 * d) + h * DH + half * 32;
#pragma unroll
          for (int g = 0; g < 4; g++) {
            uint4 q;
            q.x = pack_bf(__uint_as_float(rk[8 * g]) * p.scale, __uint_as_float(rk[8 * g + 1]) * p.scale);
            q.y = pack_bf(__uint_as_float(rk[8 * g + 2]) * p.scale, __uint_as_float(rk[8 * g + 3]) * p.scale);
            q.z = pack_bf(__uint_as_float(rk[8 * g + 4]) * p.scale, __uint_as_float(rk[8 * g + 5]) * p.scale);
            q.w = pack_bf(__uint_as_float(rk[8 * g + 6]) * p.scale, __uint_as_float(rk[8 * g + 7]) * p.scale);
            *reinterpret_cast<uint4*>(out + d + 8 * g) = q;
            q.x = pack_bf(__uint_as_float(rv[8 * g]), __uint_as_float(rv[8 * g + 1]));
            q.y = pack_bf(__uint_as_float(rv[8 * g + 2]), __uint_as_float(rv[8 * g + 3]));
            q.z = pack_bf(__uint_as_float(rv[8 * g + 4]), __uint_as_float(rv[8 * g + 5]));
            q.w = pack_bf(__uint_as_float(rv[8 * g + 6]), __uint_as_float(rv[8 * g + 7]));
            *reinterpret_cast<uint4*>(out + 2 * d + 8 * g) = q;
          }
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 8) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(256u) : "memory");
  }
}

constexpr size_t BWD_Q_SMEM = TILE_BYTES * 3 + NST_Q * 2 * SUB_BYTES + 128;                 // 96.1 KB: two CTAs per SM
constexpr size_t BWD_KV_SMEM = TILE_BYTES * 4 + NST_KV * 2 * SUB_BYTES + 2048 + 128;       // 98.1 KB: two CTAs per SM

constexpr size_t FWD_SMEM = TILE_BYTES * 5 + P_BYTES + 128;   // two CTAs per SM: 2 x (112.1 KB + 1 KB reserved) <= 228 KB

}  // namespace

bool attention_tc_supported(int dh, int d, const void* qkv, const void* o) {
  return dh == DH && d % DH == 0 && ((reinterpret_cast<uintptr_t>(qkv) | reinterpret_cast<uintptr_t>(o)) & 15) == 0;
}

cudaError_t attention_fwd_tc(const void* qkv, void* o, float* lse, int batch, int T, int heads, int* status, cudaStream_t s) {
  const int d = heads * DH;
  CUtensorMap map;
  if (!tc_encode_rows_bf16(&map, qkv, 3LL * d, (long long)batch * T, 3LL * d, TQ)) return cudaErrorInvalidValue;
  static std::atomic<bool> attr_set[64];
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) dev = 0;
  if (!attr_set[dev].load(std::memory_order_acquire)) {
    cudaError_t e = cudaFuncSetAttribute(attn_fwd_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FWD_SMEM);
    if (e != cudaSuccess) return e;
    attr_set[dev].store(true, std::memory_order_release);
  }
  AttnArgs a;
  a.T = T; a.H = heads; a.batch = batch;
  a.scale = 0.125f;
  a.scale_log2 = 0.125f * LOG2E;
  a.o = (bf16_t*)o; a.lse = lse; a.delta = nullptr; a.dqkv = nullptr; a.status = status;
  const long long grid = attn_blocks(heads, batch, (T + TQ - 1) / TQ);
  if (grid > ATTN_MAX_BLOCKS) return cudaErrorInvalidConfiguration;
  pdl_launch(attn_fwd_tc_kernel, (unsigned)grid, AT_THREADS, FWD_SMEM, s, map, a);
  return cudaGetLastError();
}

cudaError_t attention_bwd_tc(const void* qkv, const void* o, const void* dout, const float* lse, float* delta, void* dqkv, int batch,
                             int T, int heads, int* status, cudaStream_t s) {
  const int d = heads * DH;
  const long long rows = (long long)batch * T;
  CUtensorMap qkv128, qkv64, do128, do64, o128;        // the same matrices seen as tiles of 128 or 64 rows
  if (!tc_encode_rows_bf16(&qkv128, qkv, 3LL * d, rows, 3LL * d, 128) || !tc_encode_rows_bf16(&qkv64, qkv, 3LL * d, rows, 3LL * d, TW) ||
      !tc_encode_rows_bf16(&do128, dout, d, rows, d, 128) || !tc_encode_rows_bf16(&do64, dout, d, rows, d, TW) ||
      !tc_encode_rows_bf16(&o128, o, d, rows, d, 128))
    return cudaErrorInvalidValue;
  static std::atomic<bool> attr_set[64];
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) dev = 0;
  if (!attr_set[dev].load(std::memory_order_acquire)) {
    cudaError_t e = cudaFuncSetAttribute(attn_bwd_q_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)BWD_Q_SMEM);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(attn_bwd_kv_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)BWD_KV_SMEM);
    if (e != cudaSuccess) return e;
    attr_set[dev].store(true, std::memory_order_release);
  }
  AttnArgs a;
  a.T = T; a.H = heads; a.batch = batch;
  a.scale = 0.125f;
  a.scale_log2 = 0.125f * LOG2E;
  a.o = nullptr; a.lse = const_cast<float*>(lse); a.delta = delta; a.dqkv = (bf16_t*)dqkv; a.status = status;
  const long long grid = attn_blocks(heads, batch, (T + TQ - 1) / TQ);
  if (grid > ATTN_MAX_BLOCKS) return cudaErrorInvalidConfiguration;
  // the dQ kernel also produces delta, which the dK/dV kernel reads: it runs first
  pdl_launch(attn_bwd_q_tc_kernel, (unsigned)grid, BW_THREADS, BWD_Q_SMEM, s, qkv128, qkv64, do128, o128, a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  pdl_launch(attn_bwd_kv_tc_kernel, (unsigned)grid, BW_THREADS, BWD_KV_SMEM, s, qkv128, qkv64, do64, a);
  return cudaGetLastError();
}

}  // namespace erase
