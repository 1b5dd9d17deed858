// tcgen05 / TMEM / TMA GEMM for sm_100a.  See gemm_tc.cuh for the contract.
//
// Persistent kernel: one CTA per SM walks over 128 x BN output tiles (one split of K each when
// split-K is on); 320 threads:
//   warp 0      TMA producer: one elected lane fills a ring of STAGES shared-memory stages,
//               each holding a 128 x 64 slab of A and a BN x 64 slab of B (bf16, 128-byte swizzle)
//   warp 1      allocates TMEM (two accumulators), then one elected lane issues tcgen05.mma
//               (M=128, N=BN, K=16), four per stage, commits each stage back to the producer and
//               each finished accumulator to the epilogue through mbarriers
//   warps 2..9  epilogue: wait for an accumulator, read their TMEM lane quarter with tcgen05.ld
//               (two warps per quarter, half of the columns each), apply the fused epilogue,
//               store to global memory, hand the accumulator back; this overlaps the next
//               tile's main loop
// Every mbarrier wait is bounded by a clock limit; on expiry the kernel records a status word,
// skips the rest of its work, still frees its TMEM and returns.
//
// Two more kernels further down share these roles and helpers: tc_gemm_pair_kernel (two CTAs of a
// cluster on one tile 256 rows high, tcgen05 cta_group::2) and tc_wgrad_kernel (up to four small weight gradients with
// their bias gradients in one launch, clusters sharing a tile's contraction).
#include "gemm_tc.cuh"
#include "launch.cuh"
#include "tc_ptx.cuh"
#include "ew_math.cuh"

#include <cuda.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <atomic>

namespace erase {

namespace {

constexpr int BM = 128;
constexpr int BK = 64;          // bf16 elements = 128 bytes = one swizzle row
constexpr int UMMA_K = 16;
// Operand stages and output staging buffers per epilogue warp of the single-CTA kernel.  128-wide tiles: five stages
// and one buffer against four and two: 4096 x 512 MLP step 1180 -> 1130 us; a sixth stage gives another 2 us there,
// but its 226 KB keep other streams' kernels off the SM (680-wide MLP 493 -> 513 us, CTR 1040 -> 1060 us).
__host__ __device__ constexpr int stages_for(int bn) { return bn == 256 ? 3 : (bn == 128 ? 5 : 6); }
constexpr uint32_t EPI_BIAS_BYTES = 512;              // up to 128 bias floats per epilogue warp
constexpr int EPI_WARPS = 8;                       // two per TMEM lane quarter, each takes half the columns
constexpr int TC_THREADS = 32 * (2 + EPI_WARPS);
constexpr uint32_t EPI_STAGE_BYTES = 8192;             // two buffers of 32 rows x 128 bytes per epilogue warp
struct TcArgs {
  int M, N, K;
  void* C;
  long long ldc;
  int c_f32;
  int splits;
  float* ws;
  Epilogue epi;
  int* status;
  long long* dbg;  // optional: clock64 stamps of CTA 0's first tile (development aid), else null
  int tma_c;       // C (or the split-K partials) leaves through shared memory + TMA store
  int bias_add;    // the plain epilogue adds a bias (and, with relu, clamps at zero)
  int relu;
  int aux_mode;    // fused epilogues with auxiliary operands: AUX_* of the one that arrives by TMA
  int aux2_mode;   // ... and of the second one, read straight from global memory (0: none)
  const __nv_bfloat16* aux2;
  int stages;      // CTA-pair kernel: operand stages, of
  uint32_t stage_bytes;
  int wide;        // GELU epilogue, and the second output of a post_mul: rows are 32-byte aligned
  int bn;          // CTA-pair kernel: tile width, 128, 192 or 256
  int* sched;      // {next tile counter, finished CTAs}, zero between launches; null = static round-robin
  float* xcol_out; // CTA-pair kernel: the sum of the products with B's columns N .. N + 2 goes here (GemmArgs::xcol_out)
  int xcol_ones;   // ... or with the constant tile behind map_x
  int xcol_wide;   // those columns lie in the last column tile; else in 16-wide column tiles of their own
};

// Epilogues.  PLAIN: identity, bias, bias + ReLU (the split-K partials and every weight gradient are the
// identity).  CE: local softmax head.  The fused ones work on 32 rows x 64 columns at a time in two 4 KB
// shared-memory buffers per warp:
//   AUX, AUX2  residual / DCN-v2 multiplier / ReLU derivative: the (first) auxiliary tile arrives by TMA in the
//              buffer the result leaves from, so each thread replaces a 16-byte piece in place
//   GELU       u = bf16(acc + bias) and gelu(u): the forward keeps both (the backward needs u).  No staging: a lane
//              owns a row and stores 32-byte sectors, which needs no wait for a buffer (two TMA stores per chunk
//              through shared memory: 4096 x 512 MLP step 1180 against 1175 us, larger LM 23.0 against 22.7 ms; 16
//              epilogue warps instead of 8: 1138 against 1129 us)
//   DGELU      bf16(acc) * gelu'(u) with u arriving by TMA, in place
// The GELU pair replaces a separate elementwise pass over the matrix and rounds exactly as that pass did (GELU of
// the bf16 pre-activation; derivative times the bf16 gradient), which the dual-list kernel still runs.  Measured
// (GEMM + pass, then fused): 32768 x 4096 x 1024 forward 315 -> 250 us, dgrad 373 -> 240 us; 8192 x 3072 x 768
// forward 74 -> 57, dgrad 79 -> 60; 4096 x 2048 x 512 forward 31 -> 25, dgrad 32 -> 27.
enum { EPI_PLAIN = 0, EPI_CE = 1, EPI_AUX = 2, EPI_AUX2 = 3, EPI_GELU = 4, EPI_DGELU = 5 };
enum { AUX_NONE = 0, AUX_RES = 1, AUX_MUL = 2, AUX_DRELU = 3, AUX_POST = 4 };     // AUX_POST: Epilogue::post_mul
__host__ __device__ constexpr bool epi_fused(int epi) { return epi >= EPI_AUX; }
__host__ __device__ constexpr bool epi_by_tma(int epi) { return epi_fused(epi) && epi != EPI_GELU; }   // an auxiliary tile arrives in the buffer
__host__ __device__ constexpr int single_bufs(int bn, int epi) { return epi == EPI_GELU ? 0 : (epi_by_tma(epi) && bn == 256 ? 2 : 1); }

// 8 bf16 held in a 16-byte register quad -> floats
__device__ __forceinline__ void unpack8_bf16(uint4 q, float* out) {
  out[0] = __uint_as_float(q.x << 16); out[1] = __uint_as_float(q.x & 0xffff0000u);
  out[2] = __uint_as_float(q.y << 16); out[3] = __uint_as_float(q.y & 0xffff0000u);
  out[4] = __uint_as_float(q.z << 16); out[5] = __uint_as_float(q.z & 0xffff0000u);
  out[6] = __uint_as_float(q.w << 16); out[7] = __uint_as_float(q.w & 0xffff0000u);
}

__device__ __forceinline__ uint32_t pack2(float a, float b) {
  __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&h);
}
__device__ __forceinline__ void store8_bf16(__nv_bfloat16* p, int valid, bool vec, const float* v) {
  if (vec) {
    uint4 q;
    q.x = pack2(v[0], v[1]); q.y = pack2(v[2], v[3]); q.z = pack2(v[4], v[5]); q.w = pack2(v[6], v[7]);
    *reinterpret_cast<uint4*>(p) = q;
  } else {
#pragma unroll
    for (int j = 0; j < 8; j++)
      if (j < valid) p[j] = __float2bfloat16_rn(v[j]);
  }
}


struct F8 { float v[8]; };

// Direct global store of 8 finished values (used when the output cannot go through TMA).
__device__ __forceinline__ void direct_store8(const TcArgs& p, F8 in, int row, int n, int split) {
  const float* v = in.v;
  const int valid = min(8, p.N - n);
  if (p.splits > 1 || p.c_f32) {
    float* dst = p.splits > 1 ? p.ws + (long long)split * p.M * p.N + (long long)row * p.N + n
                              : (float*)p.C + (long long)row * p.ldc + n;
    if (valid == 8 && ((reinterpret_cast<uintptr_t>(dst) & 15) == 0)) {
      reinterpret_cast<float4*>(dst)[0] = make_float4(v[0], v[1], v[2], v[3]);
      reinterpret_cast<float4*>(dst)[1] = make_float4(v[4], v[5], v[6], v[7]);
    } else {
#pragma unroll
      for (int j = 0; j < 8; j++) if (j < valid) dst[j] = v[j];
    }
  } else {
    __nv_bfloat16* dst = (__nv_bfloat16*)p.C + (long long)row * p.ldc + n;
    store8_bf16(dst, valid, valid == 8 && ((reinterpret_cast<uintptr_t>(dst) & 15) == 0), v);
  }
}

__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, uint32_t src, int x, int y) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];"
               ::"l"(map), "r"(x), "r"(y), "r"(src) : "memory");
}
__device__ __forceinline__ void tma_store_3d(const CUtensorMap* map, uint32_t src, int x, int y, int z) {
  asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%1, %2, %3}], [%4];"
               ::"l"(map), "r"(x), "r"(y), "r"(z), "r"(src) : "memory");
}
__device__ __forceinline__ void tma_store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// all but the most recent store of this thread have finished reading their shared-memory source
__device__ __forceinline__ void tma_store_wait_read1() { asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory"); }

__device__ __forceinline__ uint4 ld_shared_v4(uint32_t addr) {
  uint4 q;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(q.x), "=r"(q.y), "=r"(q.z), "=r"(q.w) : "r"(addr) : "memory");
  return q;
}
__device__ __forceinline__ uint4 pack8(const float* q) {
  return make_uint4(pack2(q[0], q[1]), pack2(q[2], q[3]), pack2(q[4], q[5]), pack2(q[6], q[7]));
}

// One epilogue warp's 4 KB buffers (up to two), the barriers its auxiliary tiles arrive on, and how many have arrived.
struct WarpEpi {
  uint32_t stage0, auxbar, taken;
  bool store_pending;       // lane 0: TMA stores may still be reading the buffers
};

// Requests the auxiliary tiles of this warp's part of the next output tile (at most two 64-column chunks, one per
// buffer): called before the warp starts waiting for the accumulator, so the round trip hides behind the MMAs.
template <int EPI, int NB>
__device__ __forceinline__ void fused_prefetch(const CUtensorMap* map_x, WarpEpi& w, int x0, int y0, int ncols, int lane) {
  if (!epi_by_tma(EPI) || lane != 0) return;
  if (w.store_pending) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
  for (int c = 0; c < ncols; c += 64) {
    const uint32_t buf = NB == 2 ? (w.taken + (c >> 6)) & 1 : 0;
    mbar_expect_tx(w.auxbar + 8 * buf, 4096);
    tma_load_2d(w.stage0 + buf * 4096, map_x, x0 + c, y0, w.auxbar + 8 * buf);
  }
}

// 16 finished columns of one row straight to global memory: a lane owns a row, so they are a full 32-byte sector
__device__ __forceinline__ void store_row16(const TcArgs& p, __nv_bfloat16* base, long long ld, int row, int col, int col_end, const uint4 (&q)[2]) {
  if (row >= p.M) return;
  __nv_bfloat16* dst = base + (long long)row * ld + col;
  if (p.wide && col + 16 <= col_end) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "r"(q[0].x), "r"(q[0].y), "r"(q[0].z), "r"(q[0].w),
                 "r"(q[1].x), "r"(q[1].y), "r"(q[1].z), "r"(q[1].w) : "memory");
    return;
  }
#pragma unroll
  for (int g = 0; g < 2; g++)
    if (col + 8 * g < col_end) *reinterpret_cast<uint4*>(dst + 8 * g) = q[g];
}
__device__ __forceinline__ void apply_aux(int mode, float* v, const float* t) {
#pragma unroll
  for (int j = 0; j < 8; j++) v[j] = mode == AUX_RES ? v[j] + t[j] : (mode == AUX_MUL ? v[j] * t[j] : (t[j] > 0.f ? v[j] : 0.f));
}

// This warp's 32 rows x ncols columns of a finished accumulator (tmem: address of its first column) through a
// fused epilogue.  x0, y0: first column and row in the matrix; row: this lane's; bias_s: the slice for x0.
// False if an auxiliary tile did not arrive in time.
template <int EPI, int NB>
__device__ __forceinline__ bool fused_tile(const TcArgs& p, const CUtensorMap* map_c, const CUtensorMap* map_x, WarpEpi& w, uint32_t tmem,
                                           int x0, int y0, int ncols, int row, const float* bias_s, int lane) {
#pragma unroll 1
  for (int c = 0; c < ncols; c += 64) {
    uint32_t buf = 0;
    if (EPI != EPI_GELU) {
      buf = NB == 2 ? w.taken & 1 : 0;
      const bool ok = mbar_wait(w.auxbar + 8 * buf, NB == 2 ? (w.taken >> 1) & 1 : w.taken & 1);
      if (!__all_sync(0xffffffffu, ok)) return false;
      w.taken++;
    }
    const uint32_t my_row = w.stage0 + buf * 4096 + lane * 128;
#pragma unroll 1
    for (int h = 0; h < 64; h += 32) {
      const int cc = c + h;
      if (cc >= ncols) break;     // warp-uniform
      uint4 second[4];
      if (EPI == EPI_AUX2) {
        const __nv_bfloat16* src = p.aux2 + (long long)row * p.epi.ld_aux + x0 + cc;
#pragma unroll
        for (int g8 = 0; g8 < 4; g8++)
          second[g8] = row < p.M && cc + 8 * g8 < ncols ? *reinterpret_cast<const uint4*>(src + 8 * g8) : make_uint4(0u, 0u, 0u, 0u);
      }
      uint32_t r[32];
      tc_ld32_issue(tmem + (uint32_t)cc, r);
      tc_ld_wait(r);
      if (EPI != EPI_DGELU && p.epi.bias) {
#pragma unroll
        for (int g4 = 0; g4 < 8; g4++) {
          const float4 b = *reinterpret_cast<const float4*>(bias_s + cc + g4 * 4);
          r[4 * g4 + 0] = __float_as_uint(__uint_as_float(r[4 * g4 + 0]) + b.x);
          r[4 * g4 + 1] = __float_as_uint(__uint_as_float(r[4 * g4 + 1]) + b.y);
          r[4 * g4 + 2] = __float_as_uint(__uint_as_float(r[4 * g4 + 2]) + b.z);
          r[4 * g4 + 3] = __float_as_uint(__uint_as_float(r[4 * g4 + 3]) + b.w);
        }
      }
      constexpr int W = 16;       // columns worked on side by side
#pragma unroll
      for (int w0 = 0; w0 < 32; w0 += W) {
        float v[W], t[W];
        uint32_t piece[W / 8];
        uint4 uq[W / 8], uq2[W / 8];
#pragma unroll
        for (int j = 0; j < W; j++) v[j] = __uint_as_float(r[w0 + j]);
#pragma unroll
        for (int g = 0; g < W / 8; g++) {
          piece[g] = my_row + (((((h + w0) >> 3) + g) ^ (lane & 7)) << 4);
          if (EPI != EPI_GELU) unpack8_bf16(ld_shared_v4(piece[g]), t + 8 * g);
        }
        if (EPI == EPI_GELU || EPI == EPI_DGELU) {
#pragma unroll
          for (int g = 0; g < W / 8; g++) {        // a pass over the stored matrix would read bf16
            const uint4 u = pack8(v + 8 * g);
            if (EPI == EPI_GELU) uq[g] = u;
            unpack8_bf16(u, v + 8 * g);
          }
          if (EPI == EPI_GELU) store_row16(p, (__nv_bfloat16*)p.epi.pre_out, p.epi.ld_aux, row, x0 + cc + w0, x0 + ncols, uq);
          if (EPI == EPI_GELU) gelu_bf16_n<W>(v);
          else dgelu_bf16_n<W>(t, v);
        } else {      // relu, then multiplier, residual, ReLU derivative -- in this order
#pragma unroll
          for (int g = 0; g < W / 8; g++) {
            float* q = v + 8 * g;
            if (p.relu) {
#pragma unroll
              for (int j = 0; j < 8; j++) q[j] = fmaxf(q[j], 0.f);
            }
            if (EPI == EPI_AUX2) {
              float t2[8];
              unpack8_bf16(second[(w0 >> 3) + g], t2);
              if (p.aux2_mode == AUX_MUL) apply_aux(AUX_MUL, q, t2);
              apply_aux(AUX_RES, q, t + 8 * g);
              if (p.aux2_mode == AUX_DRELU) apply_aux(AUX_DRELU, q, t2);
              if (p.aux2_mode == AUX_POST) {
                apply_aux(AUX_MUL, t2, q);
                if (p.epi.post_out) {
                  uq2[g] = pack8(t2);
                } else {
#pragma unroll
                  for (int j = 0; j < 8; j++) q[j] = t2[j];
                }
              }
            } else {
              apply_aux(p.aux_mode, q, t + 8 * g);
            }
          }
        }
#pragma unroll
        for (int g = 0; g < W / 8; g++) {
          const uint4 o = pack8(v + 8 * g);
          if (EPI == EPI_GELU) uq[g] = o;
          else st_shared_v4(piece[g], o.x, o.y, o.z, o.w);
        }
        if (EPI == EPI_AUX2 && p.epi.post_out) store_row16(p, (__nv_bfloat16*)p.epi.post_out, p.epi.ld_aux, row, x0 + cc + w0, x0 + ncols, uq2);
        if (EPI == EPI_GELU) store_row16(p, (__nv_bfloat16*)p.C, p.ldc, row, x0 + cc + w0, x0 + ncols, uq);
      }
    }
    if (EPI == EPI_GELU) continue;
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncwarp();
    if (lane == 0) {
      tma_store_2d(map_c, w.stage0 + buf * 4096, x0 + c, y0);
      tma_store_commit();
      w.store_pending = true;
    }
  }
  return true;
}

// The plain and cross-entropy epilogues work on 32 x 32 pieces of this warp's part of a tile.  The TMEM load of the
// next piece is in flight while one is worked on, and a piece is finished in registers before the warp waits for the
// staging buffer it goes to: the read by the buffer's last TMA store hides behind that work.  One buffer per warp is
// then enough (two: within 1 % over 64 shapes).  With the cross-entropy's arithmetic on f32x2 pairs (before: a serial
// sum per row, the load and the store's read in the open) the head's forward takes, 4096 x 8192 x 256: 36.0 -> 27.6 us,
// where the identity takes 24.8 (its 200 MB through L2); 4096 x 16384 x 512: 73.5 -> 68.6; 8192 x 32768 x 768:
// 346 -> 330; 1407 x 5008 x 320: 14.3 -> 12.3.
template <typename F>
__device__ __forceinline__ void walk_pieces(uint32_t tmem, int ncols, bool empty_k, F piece) {
  uint32_t ra[32], rb[32];
  if (empty_k) {       // a trailing split with no K range: zeros
#pragma unroll 1
    for (int cc = 0; cc < ncols; cc += 32) {
#pragma unroll
      for (int j = 0; j < 32; j++) ra[j] = 0u;
      piece(ra, cc);
    }
    return;
  }
  tc_ld32_issue(tmem, ra);
#pragma unroll 1
  for (int cc = 0; cc < ncols; cc += 64) {
    tc_ld_wait(ra);
    if (cc + 32 < ncols) tc_ld32_issue(tmem + cc + 32, rb);
    piece(ra, cc);
    if (cc + 32 < ncols) {
      tc_ld_wait(rb);
      if (cc + 64 < ncols) tc_ld32_issue(tmem + cc + 64, ra);
      piece(rb, cc + 32);
    }
  }
}
// waits until the last TMA store has read the staging buffer
__device__ __forceinline__ void free_buffer(const WarpEpi& w, int lane) {
  if (lane == 0 && w.store_pending) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
  __syncwarp();
}
__device__ __forceinline__ void send_buffer(const TcArgs& p, const CUtensorMap* map_c, WarpEpi& w, int x, int y, int split, int lane) {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncwarp();
  if (lane == 0 && y < p.M) {
    if (p.splits > 1) tma_store_3d(map_c, w.stage0, x, y, split);
    else tma_store_2d(map_c, w.stage0, x, y);
    tma_store_commit();
    w.store_pending = true;
  }
}
// 32 finished bf16 columns of this lane's row (16 packed registers), columns cc .. cc + 31 of the warp's part
__device__ __forceinline__ void send_bf16(const TcArgs& p, const CUtensorMap* map_c, WarpEpi& w, const uint32_t (&q)[16], int x0, int y0, int cc, int ncols, int lane) {
  if ((cc & 63) == 0) free_buffer(w, lane);
#pragma unroll
  for (int g = 0; g < 4; g++)
    st_shared_v4(w.stage0 + lane * 128 + (((((cc & 63) >> 3) + g) ^ (lane & 7)) << 4), q[4 * g], q[4 * g + 1], q[4 * g + 2], q[4 * g + 3]);
  if ((cc & 63) == 32 || cc + 32 >= ncols) send_buffer(p, map_c, w, x0 + (cc & ~63), y0, 0, lane);
}

// The cross-entropy head's part of a tile: a logit becomes exp(logit - ref), ref: this row's, stored as bf16; the
// return value is this row's sum over the columns.  Columns past N contribute nothing.
__device__ __forceinline__ float ce_tile(const TcArgs& p, const CUtensorMap* map_c, WarpEpi& w, uint32_t tmem, int x0, int y0, int ncols,
                                         float ref, const float* bias_s, int lane) {
  const float ref2 = ref * 1.4426950408889634f;
  const f32x2 l2e = pack_f2(1.4426950408889634f, 1.4426950408889634f), nref = pack_f2(-ref2, -ref2);
  f32x2 sum0 = pack_f2(0.f, 0.f), sum1 = sum0;
  walk_pieces(tmem, ncols, false, [&](uint32_t (&r)[32], int cc) {
    if (cc + 32 > ncols) {
#pragma unroll
      for (int j = 0; j < 32; j++)
        if (cc + j >= ncols) r[j] = 0xff800000u;      // -inf
    }
    uint32_t q[16];
#pragma unroll
    for (int e = 0; e < 32; e += 4) {
      const float4 b = *reinterpret_cast<const float4*>(bias_s + cc + e);
      float v0, v1, v2, v3;
      unpack_f2(fma_f2(add_f2(pack_f2(__uint_as_float(r[e]), __uint_as_float(r[e + 1])), pack_f2(b.x, b.y)), l2e, nref), v0, v1);
      unpack_f2(fma_f2(add_f2(pack_f2(__uint_as_float(r[e + 2]), __uint_as_float(r[e + 3])), pack_f2(b.z, b.w)), l2e, nref), v2, v3);
      v0 = ex2_fast(v0); v1 = ex2_fast(v1); v2 = ex2_fast(v2); v3 = ex2_fast(v3);
      sum0 = add_f2(sum0, pack_f2(v0, v1));
      sum1 = add_f2(sum1, pack_f2(v2, v3));
      q[e / 2] = pack2(v0, v1);
      q[e / 2 + 1] = pack2(v2, v3);
    }
    send_bf16(p, map_c, w, q, x0, y0, cc, ncols, lane);
  });
  float a0, a1, a2, a3;
  unpack_f2(sum0, a0, a1);
  unpack_f2(sum1, a2, a3);
  return (a0 + a1) + (a2 + a3);
}

// identity, bias, bias + ReLU; bf16 or fp32 output or fp32 split-K partials
__device__ __forceinline__ void plain_tile(const TcArgs& p, const CUtensorMap* map_c, WarpEpi& w, uint32_t tmem, int x0, int y0, int ncols, int row,
                                           int split, bool empty_k, const float* bias_s, int lane) {
  const bool f32 = p.splits > 1 || p.c_f32;
  walk_pieces(tmem, ncols, empty_k, [&](uint32_t (&r)[32], int cc) {
    if (p.bias_add) {
#pragma unroll
      for (int e = 0; e < 32; e += 4) {
        const float4 b = *reinterpret_cast<const float4*>(bias_s + cc + e);
        const float bb[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
        for (int j = 0; j < 4; j++) {
          float v = __uint_as_float(r[e + j]) + bb[j];
          if (p.relu) v = fmaxf(v, 0.f);
          r[e + j] = __float_as_uint(v);
        }
      }
    }
    if (!p.tma_c) {
#pragma unroll
      for (int g = 0; g < 4; g++) {
        F8 f;
#pragma unroll
        for (int j = 0; j < 8; j++) f.v[j] = __uint_as_float(r[8 * g + j]);
        if (row < p.M && cc + 8 * g < ncols) direct_store8(p, f, row, x0 + cc + 8 * g, split);
      }
    } else if (f32) {        // 32 floats per row
      free_buffer(w, lane);
#pragma unroll
      for (int g = 0; g < 8; g++) st_shared_v4(w.stage0 + lane * 128 + ((g ^ (lane & 7)) << 4), r[4 * g], r[4 * g + 1], r[4 * g + 2], r[4 * g + 3]);
      send_buffer(p, map_c, w, x0 + cc, y0, split, lane);
    } else {
      uint32_t q[16];
#pragma unroll
      for (int e = 0; e < 16; e++) q[e] = pack2(__uint_as_float(r[2 * e]), __uint_as_float(r[2 * e + 1]));
      send_bf16(p, map_c, w, q, x0, y0, cc, ncols, lane);
    }
  });
}

// Tile order: splits outermost; inside a split, bands of 8 column tiles, and inside a band m
// outer / n inner.  The ~148 tiles in flight at any time then cover about 18 row tiles x 8
// column tiles, so each operand slab fetched from HBM is reused out of L2 by its neighbours.
__device__ __forceinline__ void tile_coords(int t, int tiles_m, int tiles_n, int& mt, int& nt, int& split) {
  const int per_split = tiles_m * tiles_n;
  split = t / per_split;
  const int r = t - split * per_split;
  const int band = r / (8 * tiles_m);
  const int n_first = band * 8;
  const int width = min(8, tiles_n - n_first);
  const int rr = r - band * 8 * tiles_m;
  mt = rr / width;
  nt = n_first + rr - mt * width;
}

// Persistent kernel: CTA c works on tiles c, c + gridDim.x, ... in the order of tile_coords.
// Each epilogue is an instantiation of its own: the loop body's size is part of what bounds it (instruction
// fetch: it runs once per tile and warp).
// EPI_CE (local softmax cross-entropy head, forward): the epilogue turns a logit l into
// exp(l - ref[row]) with a per-row reference known before the GEMM, stores that (bf16) instead of
// the logit and leaves, per row and group of CPW columns, the fp32 sum of the unrounded
// exponentials in ce_psum[row][group]: the head's loss and gradient then need no pass over logits.
template <int BN, bool A_MN, bool B_MN, int EPI>
__global__ void __launch_bounds__(TC_THREADS, 1)
tc_gemm_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
               const __grid_constant__ CUtensorMap map_c, const __grid_constant__ CUtensorMap map_x,
               const __grid_constant__ TcArgs p) {
  constexpr bool CE = EPI == EPI_CE;
  constexpr bool FUSED = epi_fused(EPI);
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  constexpr uint32_t A_BYTES = BM * BK * 2;
  constexpr uint32_t B_BYTES = BN * BK * 2;
  constexpr uint32_t STAGE_BYTES = A_BYTES + B_BYTES;
  constexpr uint32_t TMEM_COLS = 2 * BN;            // two accumulators: epilogue(i) overlaps mainloop(i+1)
  constexpr int CPW = BN >= 128 ? BN / 2 : 64;      // tile columns per epilogue warp (two warps per lane quarter)
  constexpr int STAGES = stages_for(BN), EPI_BUFS = single_bufs(BN, EPI), NB = EPI_BUFS == 2 ? 2 : 1;
  constexpr uint32_t EPI_BYTES = 4096u * EPI_BUFS, BIAS_BYTES = 2u * 2u * CPW * 4u;   // two column halves x two tile parities

  const uint32_t smem_base = smem_u32(smem_raw);       // no static shared memory: the window's start, 1024-byte aligned
  const uint32_t epi_base = smem_base + STAGES * STAGE_BYTES;          // EPI_WARPS x EPI_BUFS 4 KB staging buffers
  const uint32_t bias_base = epi_base + EPI_WARPS * EPI_BYTES;    // CPW floats of bias for each column half and tile parity
  const uint32_t bar_base = bias_base + BIAS_BYTES;
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (STAGES + s); };
  auto tfull_bar = [&](int a) { return bar_base + 8u * (2 * STAGES + a); };
  auto tempty_bar = [&](int a) { return bar_base + 8u * (2 * STAGES + 2 + a); };
  // tile queue: the producer publishes the tiles this CTA works on (dynamic scheduling) to the MMA
  // and epilogue warps through a 4-entry ring
  auto tq_full = [&](int i) { return bar_base + 8u * (2 * STAGES + 6 + i); };
  auto tq_empty = [&](int i) { return bar_base + 8u * (2 * STAGES + 10 + i); };
  uint8_t* gen_base = smem_raw + (smem_base - smem_u32(smem_raw));
  volatile uint32_t* tmem_slot_ptr =
      reinterpret_cast<volatile uint32_t*>(gen_base + STAGES * STAGE_BYTES + (EPI_WARPS * EPI_BYTES + BIAS_BYTES) + 8u * (2 * STAGES + 4));
  volatile int* tile_ring =
      reinterpret_cast<volatile int*>(gen_base + STAGES * STAGE_BYTES + (EPI_WARPS * EPI_BYTES + BIAS_BYTES) + 8u * (2 * STAGES + 14));
  const uint32_t tmem_slot = bar_base + 8u * (2 * STAGES + 4);
  auto aux_bar = [&](int w, int b) { return bar_base + 8u * (2 * STAGES + 16 + 2 * w + b); };

  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // (warp: known to be uniform)
  int st0 = status_peek(p.status);
  if (threadIdx.x == 0 && (smem_base & 1023u) != 0) { atomicExch(p.status, 9); st0 = 9; }     // never expected
#ifdef ERASE_DEV_AIDS   // clock stamps of CTA 0's first tile: compiled in only with -DERASE_DEV_AIDS
  const bool dbg = p.dbg != nullptr && blockIdx.x == 0;
#else
  constexpr bool dbg = false;
#endif
  if (dbg && threadIdx.x == 0) p.dbg[0] = clock64();
  if (threadIdx.x == 32) {   // descriptor fetches overlap the barrier and TMEM set-up
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_a) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_b) : "memory");
    if (EPI != EPI_GELU && p.tma_c) asm volatile("prefetch.tensormap [%0];" ::"l"(&map_c) : "memory");
    if (epi_by_tma(EPI)) asm volatile("prefetch.tensormap [%0];" ::"l"(&map_x) : "memory");
  }
  const int tiles_m = (p.M + BM - 1) / BM, tiles_n = (p.N + BN - 1) / BN;
  const int total = tiles_m * tiles_n * p.splits;
  const int kchunk = (((p.K + p.splits - 1) / p.splits) + BK - 1) / BK * BK;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; s++) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    for (int a = 0; a < 2; a++) {
      mbar_init(tfull_bar(a), 1);
      mbar_init(tempty_bar(a), EPI_WARPS);
    }
    for (int i = 0; i < 4; i++) {
      mbar_init(tq_full(i), 1);
      mbar_init(tq_empty(i), 1 + EPI_WARPS);
    }
    if (FUSED)
      for (int i = 0; i < 2 * EPI_WARPS; i++) mbar_init(aux_bar(0, i), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tmem_slot), "r"(TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  pdl_wait();
  const bool dead = __syncthreads_or(st0 != 0) != 0;
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot_ptr;
  if (dbg && threadIdx.x == 0) p.dbg[1] = clock64();

  if (dead) {
    // the step is already void: do nothing but free TMEM below
  } else if (warp == 0) {
    // ------------------------------ TMA producer (the whole warp, one elected lane issues) ------------------------------
    uint32_t s = 0, ph = 0, slot = 0;
    bool ok = true;
    int t = (int)blockIdx.x < total ? (int)blockIdx.x : -1;
    while (ok) {
      // publish the tile (or the end marker -1) to the other roles
      if (!mbar_wait_warp(tq_empty(slot & 3), ((slot >> 2) & 1) ^ 1)) { if (lane == 0) atomicExch(p.status, 5); ok = false; break; }
      int next = t + (int)gridDim.x;
      if (lane == 0) {
        tile_ring[slot & 3] = t;
        mbar_arrive(tq_full(slot & 3));
        // claim the next tile now: the atomic's latency hides behind this tile's loads
        if (p.sched && t >= 0) next = (int)gridDim.x + atomicAdd(p.sched, 1);
      }
      slot++;
      if (t < 0) break;
      int mt, nt, split;
      tile_coords(t, tiles_m, tiles_n, mt, nt, split);
      const int m0 = mt * BM, n0 = nt * BN;
      const int kbeg = split * kchunk, kend = min(p.K, kbeg + kchunk);
      const int num_kb = kend > kbeg ? (kend - kbeg + BK - 1) / BK : 0;
      for (int kb = 0; kb < num_kb; kb++) {
        if (!mbar_wait_warp(empty_bar(s), ph ^ 1)) { if (lane == 0) atomicExch(p.status, 1); ok = false; break; }
        const uint32_t a_dst = smem_base + s * STAGE_BYTES;
        const uint32_t b_dst = a_dst + A_BYTES;
        const int k0 = kbeg + kb * BK;
        if (elect_one()) {
          mbar_expect_tx(full_bar(s), STAGE_BYTES);
          if (!A_MN) {
            tma_load_2d(a_dst, &map_a, k0, m0, full_bar(s));
          } else {
#pragma unroll
            for (int a = 0; a < BM / 64; a++) tma_load_2d(a_dst + a * (BK * 128), &map_a, m0 + a * 64, k0, full_bar(s));
          }
          if (!B_MN) {
            tma_load_2d(b_dst, &map_b, k0, n0, full_bar(s));
          } else {
#pragma unroll
            for (int a = 0; a < BN / 64; a++) tma_load_2d(b_dst + a * (BK * 128), &map_b, n0 + a * 64, k0, full_bar(s));
          }
        }
        if (++s == STAGES) { s = 0; ph ^= 1; }
      }
      next = __shfl_sync(0xffffffffu, next, 0);
      t = next < total ? next : -1;
    }
    if (!ok) {  // give copies already in flight time to land before the CTA's shared memory is released
      const long long t0 = clock64();
      while (clock64() - t0 < 2000000LL) {}
    }
    pdl_trigger();
  } else if (warp == 1) {
    // ------------------------------ MMA issuer (the whole warp, one elected lane issues) ------------------------------
    // instruction descriptor: fp32 accumulate, bf16 x bf16, majors, N>>3 at bit 17, M>>4 at bit 24
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((A_MN ? 1u : 0u) << 15) | ((B_MN ? 1u : 0u) << 16) |
                           ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
    // K-major: rows of 128 bytes, 8-row groups 1024 bytes apart; a K step of 16 elements is
    //          32 bytes inside the swizzled row.
    // MN-major: 64-element (128-byte) runs along M/N, one per K index; 8 K rows form a
    //          1024-byte group (stride offset), the next 64 M/N elements sit BK*128 bytes
    //          further (leading offset); a K step of 16 is 16 rows = 2048 bytes.
    const uint64_t ad0 = smem_desc(smem_base, A_MN ? BK * 128 : 16, 1024), bd0 = smem_desc(smem_base + A_BYTES, B_MN ? BK * 128 : 16, 1024);
    constexpr int STEP_A = (A_MN ? UMMA_K * 128 : UMMA_K * 2) >> 4, STEP_B = (B_MN ? UMMA_K * 128 : UMMA_K * 2) >> 4;
    uint32_t s = 0, ph = 0, lt = 0;
    bool ok = true;
    for (;; lt++) {
      if (!mbar_wait_warp(tq_full(lt & 3), (lt >> 2) & 1)) { if (lane == 0) atomicExch(p.status, 6); break; }
      const int t = __shfl_sync(0xffffffffu, tile_ring[lt & 3], 0);
      if (lane == 0) mbar_arrive(tq_empty(lt & 3));
      if (t < 0 || !ok) break;
      const int split = t / (tiles_m * tiles_n);
      const int kbeg = split * kchunk, kend = min(p.K, kbeg + kchunk);
      const int num_kb = kend > kbeg ? (kend - kbeg + BK - 1) / BK : 0;
      const uint32_t ab = lt & 1, aph = (lt >> 1) & 1;
      if (!mbar_wait_warp(tempty_bar(ab), aph ^ 1)) { if (lane == 0) atomicExch(p.status, 4); ok = false; break; }
      tc_fence_after();
      const uint32_t tmem_d = tmem_base + ab * BN;
      for (int kb = 0; kb < num_kb; kb++) {
        if (!mbar_wait_warp(full_bar(s), ph)) { if (lane == 0) atomicExch(p.status, 2); ok = false; break; }
        tc_fence_after();
        const uint32_t off = s * (STAGE_BYTES >> 4);
        tc_mma_block<1, STEP_A, STEP_B>(tmem_d, ad0 + off, bd0 + off, idesc, kb > 0, empty_bar(s));   // the stage may be refilled once they have read it
        if (++s == STAGES) { s = 0; ph ^= 1; }
      }
      tc_commit_warp<1>(tfull_bar(ab));   // accumulator ab complete (also fires when the loop bailed out)
    }
  } else {
    // ------------------------------ epilogue ------------------------------
    // A warp owns 32 rows (its TMEM lane quarter) x half of the tile's columns (all of 64), in
    // 32-column pieces.  Finished values go to a 4 KB staging buffer in shared memory (one 128-byte
    // row per lane, 16-byte pieces XOR-swizzled with the row so that writes are conflict-free and
    // match the tensor map's 128-byte swizzle) and leave with one TMA store per 128-byte-wide
    // box, which also clips the M and N tails.  The GELU epilogue, and outputs that cannot be
    // described to TMA (unaligned leading dimension), are stored directly.
    const int ew = warp - 2;
    const int q = warp & 3;                       // TMEM lane quarter this warp may read
    const int cbeg = (ew / 4) * CPW;              // first tile column of this warp
    const bool active = cbeg < BN;                // BN = 64: only one warp per quarter has columns
    const uint32_t stage0 = epi_base + ew * EPI_BYTES;   // EPI_BUFS buffers of 4 KB
    WarpEpi we{stage0, aux_bar(ew, 0), 0u, false};
    uint32_t lt = 0;
    for (;; lt++) {
      int t = -1;
      if (lane == 0) {
        if (mbar_wait(tq_full(lt & 3), (lt >> 2) & 1)) {
          t = tile_ring[lt & 3];
          mbar_arrive(tq_empty(lt & 3));
        } else {
          atomicExch(p.status, 7);
        }
      }
      t = __shfl_sync(0xffffffffu, t, 0);
      if (t < 0) break;
      int mt, nt, split;
      tile_coords(t, tiles_m, tiles_n, mt, nt, split);
      const int m0 = mt * BM, n0 = nt * BN;
      const int kbeg = split * kchunk, kend = min(p.K, kbeg + kchunk);
      const bool empty_k = kend <= kbeg;          // a trailing split with no K range: partial sum is zero
      const uint32_t ab = lt & 1, aph = (lt >> 1) & 1;
      // bias: fetched into registers now, written to the slice the four warps of a column half share once the
      // accumulator is complete (see the CTA-pair kernel for why that needs no barrier)
      const bool need_bias = p.epi.bias != nullptr && p.splits == 1 && active;
      float* bias_s = reinterpret_cast<float*>(gen_base + STAGES * STAGE_BYTES + EPI_WARPS * EPI_BYTES) + ((ew / 4) * 2 + (lt & 1)) * CPW;
      float4 bias_pre = make_float4(0.f, 0.f, 0.f, 0.f);
      if (need_bias) {
        const int n = lane * 4 < CPW ? n0 + cbeg + lane * 4 : p.N;
        const float* bp = p.epi.bias + n;
        if (n + 4 <= p.N) {
          bias_pre = *reinterpret_cast<const float4*>(bp);
        } else {
          if (n < p.N) bias_pre.x = bp[0];
          if (n + 1 < p.N) bias_pre.y = bp[1];
          if (n + 2 < p.N) bias_pre.z = bp[2];
        }
      }
      const int row = m0 + q * 32 + lane;
      const bool row_ok = row < p.M;
      const float ce_ref = CE && row_ok ? p.epi.ce_ref[row] : 0.f;      // (in front of the wait, like the bias)
      const int fx = n0 + cbeg, fy = m0 + q * 32, fcols = active && fy < p.M ? min(CPW, p.N - fx) : 0;   // fused epilogues: this warp's part
      if (FUSED) fused_prefetch<EPI, NB>(&map_x, we, fx, fy, fcols, lane);
      bool ok = mbar_wait(tfull_bar(ab), aph);
      if (!ok) atomicExch(p.status, 3);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      if (dbg && lt == 0 && threadIdx.x == 64) p.dbg[5] = clock64();
      if (need_bias) {
        if (lane * 4 < CPW) *reinterpret_cast<float4*>(bias_s + lane * 4) = bias_pre;
        __syncwarp();
      }
      if (FUSED) {
        if (!fused_tile<EPI, NB>(p, &map_c, &map_x, we, tmem_base + ab * BN + ((uint32_t)(q * 32) << 16) + (uint32_t)cbeg, fx, fy, fcols, row,
                             bias_s, lane)) {
          if (lane == 0) atomicExch(p.status, 10);
          break;
        }
      } else if (CE) {
        if (fcols > 0) {
          const float sum = ce_tile(p, &map_c, we, tmem_base + ab * BN + ((uint32_t)(q * 32) << 16) + (uint32_t)cbeg, fx, fy, fcols, ce_ref, bias_s, lane);
          if (row_ok) p.epi.ce_psum[(long long)row * p.epi.ce_groups + fx / CPW] = sum;
        }
      } else if (fcols > 0) {
        plain_tile(p, &map_c, we, tmem_base + ab * BN + ((uint32_t)(q * 32) << 16) + (uint32_t)cbeg, fx, fy, fcols, row, split, empty_k, bias_s, lane);
      }
      // all TMEM reads of this warp are complete (tcgen05.wait::ld): hand the accumulator back
      if (dbg && lt == 0 && threadIdx.x == 64) p.dbg[12] = clock64();
      tc_fence_before();
      __syncwarp();
      if (dbg && lt == 0 && threadIdx.x == 64) p.dbg[13] = clock64();
      if (lane == 0) mbar_arrive(tempty_bar(ab));
      if (dbg && lt == 0 && threadIdx.x == 64) p.dbg[6] = clock64();
    }
    if (lane == 0 && we.store_pending) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");  // the buffers have been read; kernel completion covers the writes
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
  }
  if (p.sched && threadIdx.x == 0) {   // the CTA that finishes last leaves the scheduler words at zero
    __threadfence();
    if (atomicAdd(p.sched + 1, 1) == (int)gridDim.x - 1) {
      p.sched[0] = 0;
      p.sched[1] = 0;
      __threadfence();
    }
  }
  if (dbg && threadIdx.x == 0) p.dbg[7] = clock64();
}

// =================================================================================================
// CTA-pair kernel (tcgen05 cta_group::2): two CTAs of a cluster, on neighbouring SMs, share one
// output tile of 256 rows and 128, 192 or 256 columns (TcArgs::bn).  Each CTA stages its own 128
// rows of A and HALF of the B slab per K block; the pair's tensor cores read both halves, so at 256
// columns every SM moves 32 KB per K block through shared memory and L2 instead of the 48 KB of
// the single-CTA 128 x 256 tile -- which is what bounds the large GEMMs.  The leader CTA (cluster
// rank 0) issues the MMAs (M = 256, N = bn, K = 16) for both; the accumulator rows 0..127 land in
// the leader's TMEM, rows 128..255 in the peer's, and each CTA's epilogue warps drain their own.
//   full[s]    leader only: TMA bytes of BOTH CTAs' stage s have landed (both CTAs' copies signal it)
//   empty[s]   per CTA: the MMAs that read stage s are done (one commit, delivered to both CTAs)
//   tfull[a]   per CTA: accumulator a is complete (delivered to both CTAs)
//   tempty[a]  leader only: both CTAs' epilogue warps have drained accumulator a (the peer's warps
//              arrive on it through the cluster's shared-memory window)
// Tiles are assigned round-robin to clusters, in the order of tile_coords.  The output must be
// describable to TMA (all but GELU's leave through staged TMA stores).
constexpr int PAIR_BN = 256;        // the widest
// Plain and softmax epilogues: one staging buffer per epilogue warp, not two: the warp then waits for its previous store to have read the
// buffer before refilling it, which costs the epilogue-bound short contractions a few per cent when they run
// alone, but the CTA takes 194 KB of shared memory instead of 226 KB and other streams' small kernels find
// room beside it: under the overlapped schedule every configuration measured 0.5-1 % faster.
constexpr int PAIR_MAX_STAGES = 8;
// 4 KB output staging buffers per epilogue warp
__host__ __device__ constexpr int pair_epi_bufs(int epi) { return epi == EPI_GELU ? 0 : (epi_fused(epi) ? 2 : 1); }
constexpr uint32_t PAIR_BIAS_BYTES = 2u * 2u * (PAIR_BN / 2) * 4u;   // two column halves x two tile parities x 128 floats

__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t map_to_cta(uint32_t addr, uint32_t rank) {   // same offset in CTA `rank` of the cluster
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// copy into this CTA's shared memory; the byte count is credited to `bar`, which may be the peer's
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
      ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(bar)
      : "memory");
}
template <bool A_MN, bool B_MN, int EPI>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(TC_THREADS, 1)
tc_gemm_pair_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                    const __grid_constant__ CUtensorMap map_c, const __grid_constant__ CUtensorMap map_x,
                    const __grid_constant__ TcArgs p, const uint32_t tmem_cols) {
  constexpr bool CE = EPI == EPI_CE;
  constexpr bool FUSED = epi_fused(EPI);
  constexpr int EPI_BUFS = pair_epi_bufs(EPI), NB = EPI_BUFS == 2 ? 2 : 1;
  constexpr uint32_t EPI_BYTES = 4096u * EPI_BUFS;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const int BN = p.bn;
  constexpr int ACC_COLS = PAIR_BN;     // TMEM columns between the two accumulators
  constexpr int STAGES = PAIR_MAX_STAGES;     // barriers; p.stages of them are used
  const int stages = FUSED ? 5 : p.stages;
  constexpr uint32_t A_BYTES = BM * BK * 2;
  // (compile-time for the fused epilogues: with run-time values 4096 x 1680 x 1680 with multiplier and residual took
  // 24.6 us instead of 21.9, about the pace of MMAs issued from a single-lane branch; why is not known)
  const uint32_t stage_bytes = FUSED ? 2u * BM * BK * 2u : p.stage_bytes, epi_off = stages * stage_bytes;
  const int half0 = (BN / 2 + 63) / 64 * 64;   // columns of the first four epilogue warps (whole 64-column stores); the other four take the rest

  // The operand stages need a 1024-byte aligned base (128-byte swizzle); the kernel has no static shared
  // memory, so the dynamic array starts the CTA's window.  Should it ever not, the kernel reports it and works on nothing.
  const uint32_t smem_base = smem_u32(smem_raw);
  const uint32_t epi_base = smem_base + epi_off;
  const uint32_t bar_base = epi_base + EPI_WARPS * EPI_BYTES + PAIR_BIAS_BYTES;
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (STAGES + s); };
  auto tfull_bar = [&](int a) { return bar_base + 8u * (2 * STAGES + a); };
  auto tempty_bar = [&](int a) { return bar_base + 8u * (2 * STAGES + 2 + a); };
  uint8_t* gen_base = smem_raw + (smem_base - smem_u32(smem_raw));
  volatile uint32_t* tmem_slot_ptr =
      reinterpret_cast<volatile uint32_t*>(gen_base + epi_off + EPI_WARPS * EPI_BYTES + PAIR_BIAS_BYTES + 8u * (2 * STAGES + 4));
  const uint32_t tmem_slot = bar_base + 8u * (2 * STAGES + 4);
  auto aux_bar = [&](int w, int b) { return bar_base + 8u * (2 * STAGES + 8 + 2 * w + b); };

  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // (warp: known to be uniform)
  volatile int* dead_flag_ptr = reinterpret_cast<volatile int*>(gen_base + epi_off + EPI_WARPS * EPI_BYTES + PAIR_BIAS_BYTES + 8u * (2 * STAGES + 6));
  if (threadIdx.x == 0) {
    const bool misaligned = (smem_base & 1023u) != 0;
    if (misaligned) atomicExch(p.status, 9);
    *dead_flag_ptr = (misaligned || status_peek(p.status) != 0) ? 1 : 0;
  }
  const uint32_t rank = cluster_ctarank();
  const bool leader = rank == 0;
  const int cluster_id = blockIdx.x >> 1, n_clusters = gridDim.x >> 1;
  const int naccum = tmem_cols >= 2u * ACC_COLS ? 2 : 1;      // accumulators in TMEM (two: epilogue overlaps the next main loop)
  if (threadIdx.x == 32) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_a) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_b) : "memory");
    if (EPI != EPI_GELU) asm volatile("prefetch.tensormap [%0];" ::"l"(&map_c) : "memory");
    if (epi_by_tma(EPI)) asm volatile("prefetch.tensormap [%0];" ::"l"(&map_x) : "memory");
  }
  // xcol: behind the column tiles of C comes one narrow tile per row tile, at n = N, 16 wide; or (xwide: columns of B, where they fit)
  // the last column tile is up to 32 wider.  (Narrow tiles read A again, and with 74 pairs and rows of three tiles
  // and a narrow one, every second pair got all the full ones: 32768 x 768 x 8192 355 us, 313 in a wider last tile; 16384 x 512 x 4096
  // 67.5 and 65.7; 8192 x 256 x 4096 31 both.  16 wider instead of 32, with halves of 104 columns: 399.)
  const bool xcol = p.xcol_out != nullptr && !p.xcol_wide, xwide = p.xcol_out != nullptr && p.xcol_wide;
  const int tiles_n_main = (p.N + BN - 1) / BN;
  const int xcol_at = p.N - (tiles_n_main - 1) * BN;                  // place of column N in the last column tile, <= BN
  const int bn_last = xwide ? max(BN, (xcol_at + 16 + 31) / 32 * 32) : BN;      // and that tile's width: its halves start on 32-byte sectors
  const int tiles_m = (p.M + 2 * BM - 1) / (2 * BM), tiles_n = tiles_n_main + (xcol ? 1 : 0);
  constexpr int XCOL_N = 16;
  const int total = tiles_m * tiles_n * p.splits;
  const int kchunk = (((p.K + p.splits - 1) / p.splits) + BK - 1) / BK * BK;
  // The narrow tiles come behind their row tile's others, which then leave A in L2; or, if the others are not more than
  // the pairs, behind all of them: idle pairs take them (32768-deep 4096 x 1024: else six full tiles wait for a second round)
  const int narrow_last = xcol && tiles_m * tiles_n_main <= n_clusters ? tiles_m * tiles_n_main : total;
  auto coords = [&](int t, int& mt, int& nt, int& split) {
    if (t < narrow_last) {
      tile_coords(t, tiles_m, narrow_last < total ? tiles_n_main : tiles_n, mt, nt, split);
    } else {
      mt = t - narrow_last; nt = tiles_n_main; split = 0;
    }
  };

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; s++) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    for (int a = 0; a < 2; a++) {
      mbar_init(tfull_bar(a), 1);
      mbar_init(tempty_bar(a), 2 * EPI_WARPS);
    }
    if (FUSED)
      for (int i = 0; i < 2 * EPI_WARPS; i++) mbar_init(aux_bar(0, i), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {   // one warp of EACH CTA of the pair takes part in the allocation
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tmem_slot), "r"(tmem_cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  pdl_wait();
  __syncthreads();
  cluster_sync_all();      // the peer's barriers exist before anything is sent to them
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot_ptr;
#ifdef ERASE_DEV_AIDS
  if (p.dbg && threadIdx.x == 0 && cluster_id == 0) p.dbg[8 + rank] = (long long)tmem_base;
#endif
  int dead;   // both CTAs of the pair take the LEADER's reading, so that they skip (or work) together
  asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(dead) : "r"(map_to_cta(bar_base + 8u * (2 * STAGES + 6), 0)) : "memory");

  if (dead) {
    // the step is already void: do nothing but free TMEM below
  } else if (warp == 0) {
    // ---------------- TMA producer (both CTAs; the whole warp, one elected lane issues) ----------------
    uint32_t s = 0, ph = 0;
    bool ok = true;
    const uint32_t lfull0 = map_to_cta(full_bar(0), 0);
    for (int t = cluster_id; t < total && ok; t += n_clusters) {
      int mt, nt, split;
      coords(t, mt, nt, split);
      const int m0 = mt * 2 * BM + (int)rank * BM;        // this CTA's 128 rows of A
      const bool narrow = xcol && nt == tiles_n_main;
      const int width = nt == tiles_n_main - 1 ? bn_last : BN;
      const int nb0 = narrow ? p.N + (int)rank * (XCOL_N / 2) : nt * BN + (int)rank * (width / 2);     // this CTA's half of the tile's B columns
      const int kbeg = split * kchunk, kend = min(p.K, kbeg + kchunk);
      const int num_kb = kend > kbeg ? (kend - kbeg + BK - 1) / BK : 0;
      const int boxes = narrow ? 1 : (width / 2 + 63) / 64;                                         // MN-major B: 64-column boxes of this CTA's half
      const uint32_t tx = 2 * (A_BYTES + (B_MN ? boxes * (BK * 128u) : (uint32_t)(BN / 2) * (BK * 2u)));      // this CTA's bytes and the peer's
      for (int kb = 0; kb < num_kb; kb++) {
#ifdef ERASE_DEV_AIDS
        const long long w0 = clock64();
#endif
        if (!mbar_wait_warp(empty_bar(s), ph ^ 1)) { if (lane == 0) atomicExch(p.status, 1); ok = false; break; }
#ifdef ERASE_DEV_AIDS
        if (p.dbg && blockIdx.x == 0 && lane == 0) p.dbg[7] += clock64() - w0;      // producer: waiting for a free stage
#endif
        const uint32_t lfull = lfull0 + 8u * s;
        const uint32_t a_dst = smem_base + s * stage_bytes;
        const uint32_t b_dst = a_dst + A_BYTES;
        const int k0 = kbeg + kb * BK;
        if (elect_one()) {
          if (leader) mbar_expect_tx(full_bar(s), tx);
          if (!A_MN) {
            tma_load_2d_pair(a_dst, &map_a, k0, m0, lfull);
          } else {
#pragma unroll
            for (int a = 0; a < BM / 64; a++) tma_load_2d_pair(a_dst + a * (BK * 128), &map_a, m0 + a * 64, k0, lfull);
          }
          if (!B_MN) {
            tma_load_2d_pair(b_dst, &map_b, k0, nb0, lfull);
          } else {
            if (narrow && p.xcol_ones) tma_load_2d_pair(b_dst, &map_x, 0, 0, lfull);
            else tma_load_2d_pair(b_dst, &map_b, nb0, k0, lfull);
            if (boxes > 1) tma_load_2d_pair(b_dst + BK * 128, &map_b, nb0 + 64, k0, lfull);
          }
        }
        if (++s == (uint32_t)stages) { s = 0; ph ^= 1; }
      }
    }
    if (!ok) {  // give copies already in flight time to land before the CTA's shared memory is released
      const long long t0 = clock64();
      while (clock64() - t0 < 2000000LL) {}
    }
    pdl_trigger();
  } else if (warp == 1) {
    // ---------------- MMA issuer (leader CTA only; the whole warp, one elected lane issues) ----------------
    if (leader) {
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((A_MN ? 1u : 0u) << 15) | ((B_MN ? 1u : 0u) << 16) |
                             ((uint32_t)(BN >> 3) << 17) | ((uint32_t)((2 * BM) >> 4) << 24);
      // the same descriptors address this CTA's and the peer's shared memory (identical layout)
      const uint64_t ad0 = smem_desc(smem_base, A_MN ? BK * 128 : 16, 1024), bd0 = smem_desc(smem_base + A_BYTES, B_MN ? BK * 128 : 16, 1024);
      constexpr int STEP_A = (A_MN ? UMMA_K * 128 : UMMA_K * 2) >> 4, STEP_B = (B_MN ? UMMA_K * 128 : UMMA_K * 2) >> 4;
      uint32_t s = 0, ph = 0, lt = 0;
      bool ok = true;
      for (int t = cluster_id; t < total && ok; t += n_clusters, lt++) {
        int mt_, nt_, split;
        coords(t, mt_, nt_, split);
        const bool narrow = xcol && nt_ == tiles_n_main;
        const int width = narrow ? XCOL_N : (nt_ == tiles_n_main - 1 ? bn_last : BN);
        const uint32_t idesc_t = (idesc & ~(0x3Fu << 17)) | ((uint32_t)(width >> 3) << 17);
        const int kbeg = split * kchunk, kend = min(p.K, kbeg + kchunk);
        const int num_kb = kend > kbeg ? (kend - kbeg + BK - 1) / BK : 0;
        const uint32_t ab = naccum == 2 ? (lt & 1) : 0u, aph = naccum == 2 ? ((lt >> 1) & 1) : (lt & 1);
#ifdef ERASE_DEV_AIDS
        const bool acct = p.dbg && blockIdx.x == 0 && lane == 0;
        long long w0 = acct ? clock64() : 0;
        if (acct && lt == 0) p.dbg[0] = w0;
#endif
        if (!mbar_wait_warp(tempty_bar(ab), aph ^ 1)) { if (lane == 0) atomicExch(p.status, 4); ok = false; break; }
#ifdef ERASE_DEV_AIDS
        if (acct) { p.dbg[1] += clock64() - w0; p.dbg[10] += 1; }       // MMA warp: waiting for a drained accumulator
#endif
        tc_fence_after();
        const uint32_t tmem_d = tmem_base + ab * ACC_COLS;
        for (int kb = 0; kb < num_kb; kb++) {
#ifdef ERASE_DEV_AIDS
          w0 = acct ? clock64() : 0;
#endif
          if (!mbar_wait_warp(full_bar(s), ph)) { if (lane == 0) atomicExch(p.status, 2); ok = false; break; }
#ifdef ERASE_DEV_AIDS
          if (acct) { const long long w1 = clock64(); p.dbg[2] += w1 - w0; p.dbg[3] = w1; }   // MMA warp: waiting for operands
#endif
          tc_fence_after();
          const uint32_t off = s * (stage_bytes >> 4);
          tc_mma_block<2, STEP_A, STEP_B>(tmem_d, ad0 + off, bd0 + off, idesc_t, kb > 0, empty_bar(s));
          if (++s == (uint32_t)stages) { s = 0; ph ^= 1; }
        }
        tc_commit_warp<2>(tfull_bar(ab));
      }
    }
  } else {
    // ------------------------------ epilogue (both CTAs, own 128 rows) ------------------------------
    const int ew = warp - 2;
    const int q = warp & 3;
    const int cbeg = (ew / 4) * half0, CPW = ew < 4 ? half0 : BN - half0;      // this warp's columns of the tile
    const uint32_t stage0 = epi_base + ew * EPI_BYTES;
    const uint32_t ltempty0 = map_to_cta(tempty_bar(0), 0), ltempty1 = map_to_cta(tempty_bar(1), 0);
    WarpEpi we{stage0, aux_bar(ew, 0), 0u, false};
    uint32_t lt = 0;
    for (int t = cluster_id; t < total; t += n_clusters, lt++) {
      int mt, nt, split;
      coords(t, mt, nt, split);
      const int m0 = mt * 2 * BM + (int)rank * BM, n0 = nt * BN;
      const int kbeg = split * kchunk, kend = min(p.K, kbeg + kchunk);
      const bool empty_k = kend <= kbeg;
      const uint32_t ab = naccum == 2 ? (lt & 1) : 0u, aph = naccum == 2 ? ((lt >> 1) & 1) : (lt & 1);
      // Bias: the four warps that share a column half share one 128-float slice per tile parity.  Each warp
      // fetches the slice into registers now (the latency hides behind the MMAs) and writes it -- every warp
      // the same values -- once the tile's accumulator is complete: by then every warp of the pair has drained
      // the tile before the previous one, the last reader of this parity's slice.  A warp reads only behind
      // its own writes, so no barrier between the warps is needed.
      const bool need_bias = p.epi.bias != nullptr && p.splits == 1;
      float* bias_s = reinterpret_cast<float*>(gen_base + epi_off + EPI_WARPS * EPI_BYTES) + ((ew / 4) * 2 + (lt & 1)) * (PAIR_BN / 2);
      float4 bias_pre = make_float4(0.f, 0.f, 0.f, 0.f);
      if (need_bias) {
        const int n = n0 + cbeg + lane * 4;
        const float* bp = p.epi.bias + n;
        if (n + 4 <= p.N) {
          bias_pre = *reinterpret_cast<const float4*>(bp);
        } else {
          if (n < p.N) bias_pre.x = bp[0];
          if (n + 1 < p.N) bias_pre.y = bp[1];
          if (n + 2 < p.N) bias_pre.z = bp[2];
        }
      }
      const int row = m0 + q * 32 + lane;
      const bool row_ok = row < p.M;
      const float ce_ref = CE && row_ok ? p.epi.ce_ref[row] : 0.f;      // (in front of the wait, like the bias)
      const int fx = n0 + cbeg, fy = m0 + q * 32, fcols = fy < p.M ? min(CPW, p.N - fx) : 0;   // fused epilogues: this warp's part
      if (FUSED) fused_prefetch<EPI, NB>(&map_x, we, fx, fy, fcols, lane);
#ifdef ERASE_DEV_AIDS
      const bool acct = p.dbg && blockIdx.x == 0 && threadIdx.x == 64;
      const long long e0 = acct ? clock64() : 0;
#endif
      bool ok = mbar_wait(tfull_bar(ab), aph);
      if (!ok) atomicExch(p.status, 3);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
#ifdef ERASE_DEV_AIDS
      const long long e1 = acct ? clock64() : 0;
      if (acct) p.dbg[4] += e1 - e0;                                   // epilogue warp 0: waiting for a finished accumulator
#endif
      if (need_bias) {
        *reinterpret_cast<float4*>(bias_s + lane * 4) = bias_pre;
        __syncwarp();
      }
      if (FUSED) {
        if (!fused_tile<EPI, NB>(p, &map_c, &map_x, we, tmem_base + ab * ACC_COLS + ((uint32_t)(q * 32) << 16) + (uint32_t)cbeg, fx, fy, fcols, row,
                             bias_s, lane)) {
          if (lane == 0) atomicExch(p.status, 10);
          break;
        }
      } else if (CE) {
        if (fcols > 0) {
          const float sum = ce_tile(p, &map_c, we, tmem_base + ab * ACC_COLS + ((uint32_t)(q * 32) << 16) + (uint32_t)cbeg, fx, fy, fcols, ce_ref, bias_s, lane);
          if (row_ok) p.epi.ce_psum[(long long)row * p.epi.ce_groups + fx / CPW] = sum;
        }
      } else if (xcol && nt == tiles_n_main) {     // the narrow tile: the extra product in every column, or in parts in the first three
        if (cbeg == 0 && fy < p.M) {
          uint32_t r[4];
          tc_ld4(tmem_base + ab * ACC_COLS + ((uint32_t)(q * 32) << 16), r);
          const float lead = __uint_as_float(r[0]);
          if (row_ok) p.xcol_out[row] = p.xcol_ones ? lead : lead + (__uint_as_float(r[1]) + __uint_as_float(r[2]));
        }
      } else {
        if (xwide && nt == tiles_n_main - 1 && cbeg == 0 && fy < p.M) {       // columns N .. N + 2 add up to the extra product
          uint32_t r[4];
          tc_ld4(tmem_base + ab * ACC_COLS + ((uint32_t)(q * 32) << 16) + (uint32_t)xcol_at, r);
          if (row_ok) p.xcol_out[row] = __uint_as_float(r[0]) + (__uint_as_float(r[1]) + __uint_as_float(r[2]));
        }
        if (fcols > 0)
          plain_tile(p, &map_c, we, tmem_base + ab * ACC_COLS + ((uint32_t)(q * 32) << 16) + (uint32_t)cbeg, fx, fy, fcols, row, split, empty_k, bias_s, lane);
      }
      tc_fence_before();
      __syncwarp();
#ifdef ERASE_DEV_AIDS
      if (acct) p.dbg[5] += clock64() - e1;                            // epilogue warp 0: draining one accumulator
#endif
      if (lane == 0) {   // accumulator drained: tell the leader's MMA thread
        if (leader) mbar_arrive(tempty_bar(ab));
        else mbar_arrive_cluster(ab ? ltempty1 : ltempty0);
      }
    }
    if (lane == 0 && we.store_pending) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
  }

  // Neither CTA may leave (or free its TMEM) while the other can still read its shared memory,
  // write its TMEM or signal its barriers.
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(tmem_cols) : "memory");
  }
}

// =================================================================================================
// Weight-gradient kernel: up to four wgrad GEMMs (dW = dY^T X, both operands MN-major, fp32 result) and the bias
// gradients that belong to them (db = column sums of dY) in ONE launch.  A cluster of S CTAs owns a 128 x 128 tile;
// each takes 1/S of the contraction, and the partial tiles are added inside the cluster, over distributed shared
// memory, in the order of the ranks: no partials in global memory, no second launch, one fixed summation order.
//
// The bias gradient is one more, 16 columns wide product, dY^T times a constant tile of ones, formed from the A operand
// that is in shared memory anyway.  Column tile nt forms it for the 64-deep blocks nt, nt + tiles_n, .. only, so that no
// CTA is held up by it (all of it in the first column tile: 512 x 2048 x 4096 15.8 us, none 12.7); the tiles_n partial
// sums are added elsewhere.
//
// A CTA does one tile and leaves; with three stages (101 KB, 256 TMEM columns) two share an SM, so that one's prologue
// and reduction hide behind the other's MMAs; a launch that leaves no SM two CTAs takes six stages instead.
// (Two to an SM never wait for each other's TMEM: 2 x 256 columns are all there are, and shared memory admits no third
// CTA of any kernel here that allocates some.)
//
// What bounds it: about 8 us of launch, first loads, reduction and last stores, then 64-deep blocks at 0.14 us, twice
// that where rows of dY and X miss the 32-byte sectors.  Before, each weight gradient was a launch of its own (or, up to
// 32 tiles, part of one that wrote partials for another launch to add) and the bias gradients another pass over dY:
// 4096 x 512 MLP, per block 2 x 17 + 8 us, now 19 (step 1150 -> 916 us); 256-wide transformer block, 33 + 6, now 14.
constexpr int WG_MAX = 4;
struct WgradProblem {
  int M, N, K, tiles_n, tile_begin;
  long long ldc;
  float* C;
  float* db;       // [tiles_n][M] partial bias gradients, or null
};
struct WgradArgs {
  int nprob, stages;
  int first;       // tile of the launch's first cluster
  int* status;
  WgradProblem prob[WG_MAX];
};
struct WgradMaps {
  CUtensorMap a[WG_MAX], b[WG_MAX];
};
constexpr uint32_t WG_STAGE_BYTES = 2 * BM * BK * 2;
constexpr uint32_t WG_TILE_BYTES = BM * 128 * 4;                 // a partial tile, laid over the operand stages
constexpr uint32_t WG_TMEM_COLS = 256;                           // 128 columns of the tile, 16 (read as 32) of the bias
constexpr size_t wg_smem(int stages) { return (size_t)stages * WG_STAGE_BYTES + 2048 + 8 * (2 * 8 + 4) + 1024; }
static_assert(3 * WG_STAGE_BYTES >= WG_TILE_BYTES + BM * 4, "the partial tile and the bias partials fit over three stages");

__device__ __forceinline__ float4 ld_cluster_v4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ float ld_cluster(uint32_t addr) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
  return v;
}

template <int S>
__global__ void __launch_bounds__(TC_THREADS, 2)
tc_wgrad_kernel(const __grid_constant__ WgradMaps maps, const __grid_constant__ WgradArgs g) {
  extern __shared__ uint8_t smem_raw[];
  constexpr uint32_t A_BYTES = BM * BK * 2;
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t ones = smem_base + g.stages * WG_STAGE_BYTES, bar_base = ones + 2048;
  auto full_bar = [&](uint32_t s) { return bar_base + 8u * s; };
  auto empty_bar = [&](uint32_t s) { return bar_base + 64u + 8u * s; };
  const uint32_t tfull_bar = bar_base + 128, tmem_slot = bar_base + 136;
  uint8_t* gen_base = smem_raw + (smem_base - smem_u32(smem_raw));
  volatile uint32_t* tmem_slot_ptr = reinterpret_cast<volatile uint32_t*>(gen_base + (tmem_slot - smem_base));

  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // (warp: known to be uniform)
  const int st0 = status_peek(g.status);
  const int rank = S > 1 ? (int)cluster_ctarank() : 0;
  const int t = g.first + (int)blockIdx.x / S;
  int pi = 0;
  while (pi + 1 < g.nprob && t >= g.prob[pi + 1].tile_begin) pi++;
  const WgradProblem& q = g.prob[pi];
  const int mt = (t - q.tile_begin) / q.tiles_n, nt = (t - q.tile_begin) % q.tiles_n;
  const int m0 = mt * BM, n0 = nt * 128;
  const int nkb = (q.K + BK - 1) / BK;                        // this rank's 64-deep blocks: kb0 .. kb0 + num_kb - 1
  const int kb0 = (int)((long long)nkb * rank / S), num_kb = (int)((long long)nkb * (rank + 1) / S) - kb0;
  const int first_b = q.db == nullptr ? num_kb : (nt - kb0 % q.tiles_n + q.tiles_n) % q.tiles_n;    // this CTA's blocks for the bias
  const bool bias = first_b < num_kb;                                                                // gradient, if there is one

  if (threadIdx.x == 32) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(&maps.a[pi]) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&maps.b[pi]) : "memory");
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < g.stages; s++) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    mbar_init(tfull_bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (threadIdx.x < 128) st_shared_v4(ones + 16 * threadIdx.x, 0x3f803f80u, 0x3f803f80u, 0x3f803f80u, 0x3f803f80u);   // bf16 1.0
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tmem_slot), "r"(WG_TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  pdl_wait();
  const bool dead = __syncthreads_or(st0 != 0) != 0;
  tc_fence_after();
  const uint32_t tmem = *tmem_slot_ptr;

  if (dead) {
    // the step is already void; every CTA still meets its cluster below
  } else if (warp == 0) {
    uint32_t s = 0, ph = 0;
    for (int kb = 0; kb < num_kb; kb++) {
      if (!mbar_wait_warp(empty_bar(s), ph ^ 1)) {
        if (lane == 0) atomicExch(g.status, 1);
        const long long t0 = clock64();       // copies in flight land before shared memory is released
        while (clock64() - t0 < 2000000LL) {}
        break;
      }
      const uint32_t a_dst = smem_base + s * WG_STAGE_BYTES, b_dst = a_dst + A_BYTES;
      const int k0 = (kb0 + kb) * BK;
      if (elect_one()) {
        mbar_expect_tx(full_bar(s), WG_STAGE_BYTES);
#pragma unroll
        for (int a = 0; a < 2; a++) {
          tma_load_2d(a_dst + a * (BK * 128), &maps.a[pi], m0 + a * 64, k0, full_bar(s));
          tma_load_2d(b_dst + a * (BK * 128), &maps.b[pi], n0 + a * 64, k0, full_bar(s));
        }
      }
      if (++s == (uint32_t)g.stages) { s = 0; ph ^= 1; }
    }
    pdl_trigger();
  } else if (warp == 1) {
    constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | ((uint32_t)(BM >> 4) << 24);   // A MN-major
    constexpr uint32_t IDESC_W = IDESC | (1u << 16) | ((uint32_t)(128 >> 3) << 17), IDESC_B = IDESC | ((uint32_t)(16 >> 3) << 17);
    const uint64_t ad0 = smem_desc(smem_base, BK * 128, 1024), bd0 = smem_desc(smem_base + A_BYTES, BK * 128, 1024), od = smem_desc(ones, 16, 1024);
    constexpr int STEP = (UMMA_K * 128) >> 4;
    uint32_t s = 0, ph = 0;
    int next_b = first_b;
    for (int kb = 0; kb < num_kb; kb++) {
      if (!mbar_wait_warp(full_bar(s), ph)) {
        if (lane == 0) atomicExch(g.status, 2);
        break;
      }
      tc_fence_after();
      const uint32_t off = s * (WG_STAGE_BYTES >> 4);
      if (kb == next_b) {
#pragma unroll
        for (int j = 0; j < 4; j++) tc_mma_warp(tmem + 128, ad0 + off + j * STEP, od, IDESC_B, (kb > first_b || j > 0) ? 1u : 0u);
        next_b += q.tiles_n;
      }
      tc_mma_block<1, STEP, STEP>(tmem, ad0 + off, bd0 + off, IDESC_W, kb > 0, empty_bar(s));
      if (++s == (uint32_t)g.stages) { s = 0; ph ^= 1; }
    }
    tc_commit_warp<1>(tfull_bar);
  } else {
    // this CTA's partial tile into shared memory, over the operand stages (their MMAs have read them): rows of 512
    // bytes, 16-byte pieces XOR-ed with the row, behind them the 128 bias partials
    const int q4 = warp & 3, half = (warp - 2) >> 2;
    const int row = q4 * 32 + lane;
    const uint32_t lane_off = (uint32_t)(q4 * 32) << 16;
    if (!mbar_wait_warp(tfull_bar, 0)) {
      if (lane == 0) atomicExch(g.status, 3);
    } else {
      tc_fence_after();
      uint32_t ra[32], rb[32];
      if (num_kb > 0) {
        tc_ld32_issue(tmem + lane_off + half * 64, ra);
        tc_ld32_issue(tmem + lane_off + half * 64 + 32, rb);
        tc_ld_wait(ra);
        tc_ld_wait(rb);
      } else {
#pragma unroll
        for (int j = 0; j < 32; j++) ra[j] = rb[j] = 0u;
      }
      const uint32_t my_row = smem_base + row * 512;
#pragma unroll
      for (int j = 0; j < 8; j++) {
        st_shared_v4(my_row + (((half * 16 + j) ^ (row & 7)) << 4), ra[4 * j], ra[4 * j + 1], ra[4 * j + 2], ra[4 * j + 3]);
        st_shared_v4(my_row + (((half * 16 + 8 + j) ^ (row & 7)) << 4), rb[4 * j], rb[4 * j + 1], rb[4 * j + 2], rb[4 * j + 3]);
      }
      if (q.db != nullptr && half == 0) {
        uint32_t r[32];
        if (bias) tc_ld32(tmem + lane_off + 128, r);
        else r[0] = 0u;
        asm volatile("st.shared.b32 [%0], %1;" ::"r"(smem_base + WG_TILE_BYTES + row * 4), "r"(r[0]) : "memory");
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (S > 1) cluster_sync_all();
  if (!dead) {
    // rank r finishes rows r * 128/S ..: one 16-byte piece per thread and turn, the ranks' partials added in order
    constexpr int ROWS = BM / S;
    const int r0 = rank * ROWS;
    uint32_t peer[S];
#pragma unroll
    for (int r = 0; r < S; r++) peer[r] = S > 1 ? map_to_cta(smem_base, r) : smem_base;
#pragma unroll 2
    for (int i = threadIdx.x; i < ROWS * 32; i += TC_THREADS) {
      const int row = r0 + (i >> 5), piece = i & 31;
      const uint32_t off = row * 512 + ((piece ^ (row & 7)) << 4);
      float4 v[S];
#pragma unroll
      for (int r = 0; r < S; r++) v[r] = ld_cluster_v4(peer[r] + off);
#pragma unroll
      for (int r = 1; r < S; r++) { v[0].x += v[r].x; v[0].y += v[r].y; v[0].z += v[r].z; v[0].w += v[r].w; }
      const int m = m0 + row, n = n0 + 4 * piece;
      if (m < q.M && n < q.N) *reinterpret_cast<float4*>(q.C + m * q.ldc + n) = v[0];
    }
    if (q.db != nullptr && threadIdx.x < ROWS) {
      const int row = r0 + threadIdx.x;
      float v = ld_cluster(peer[0] + WG_TILE_BYTES + row * 4);
#pragma unroll
      for (int r = 1; r < S; r++) v += ld_cluster(peer[r] + WG_TILE_BYTES + row * 4);
      if (m0 + row < q.M) q.db[(long long)nt * q.M + m0 + row] = v;
    }
  }
  if (S > 1) cluster_sync_all();       // no CTA leaves while another may still read its partials
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(WG_TMEM_COLS) : "memory");
  }
}

// =================================================================================================
// Dual-list persistent kernel: the forward of block b+1 and the backward of block b in ONE launch,
// each on its own share of the SMs (paper Section 2.2: B_b overlaps F_{b+1}; Sections 1 and 3.1:
// small GEMMs leave SMs idle and can share the device).  A launch carries up to DUAL_MAX problems
// in two ordered lists.  CTAs [0, split) work through list 0, the others through list 1; inside a
// list the tiles of all problems form one sequence that the list's CTAs take round-robin.  A problem
// may name an earlier problem of its list whose output it reads: before a CTA touches such a tile
// it waits (bounded) until a device counter says every tile of that problem has been stored.
// Every CTA walks its list in order and never waits for a later problem, all CTAs of the launch
// are resident (grid <= SMs, one CTA per SM), so the waits always resolve.
//   kind 0: GEMM tile (128 x 128), roles and pipeline as in tc_gemm_kernel, operand majors
//           chosen per problem; epilogue: bias, ReLU, ReLU derivative; bf16 or fp32 output or
//           fp32 split-K partials, all through TMA stores
//   kind 1: y = gelu(u), kind 2: g = g * gelu'(u) on 32 Ki-element chunks of bf16 data, done by the
//           eight epilogue warps with the same functions as the stand-alone elementwise kernel
// The arithmetic of a tile does not depend on which CTA computes it or when: the results are the
// bits of the same operations launched one by one.
constexpr int DUAL_MAX = 8;
constexpr int DUAL_EW_CHUNK = 32768;
constexpr long long DUAL_WAIT_CYCLES = 500000000LL;
struct DualProblem {
  int kind;                       // 0 GEMM, 1 gelu, 2 gelu derivative
  int M, N, K, splits, kchunk, tiles_m, tiles_n;
  int a_mn, b_mn;
  int out_mode;                   // 0: bf16 [M, N]; 1: fp32 [M, N]; 2: fp32 split-K partials [splits, M, N]
  int relu, dact_relu;
  int dep;                        // problem whose completion this one waits for, or -1
  int signal;                     // a later problem waits for this one: count finished tiles
  int ntiles, tile_begin;         // tiles of this problem; index of its first tile in its list's sequence
  const float* bias;
  const __nv_bfloat16* dact_src;
  long long ld_aux;
  const __nv_bfloat16* ew_src;
  __nv_bfloat16* ew_dst;
  long long ew_n;
};
struct DualArgs {
  int nprob, split;
  int first[2], count[2], total[2];   // per list: first problem, number of problems, tiles
  int* done;                          // [DUAL_MAX] finished epilogue-warp tiles per problem, zero at launch
  int* status;
  DualProblem prob[DUAL_MAX];
};
struct DualMaps {
  CUtensorMap a[DUAL_MAX], b[DUAL_MAX], c[DUAL_MAX];
};

__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
// waits until problem `dep` has stored all its tiles (8 epilogue warps each); false on expiry
__device__ __forceinline__ bool dual_wait_dep(const DualArgs& g, int dep) {
  if (dep < 0) return true;
  const int need = g.prob[dep].ntiles * EPI_WARPS;
  if (ld_acquire(g.done + dep) >= need) return true;
  const long long t0 = clock64();
  while (ld_acquire(g.done + dep) < need) {
    if (clock64() - t0 > DUAL_WAIT_CYCLES) return false;
    __nanosleep(64);
  }
  return true;
}
__device__ __forceinline__ int dual_find(const DualArgs& g, int list, int t) {
  int pi = g.first[list];
  const int end = g.first[list] + g.count[list];
  while (pi + 1 < end && t >= g.prob[pi + 1].tile_begin) pi++;
  return pi;
}

__global__ void __launch_bounds__(TC_THREADS, 1)
tc_dual_kernel(const __grid_constant__ DualMaps maps, const __grid_constant__ DualArgs g) {
  extern __shared__ uint8_t smem_raw[];
  constexpr int BN = 128;
  constexpr uint32_t A_BYTES = BM * BK * 2;
  constexpr uint32_t B_BYTES = BN * BK * 2;
  constexpr uint32_t STAGE_BYTES = A_BYTES + B_BYTES;
  constexpr uint32_t TMEM_COLS = 2 * BN;
  constexpr int STAGES = 4;
  constexpr int CPW = BN / 2;

  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t epi_base = smem_base + STAGES * STAGE_BYTES;
  const uint32_t bias_base = epi_base + EPI_WARPS * EPI_STAGE_BYTES;
  const uint32_t bar_base = bias_base + EPI_WARPS * EPI_BIAS_BYTES;
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (STAGES + s); };
  auto tfull_bar = [&](int a) { return bar_base + 8u * (2 * STAGES + a); };
  auto tempty_bar = [&](int a) { return bar_base + 8u * (2 * STAGES + 2 + a); };
  uint8_t* gen_base = smem_raw + (smem_base - smem_u32(smem_raw));
  volatile uint32_t* tmem_slot_ptr = reinterpret_cast<volatile uint32_t*>(gen_base + (bar_base - smem_base) + 8u * (2 * STAGES + 4));
  const uint32_t tmem_slot = bar_base + 8u * (2 * STAGES + 4);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int list = (int)blockIdx.x < g.split ? 0 : 1;
  const int rank = list == 0 ? (int)blockIdx.x : (int)blockIdx.x - g.split;
  const int nrank = list == 0 ? g.split : (int)gridDim.x - g.split;
  const int total = g.total[list];
  const int st0 = status_peek(g.status);
  if (threadIdx.x == 32) {
    for (int i = 0; i < g.nprob; i++) {
      asm volatile("prefetch.tensormap [%0];" ::"l"(&maps.a[i]) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"(&maps.b[i]) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"(&maps.c[i]) : "memory");
    }
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; s++) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    for (int a = 0; a < 2; a++) {
      mbar_init(tfull_bar(a), 1);
      mbar_init(tempty_bar(a), EPI_WARPS);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tmem_slot), "r"(TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  pdl_wait();
  const bool dead = __syncthreads_or(st0 != 0) != 0;
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot_ptr;

  if (dead) {
    // the step is already void: do nothing but free TMEM below
  } else if (warp == 0) {
    // ------------------------------ TMA producer ------------------------------
    if (lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      for (int t = rank; t < total && ok; t += nrank) {
        const int pi = dual_find(g, list, t);
        const DualProblem& q = g.prob[pi];
        if (q.kind != 0) continue;                      // elementwise chunks need no staging
        if (!dual_wait_dep(g, q.dep)) { atomicExch(g.status, 41); ok = false; break; }
        asm volatile("fence.proxy.async;" ::: "memory");   // the other CTAs' stores are ordered before this CTA's TMA reads
        const int local = t - q.tile_begin, per = q.tiles_m * q.tiles_n;
        const int split = local / per, r = local - split * per;
        const int mt = r / q.tiles_n, nt = r - mt * q.tiles_n;
        const int m0 = mt * BM, n0 = nt * BN;
        const int kbeg = split * q.kchunk, kend = min(q.K, kbeg + q.kchunk);
        const int num_kb = kend > kbeg ? (kend - kbeg + BK - 1) / BK : 0;
        for (int kb = 0; kb < num_kb; kb++, it++) {
          const int s = it % STAGES;
          const uint32_t ph = (it / STAGES) & 1;
          if (!mbar_wait(empty_bar(s), ph ^ 1)) { atomicExch(g.status, 1); ok = false; break; }
          mbar_expect_tx(full_bar(s), STAGE_BYTES);
          const uint32_t a_dst = smem_base + s * STAGE_BYTES;
          const uint32_t b_dst = a_dst + A_BYTES;
          const int k0 = kbeg + kb * BK;
          if (!q.a_mn) {
            tma_load_2d(a_dst, &maps.a[pi], k0, m0, full_bar(s));
          } else {
#pragma unroll
            for (int a = 0; a < BM / 64; a++) tma_load_2d(a_dst + a * (BK * 128), &maps.a[pi], m0 + a * 64, k0, full_bar(s));
          }
          if (!q.b_mn) {
            tma_load_2d(b_dst, &maps.b[pi], k0, n0, full_bar(s));
          } else {
#pragma unroll
            for (int a = 0; a < BN / 64; a++) tma_load_2d(b_dst + a * (BK * 128), &maps.b[pi], n0 + a * 64, k0, full_bar(s));
          }
        }
      }
      if (!ok) {
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000LL) {}
      }
    }
    pdl_trigger();
  } else if (warp == 1) {
    // ------------------------------ MMA issuer ------------------------------
    if (lane == 0) {
      uint32_t it = 0, lt = 0;
      bool ok = true;
      for (int t = rank; t < total && ok; t += nrank) {
        const int pi = dual_find(g, list, t);
        const DualProblem& q = g.prob[pi];
        if (q.kind != 0) continue;
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((q.a_mn ? 1u : 0u) << 15) | ((q.b_mn ? 1u : 0u) << 16) |
                               ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
        const int local = t - q.tile_begin, split = local / (q.tiles_m * q.tiles_n);
        const int kbeg = split * q.kchunk, kend = min(q.K, kbeg + q.kchunk);
        const int num_kb = kend > kbeg ? (kend - kbeg + BK - 1) / BK : 0;
        const uint32_t ab = lt & 1, aph = (lt >> 1) & 1;
        if (!mbar_wait(tempty_bar(ab), aph ^ 1)) { atomicExch(g.status, 4); ok = false; break; }
        tc_fence_after();
        const uint32_t tmem_d = tmem_base + ab * BN;
        for (int kb = 0; kb < num_kb; kb++, it++) {
          const int s = it % STAGES;
          const uint32_t ph = (it / STAGES) & 1;
          if (!mbar_wait(full_bar(s), ph)) { atomicExch(g.status, 2); ok = false; break; }
          tc_fence_after();
          const uint32_t a_src = smem_base + s * STAGE_BYTES;
          const uint32_t b_src = a_src + A_BYTES;
#pragma unroll
          for (int k = 0; k < BK / UMMA_K; k++) {
            const uint64_t ad = q.a_mn ? smem_desc(a_src + k * (UMMA_K * 128), BK * 128, 1024) : smem_desc(a_src + k * (UMMA_K * 2), 16, 1024);
            const uint64_t bd = q.b_mn ? smem_desc(b_src + k * (UMMA_K * 128), BK * 128, 1024) : smem_desc(b_src + k * (UMMA_K * 2), 16, 1024);
            tc_mma(tmem_d, ad, bd, idesc, (kb > 0 || k > 0) ? 1u : 0u);
          }
          tc_commit(empty_bar(s));
        }
        tc_commit(tfull_bar(ab));
        lt++;
      }
    }
  } else {
    // ------------------------------ epilogue / elementwise warps ------------------------------
    const int ew = warp - 2;
    const int q4 = warp & 3;
    const int cbeg = (ew / 4) * CPW;
    const uint32_t stage0 = epi_base + ew * EPI_STAGE_BYTES;
    float* bias_s = reinterpret_cast<float*>(gen_base + (bias_base - smem_base) + ew * EPI_BIAS_BYTES);
    uint32_t sbuf = 0;
    bool store_pending = false;
    uint32_t lt = 0;
    for (int t = rank; t < total; t += nrank) {
      const int pi = dual_find(g, list, t);
      const DualProblem& q = g.prob[pi];
      if (q.kind != 0) {
        // ---- elementwise chunk: the 256 threads of these warps, 16 bytes per access ----
        bool ok = true;
        if (lane == 0) ok = dual_wait_dep(g, q.dep);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) { if (lane == 0) atomicExch(g.status, 42); break; }
        asm volatile("fence.proxy.async;" ::: "memory");
        const long long beg = (long long)(t - q.tile_begin) * DUAL_EW_CHUNK;
        const long long end = beg + DUAL_EW_CHUNK < q.ew_n ? beg + DUAL_EW_CHUNK : q.ew_n;
        for (long long i = beg + (long long)(ew * 32 + lane) * 8; i < end; i += 256 * 8) {     // ew_n % 8 == 0
          const uint4 u = *reinterpret_cast<const uint4*>(q.ew_src + i);
          float x[8], y[8];
          unpack8_bf16(u, x);
          if (q.kind == 1) {
#pragma unroll
            for (int j = 0; j < 8; j++) y[j] = x[j];
            gelu_bf16_n<8>(y);
          } else {
            unpack8_bf16(*reinterpret_cast<const uint4*>(q.ew_dst + i), y);
            dgelu_bf16_n<8>(x, y);
          }
          uint4 o;
          o.x = pack2(y[0], y[1]); o.y = pack2(y[2], y[3]); o.z = pack2(y[4], y[5]); o.w = pack2(y[6], y[7]);
          *reinterpret_cast<uint4*>(q.ew_dst + i) = o;
        }
        if (q.signal) {
          __threadfence();
          __syncwarp();
          if (lane == 0) atomicAdd(g.done + pi, 1);
        }
        continue;
      }
      const int local = t - q.tile_begin, per = q.tiles_m * q.tiles_n;
      const int split = local / per, r = local - split * per;
      const int mt = r / q.tiles_n, nt = r - mt * q.tiles_n;
      const int m0 = mt * BM, n0 = nt * BN;
      const int kbeg = split * q.kchunk, kend = min(q.K, kbeg + q.kchunk);
      const bool empty_k = kend <= kbeg;
      const uint32_t ab = lt & 1, aph = (lt >> 1) & 1;
      lt++;
      if (q.bias) {
        __syncwarp();
        for (int j = lane; j < CPW; j += 32) {
          const int n = n0 + cbeg + j;
          bias_s[j] = n < q.N ? q.bias[n] : 0.f;
        }
        __syncwarp();
      }
      const int row = m0 + q4 * 32 + lane;
      const bool row_ok = row < q.M;
      bool ok = mbar_wait(tfull_bar(ab), aph);
      if (!ok) atomicExch(g.status, 3);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      const bool rows_in = m0 + q4 * 32 < q.M;
      const bool f32 = q.out_mode != 0;
      if (n0 + cbeg < q.N) {
#pragma unroll 1
        for (int cc = 0; cc < CPW; cc += 32) {
          const int c0 = cbeg + cc;
          if (n0 + c0 >= q.N) break;
          uint32_t rr[32];
          if (!empty_k) {
            tc_ld32(tmem_base + ab * BN + ((uint32_t)(q4 * 32) << 16) + (uint32_t)c0, rr);
          } else {
#pragma unroll
            for (int j = 0; j < 32; j++) rr[j] = 0u;
          }
          if (f32 || (cc & 63) == 0) {
            sbuf ^= 1;
            if (lane == 0 && store_pending) tma_store_wait_read1();
            __syncwarp();
          }
          const uint32_t stage = stage0 + sbuf * 4096;
          const uint32_t my_row = stage + lane * 128;
#pragma unroll
          for (int g8 = 0; g8 < 4; g8++) {
            float v[8];
#pragma unroll
            for (int j = 0; j < 8; j++) v[j] = __uint_as_float(rr[g8 * 8 + j]);
            const int n = n0 + c0 + g8 * 8;
            if (q.bias) {
              const float4 b0 = *reinterpret_cast<const float4*>(bias_s + cc + g8 * 8);
              const float4 b1 = *reinterpret_cast<const float4*>(bias_s + cc + g8 * 8 + 4);
              v[0] += b0.x; v[1] += b0.y; v[2] += b0.z; v[3] += b0.w;
              v[4] += b1.x; v[5] += b1.y; v[6] += b1.z; v[7] += b1.w;
            }
            if (q.relu) {
#pragma unroll
              for (int j = 0; j < 8; j++) v[j] = fmaxf(v[j], 0.f);
            }
            if (q.dact_relu && row_ok && n < q.N) {       // N % 8 == 0 whenever an auxiliary operand is present
              float tsrc[8];
              unpack8_bf16(*reinterpret_cast<const uint4*>(q.dact_src + (long long)row * q.ld_aux + n), tsrc);
#pragma unroll
              for (int j = 0; j < 8; j++) v[j] = tsrc[j] > 0.f ? v[j] : 0.f;
            }
            if (f32) {
              const uint32_t s0 = my_row + (((2 * g8) ^ (lane & 7)) << 4), s1 = my_row + (((2 * g8 + 1) ^ (lane & 7)) << 4);
              st_shared_v4(s0, __float_as_uint(v[0]), __float_as_uint(v[1]), __float_as_uint(v[2]), __float_as_uint(v[3]));
              st_shared_v4(s1, __float_as_uint(v[4]), __float_as_uint(v[5]), __float_as_uint(v[6]), __float_as_uint(v[7]));
            } else {
              const uint32_t s0 = my_row + (((((cc & 63) >> 3) + g8) ^ (lane & 7)) << 4);
              st_shared_v4(s0, pack2(v[0], v[1]), pack2(v[2], v[3]), pack2(v[4], v[5]), pack2(v[6], v[7]));
            }
          }
          const bool last_chunk = (cc & 63) == 32 || n0 + c0 + 32 >= q.N;
          if (f32 || last_chunk) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0 && rows_in) {
              const int x = f32 ? n0 + c0 : n0 + cbeg + (cc & ~63), y = m0 + q4 * 32;
              if (q.out_mode == 2) tma_store_3d(&maps.c[pi], stage, x, y, split);
              else tma_store_2d(&maps.c[pi], stage, x, y);
              tma_store_commit();
              store_pending = true;
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(tempty_bar(ab));
      if (q.signal) {     // a later problem reads this output: report the tile once its stores have landed
        if (lane == 0) {
          if (store_pending) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
          store_pending = false;
          asm volatile("fence.proxy.async;" ::: "memory");
          __threadfence();
          atomicAdd(g.done + pi, 1);
        }
        __syncwarp();
      }
    }
    if (lane == 0 && store_pending) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
  }
}

// The bounded wait on its own: one thread waits, with the given limit, on a barrier that nothing
// ever signals, records status code 8 and returns.  It returns by construction (the wait is
// clock-bounded) and touches no tensor memory; used to check that an expired wait surfaces as
// ERASE_ETIMEOUT and leaves the context usable.
__global__ void wait_selftest_kernel(int* status, long long limit_cycles) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bar), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (!mbar_wait(smem_u32(&bar), 0, limit_cycles)) atomicExch(status, 8);
  }
}

// Host-side caches are per device: a process may drive several GPUs.
constexpr int MAX_DEVICES = 64;
int current_device() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) dev = 0;
  return dev;
}
int sm_count() {
  static std::atomic<int> cache[MAX_DEVICES];
  const int dev = current_device();
  int n = cache[dev].load(std::memory_order_relaxed);
  if (n == 0) {
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 2) n = 148;
    cache[dev].store(n, std::memory_order_relaxed);
  }
  return n;
}
// cudaFuncSetAttribute(MaxDynamicSharedMemorySize) once per (kernel, device); `done` is the kernel's own table
template <typename K>
cudaError_t ensure_smem(K kernel, size_t smem, std::atomic<bool>* done) {
  const int dev = current_device();
  if (done[dev].load(std::memory_order_acquire)) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess) done[dev].store(true, std::memory_order_release);
  return e;
}

typedef CUresult (*EncodeFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                             const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                             CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeFn encode_fn() {
  static const EncodeFn fn = []() -> EncodeFn {   // initialised once, thread-safe (the entry point is process-wide)
    const char* off = getenv("ERASE_TC_ENCODE");  // 0: as if the driver had no encoder (for checking what then runs instead)
    if (off && atoi(off) == 0) return nullptr;
    void* p = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) == cudaSuccess &&
        qres == cudaDriverEntryPointSuccess)
      return (EncodeFn)p;
    cudaGetLastError();
    return nullptr;
  }();
  return fn;
}

// Tensor map of a row-major bf16 or fp32 matrix (rank 2) or stack of matrices (rank 3):
// dims[0] contiguous elements per row, rows stride_bytes[0] apart, 128-byte swizzle; the box's
// inner extent is 128 bytes.  Out-of-bounds elements read as zero and are not written.
bool encode_map(void* out, const void* base, bool f32, int rank, const cuuint64_t* dims, const cuuint64_t* stride_bytes,
                const cuuint32_t* box) {
  EncodeFn fn = encode_fn();
  if (!fn) return false;
  for (int i = 0; i + 1 < rank; i++)
    if (stride_bytes[i] % 16) return false;
  if (reinterpret_cast<uintptr_t>(base) & 15) return false;
  CUtensorMap tmp;
  cuuint32_t estr[3] = {1u, 1u, 1u};
  CUresult r = fn(&tmp, f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank,
                  const_cast<void*>(base), dims, stride_bytes, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r == CUDA_SUCCESS) memcpy(out, &tmp, sizeof(tmp));
  return r == CUDA_SUCCESS;
}

// operand map: `inner` contiguous bf16 elements per row, `outer` rows `ld` elements apart; box 64 x box_outer
bool encode_2d(void* out, const void* base, long long inner, long long outer, long long ld, int box_outer) {
  cuuint64_t dims[2] = {(cuuint64_t)inner, (cuuint64_t)outer};
  cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  cuuint32_t box[2] = {64u, (cuuint32_t)box_outer};
  return encode_map(out, base, false, 2, dims, strides, box);
}

// Which epilogue a GEMM takes, and the auxiliary operand that arrives by TMA (a residual before a multiplier or a
// derivative source; the other one, if any, is read from global memory by the epilogue's threads).
int epi_kind(const GemmArgs& g) {
  const Epilogue& e = g.epi;
  if (e.ce_ref) return EPI_CE;
  if (g.splits > 1) return EPI_PLAIN;
  if (e.act == ACT_GELU) return EPI_GELU;
  if (e.dact == ACT_GELU) return EPI_DGELU;
  const int n = (e.res ? 1 : 0) + (e.mul || e.dact != ACT_NONE || e.post_mul ? 1 : 0);
  return n == 0 ? EPI_PLAIN : (n == 1 ? EPI_AUX : EPI_AUX2);
}
const void* aux_by_tma(const GemmArgs& g) {
  const Epilogue& e = g.epi;
  return e.res ? e.res : (e.mul ? e.mul : e.dact_src);
}
void fill_args(TcArgs& p, const GemmArgs& g, const TcPlan& plan) {
  const Epilogue& e = g.epi;
  p.M = g.M; p.N = g.N; p.K = g.K;
  p.C = g.C; p.ldc = g.ldc; p.c_f32 = g.c_f32;
  p.splits = g.splits; p.ws = g.ws; p.epi = e; p.epi.ld_aux = e.ld_aux ? e.ld_aux : g.N; p.status = plan.status; p.dbg = plan.dbg;
  p.tma_c = plan.tma_c;
  p.bias_add = e.bias && g.splits == 1;
  p.relu = e.act == ACT_RELU && g.splits == 1;
  const int second = e.post_mul ? AUX_POST : (e.mul ? AUX_MUL : (e.dact != ACT_NONE ? AUX_DRELU : AUX_NONE));
  p.aux_mode = e.res ? AUX_RES : second;
  p.aux2_mode = e.res ? second : AUX_NONE;
  p.wide = g.ldc % 16 == 0 && ((!e.pre_out && !e.post_out) || p.epi.ld_aux % 16 == 0) &&
           ((reinterpret_cast<uintptr_t>(g.C) | reinterpret_cast<uintptr_t>(e.pre_out) | reinterpret_cast<uintptr_t>(e.post_out)) & 31) == 0;
  p.aux2 = (const __nv_bfloat16*)(e.post_mul ? e.post_mul : (e.mul ? e.mul : e.dact_src));
}

template <int BN, bool A_MN, bool B_MN, int EPI>
cudaError_t launch_t(const GemmArgs& g, const TcPlan& plan, cudaStream_t s, int max_ctas) {
  constexpr int STAGES = stages_for(BN);
  constexpr size_t smem = (size_t)STAGES * (BM * BK * 2 + BN * BK * 2) + EPI_WARPS * 4096u * single_bufs(BN, EPI) + 16u * (BN >= 128 ? BN / 2 : 64) + 8 * (2 * STAGES + 32);
  static_assert(smem <= 232448, "single-CTA kernel: shared memory over the per-CTA limit");
  static std::atomic<bool> attr_set[MAX_DEVICES];
  if (cudaError_t e = ensure_smem(tc_gemm_kernel<BN, A_MN, B_MN, EPI>, smem, attr_set)) return e;
  TcArgs p;
  fill_args(p, g, plan);
  p.sched = plan.sched;
  p.xcol_out = nullptr;
  const int num_sms = sm_count();
  const long long total = (long long)((g.N + BN - 1) / BN) * ((g.M + BM - 1) / BM) * g.splits;
  long long cap = (max_ctas > 0 && max_ctas < num_sms) ? max_ctas : num_sms;
  dim3 grid((unsigned)(total < cap ? total : cap));
  CUtensorMap ma, mb, mc, mx;
  static_assert(sizeof(CUtensorMap) == 128, "tensor map size");
  memcpy(&ma, plan.map_a, sizeof(ma));
  memcpy(&mb, plan.map_b, sizeof(mb));
  memcpy(&mc, plan.map_c, sizeof(mc));
  memcpy(&mx, plan.map_x, sizeof(mx));
  if (total <= (long long)grid.x) p.sched = nullptr;   // one tile per CTA: nothing to balance
  pdl_launch(tc_gemm_kernel<BN, A_MN, B_MN, EPI>, grid, TC_THREADS, smem, s, ma, mb, mc, mx, p);
  return cudaGetLastError();
}

template <bool A_MN, bool B_MN, int EPI>
cudaError_t launch_pair_t(const GemmArgs& g, const TcPlan& plan, cudaStream_t s, int max_ctas) {
  constexpr size_t fixed = EPI_WARPS * 4096u * pair_epi_bufs(EPI) + PAIR_BIAS_BYTES + 8 * (2 * PAIR_MAX_STAGES + 8 + 2 * EPI_WARPS);
  const bool xwide = plan.xcol == XCOL_WIDE;
  const int widest = xwide ? std::min(PAIR_BN, plan.bn + 32) : plan.bn;
  const uint32_t stage_bytes = epi_fused(EPI) ? 2 * BM * BK * 2 : BM * BK * 2 + (B_MN ? (widest / 2 + 63) / 64 * (BK * 128) : plan.bn / 2 * (BK * 2));
  // five stages, more where a narrow tile's smaller ones fit into about the same 205 KB
  const int stages = epi_fused(EPI) ? 5 : std::min(PAIR_MAX_STAGES, std::max(5, (int)((205u * 1024 - fixed) / stage_bytes)));
  const size_t smem = stages * (size_t)stage_bytes + fixed;
  static std::atomic<bool> attr_set[MAX_DEVICES];
  if (cudaError_t e = ensure_smem(tc_gemm_pair_kernel<A_MN, B_MN, EPI>, 232448, attr_set)) return e;
  TcArgs p;
  fill_args(p, g, plan);
  p.sched = nullptr;
  p.xcol_out = plan.xcol ? g.xcol_out : nullptr;
  p.xcol_ones = g.xcol_ones != nullptr;
  p.xcol_wide = xwide;
  p.bn = plan.bn;
  p.stages = stages;
  p.stage_bytes = stage_bytes;
  const int num_sms = sm_count();
  const long long total = (long long)((g.N + plan.bn - 1) / plan.bn + (plan.xcol && !xwide ? 1 : 0)) * ((g.M + 2 * BM - 1) / (2 * BM)) * g.splits;
  long long cap = ((max_ctas > 1 && max_ctas < num_sms) ? max_ctas : num_sms) / 2;
  dim3 grid(2u * (unsigned)(total < cap ? total : cap));
  CUtensorMap ma, mb, mc, mx;
  memcpy(&mx, plan.map_x, sizeof(mx));
  memcpy(&ma, plan.map_a, sizeof(ma));
  memcpy(&mb, plan.map_b, sizeof(mb));
  memcpy(&mc, plan.map_c, sizeof(mc));
  pdl_launch(tc_gemm_pair_kernel<A_MN, B_MN, EPI>, grid, TC_THREADS, smem, s, ma, mb, mc, mx, p, (uint32_t)plan.pair_tmem_cols);
  return cudaGetLastError();
}

// Fused epilogues occur on the layouts that carry them: the forward (both operands K-major) and the dgrad (B MN-major).
template <int BN>
cudaError_t launch_bn(const GemmArgs& g, const TcPlan& plan, cudaStream_t s, int max_ctas) {
  switch (epi_kind(g)) {
    case EPI_CE: return launch_t<BN, false, false, EPI_CE>(g, plan, s, max_ctas);
    case EPI_GELU: return launch_t<BN, false, false, EPI_GELU>(g, plan, s, max_ctas);
    case EPI_DGELU: return launch_t<BN, false, true, EPI_DGELU>(g, plan, s, max_ctas);
    case EPI_AUX: return plan.b_mn ? launch_t<BN, false, true, EPI_AUX>(g, plan, s, max_ctas) : launch_t<BN, false, false, EPI_AUX>(g, plan, s, max_ctas);
    case EPI_AUX2: return plan.b_mn ? launch_t<BN, false, true, EPI_AUX2>(g, plan, s, max_ctas) : launch_t<BN, false, false, EPI_AUX2>(g, plan, s, max_ctas);
  }
  if (plan.a_mn) return plan.b_mn ? launch_t<BN, true, true, EPI_PLAIN>(g, plan, s, max_ctas) : launch_t<BN, true, false, EPI_PLAIN>(g, plan, s, max_ctas);
  return plan.b_mn ? launch_t<BN, false, true, EPI_PLAIN>(g, plan, s, max_ctas) : launch_t<BN, false, false, EPI_PLAIN>(g, plan, s, max_ctas);
}
cudaError_t launch_pair(const GemmArgs& g, const TcPlan& plan, cudaStream_t s, int max_ctas) {
  switch (epi_kind(g)) {
    case EPI_CE: return launch_pair_t<false, false, EPI_CE>(g, plan, s, max_ctas);
    case EPI_GELU: return launch_pair_t<false, false, EPI_GELU>(g, plan, s, max_ctas);
    case EPI_DGELU: return launch_pair_t<false, true, EPI_DGELU>(g, plan, s, max_ctas);
    case EPI_AUX: return plan.b_mn ? launch_pair_t<false, true, EPI_AUX>(g, plan, s, max_ctas) : launch_pair_t<false, false, EPI_AUX>(g, plan, s, max_ctas);
    case EPI_AUX2: return plan.b_mn ? launch_pair_t<false, true, EPI_AUX2>(g, plan, s, max_ctas) : launch_pair_t<false, false, EPI_AUX2>(g, plan, s, max_ctas);
  }
  if (plan.a_mn) return plan.b_mn ? launch_pair_t<true, true, EPI_PLAIN>(g, plan, s, max_ctas) : launch_pair_t<true, false, EPI_PLAIN>(g, plan, s, max_ctas);
  return plan.b_mn ? launch_pair_t<false, true, EPI_PLAIN>(g, plan, s, max_ctas) : launch_pair_t<false, false, EPI_PLAIN>(g, plan, s, max_ctas);
}

}  // namespace

// ---- dual-list persistent kernel: host side ---------------------------------------------------
struct TcDualPlan {
  DualArgs args;
  DualMaps maps;
  int grid;
};

int tc_dual_max() { return DUAL_MAX; }

TcDualPlan* tc_dual_plan(const DualItem* items_in, int n, int* done_dev, int* status) {
  if (n < 1 || n > DUAL_MAX || !done_dev) return nullptr;
  // list 0 first, then list 1, each in the given order
  DualItem items[DUAL_MAX];
  int cnt = 0, first1 = 0;
  for (int l = 0; l < 2; l++) {
    if (l == 1) first1 = cnt;
    for (int i = 0; i < n; i++)
      if (items_in[i].list == l) items[cnt++] = items_in[i];
  }
  if (cnt != n) return nullptr;
  for (int i = 0; i < n; i++)
    if (items[i].kind == 0 && items[i].g.xcol_out) return nullptr;   // the extra-column product exists in the pair kernel only
  TcDualPlan* plan = new TcDualPlan();
  DualArgs& a = plan->args;
  memset(&a, 0, sizeof(a));
  a.nprob = n;
  a.done = done_dev;
  a.status = status;
  a.first[0] = 0; a.count[0] = first1;
  a.first[1] = first1; a.count[1] = n - first1;
  double work[2] = {0, 0};
  auto fail = [&]() { delete plan; return (TcDualPlan*)nullptr; };
  for (int l = 0; l < 2; l++) {
    int tiles = 0, last_chain = -1;
    for (int i = a.first[l]; i < a.first[l] + a.count[l]; i++) {
      const DualItem& it = items[i];
      DualProblem& q = a.prob[i];
      q.kind = it.kind;
      q.dep = last_chain;
      q.tile_begin = tiles;
      if (it.kind == 0) {
        const GemmArgs& g = it.g;
        const Epilogue& e = g.epi;
        if (!tc_gemm_supported(g) || e.alpha != 1.f || e.mul || e.res || e.pre_out || e.ce_ref || (e.act != ACT_NONE && e.act != ACT_RELU) ||
            (e.dact != ACT_NONE && e.dact != ACT_RELU) || (g.splits > 1 && (!g.ws || e.bias || e.act != ACT_NONE || e.dact != ACT_NONE)))
          return fail();
        q.M = g.M; q.N = g.N; q.K = g.K; q.splits = g.splits;
        q.kchunk = (((g.K + g.splits - 1) / g.splits) + BK - 1) / BK * BK;
        q.tiles_m = (g.M + BM - 1) / BM;
        q.tiles_n = (g.N + 127) / 128;
        q.a_mn = g.sa_k != 1; q.b_mn = g.sb_k != 1;
        q.relu = e.act == ACT_RELU; q.dact_relu = e.dact == ACT_RELU;
        q.bias = e.bias;
        q.dact_src = (const __nv_bfloat16*)e.dact_src;
        q.ld_aux = e.ld_aux ? e.ld_aux : g.N;
        q.ntiles = q.tiles_m * q.tiles_n * g.splits;
        bool ok = q.a_mn ? encode_2d(&plan->maps.a[i], g.A, g.M, g.K, g.sa_k, BK) : encode_2d(&plan->maps.a[i], g.A, g.K, g.M, g.sa_m, BM);
        ok = ok && (q.b_mn ? encode_2d(&plan->maps.b[i], g.B, g.N, g.K, g.sb_k, BK) : encode_2d(&plan->maps.b[i], g.B, g.K, g.N, g.sb_n, 128));
        if (!ok) return fail();
        if (g.splits > 1) {
          q.out_mode = 2;
          cuuint64_t dims[3] = {(cuuint64_t)g.N, (cuuint64_t)g.M, (cuuint64_t)g.splits};
          cuuint64_t str[2] = {(cuuint64_t)g.N * 4, (cuuint64_t)g.M * g.N * 4};
          cuuint32_t box[3] = {32u, 32u, 1u};
          ok = encode_map(&plan->maps.c[i], g.ws, true, 3, dims, str, box);
        } else if (g.c_f32) {
          q.out_mode = 1;
          cuuint64_t dims[2] = {(cuuint64_t)g.N, (cuuint64_t)g.M};
          cuuint64_t str[1] = {(cuuint64_t)g.ldc * 4};
          cuuint32_t box[2] = {32u, 32u};
          ok = encode_map(&plan->maps.c[i], g.C, true, 2, dims, str, box);
        } else {
          q.out_mode = 0;
          cuuint64_t dims[2] = {(cuuint64_t)g.N, (cuuint64_t)g.M};
          cuuint64_t str[1] = {(cuuint64_t)g.ldc * 2};
          cuuint32_t box[2] = {64u, 32u};
          ok = encode_map(&plan->maps.c[i], g.C, false, 2, dims, str, box);
        }
        if (!ok) return fail();
        work[l] += (double)q.ntiles * ((q.kchunk + BK - 1) / BK + 6);
      } else {
        if (it.ew_n < 8 || it.ew_n % 8 || ((reinterpret_cast<uintptr_t>(it.ew_src) | reinterpret_cast<uintptr_t>(it.ew_dst)) & 15)) return fail();
        q.ew_src = (const __nv_bfloat16*)it.ew_src;
        q.ew_dst = (__nv_bfloat16*)it.ew_dst;
        q.ew_n = it.ew_n;
        q.ntiles = (int)((it.ew_n + DUAL_EW_CHUNK - 1) / DUAL_EW_CHUNK);
        plan->maps.a[i] = plan->maps.a[0]; plan->maps.b[i] = plan->maps.b[0]; plan->maps.c[i] = plan->maps.c[0];
        work[l] += (double)q.ntiles * 8;
      }
      tiles += q.ntiles;
      if (!it.leaf) last_chain = i;
    }
    a.total[l] = tiles;
  }
  for (int i = 0; i < n; i++)
    for (int j = i + 1; j < n; j++)
      if (a.prob[j].dep == i) a.prob[i].signal = 1;
  for (int i = n; i < DUAL_MAX; i++) { plan->maps.a[i] = plan->maps.a[0]; plan->maps.b[i] = plan->maps.b[0]; plan->maps.c[i] = plan->maps.c[0]; }
  const int sms = sm_count();
  plan->grid = sms;
  if (a.total[0] == 0) a.split = 0;
  else if (a.total[1] == 0) a.split = sms;
  else {
    int sp = (int)(sms * work[0] / (work[0] + work[1]) + 0.5);
    a.split = sp < 1 ? 1 : (sp > sms - 1 ? sms - 1 : sp);
  }
  return plan;
}

void tc_dual_free(TcDualPlan* plan) { delete plan; }

cudaError_t tc_dual_launch(const TcDualPlan* plan, cudaStream_t s) {
  constexpr size_t smem = (size_t)4 * (BM * BK * 2 + 128 * BK * 2) + EPI_WARPS * (EPI_STAGE_BYTES + EPI_BIAS_BYTES) + 8 * (2 * 4 + 16) + 1024;
  static std::atomic<bool> attr_set[MAX_DEVICES];
  if (cudaError_t e = ensure_smem(tc_dual_kernel, smem, attr_set)) return e;
  cudaError_t e = cudaMemsetAsync(plan->args.done, 0, DUAL_MAX * sizeof(int), s);
  if (e != cudaSuccess) return e;
  pdl_launch(tc_dual_kernel, plan->grid, TC_THREADS, smem, s, plan->maps, plan->args);
  return cudaGetLastError();
}

bool tc_encode_rows_bf16(void* map128, const void* base, long long inner, long long outer, long long ld, int box_rows) {
  return encode_2d(map128, base, inner, outer, ld, box_rows);
}

cudaError_t tc_wait_selftest(int* status, long long limit_cycles, cudaStream_t s) {
  wait_selftest_kernel<<<1, 32, 0, s>>>(status, limit_cycles);
  return cudaGetLastError();
}

template <int S>
static cudaError_t launch_wgrad(const WgradMaps& maps, WgradArgs g, int tiles, int max_ctas, cudaStream_t s, int* launches) {
  static std::atomic<bool> attr_set[MAX_DEVICES];
  if (cudaError_t e = ensure_smem(tc_wgrad_kernel<S>, wg_smem(6), attr_set)) return e;
  // A CTA leaves with its tile, so a cap on them is kept by launches one behind the other (not dependent ones: those
  // would hold SMs beside the launch before).
  const int per = max_ctas > 0 ? std::max(1, max_ctas / S) : tiles;
  for (*launches = 0; g.first < tiles; g.first += per, ++*launches) {
    const dim3 grid((unsigned)(std::min(per, tiles - g.first) * S));
    if (cudaError_t e = pdl_launch_cluster(tc_wgrad_kernel<S>, grid, TC_THREADS, wg_smem(g.stages), s, (unsigned)S, g.first == 0, maps, g)) return e;
  }
  return cudaSuccess;
}

bool tc_wgrad_plan(const GemmArgs* gs, float* const* db, int n, int splits, int* status, TcWgradPlan* plan) {
  if (n < 1 || n > WG_MAX || (splits != 1 && splits != 2 && splits != 4 && splits != 8)) return false;
  plan->n = n;
  plan->splits = splits;
  plan->status = status;
  plan->tiles = 0;
  for (int i = 0; i < n; i++) {
    const GemmArgs& g = gs[i];
    if (!tc_gemm_supported(g) || g.sa_k == 1 || g.sb_k == 1 || !g.c_f32 || g.N % 4 != 0 || g.ldc % 4 != 0 || (reinterpret_cast<uintptr_t>(g.C) & 15) != 0) return false;
    plan->M[i] = g.M; plan->N[i] = g.N; plan->K[i] = g.K; plan->C[i] = (float*)g.C; plan->ldc[i] = g.ldc; plan->db[i] = db[i];
    plan->tiles_n[i] = (g.N + 127) / 128;
    plan->tile_begin[i] = plan->tiles;
    plan->tiles += (g.M + BM - 1) / BM * plan->tiles_n[i];
    if (!encode_2d(plan->map_a[i], g.A, g.M, g.K, g.sa_k, BK) || !encode_2d(plan->map_b[i], g.B, g.N, g.K, g.sb_k, BK)) return false;
  }
  plan->stages = plan->tiles * splits > sm_count() ? 3 : 6;
  return true;
}

cudaError_t tc_wgrad_launch(const TcWgradPlan& plan, cudaStream_t s, int max_ctas, int* launches) {
  WgradMaps maps;
  WgradArgs g;
  memset(&g, 0, sizeof(g));
  g.nprob = plan.n; g.stages = plan.stages; g.status = plan.status;
  for (int i = 0; i < WG_MAX; i++) {
    const int k = i < plan.n ? i : 0;
    memcpy(&maps.a[i], plan.map_a[k], 128);
    memcpy(&maps.b[i], plan.map_b[k], 128);
    if (i < plan.n) g.prob[i] = WgradProblem{plan.M[i], plan.N[i], plan.K[i], plan.tiles_n[i], plan.tile_begin[i], plan.ldc[i], plan.C[i], plan.db[i]};
  }
  switch (plan.splits) {
    case 1: return launch_wgrad<1>(maps, g, plan.tiles, max_ctas, s, launches);
    case 2: return launch_wgrad<2>(maps, g, plan.tiles, max_ctas, s, launches);
    case 4: return launch_wgrad<4>(maps, g, plan.tiles, max_ctas, s, launches);
    default: return launch_wgrad<8>(maps, g, plan.tiles, max_ctas, s, launches);
  }
}

// Time of the weight-gradient kernel on a set of problems, with the split (1, 2, 4 or 8 CTAs a tile) that makes it
// smallest.  One CTA per SM: a fixed part and a pace per 64-deep block that falls off as more SMs pull from L2; more
// CTAs than SMs: the blocks of the fullest SM at the pace of two sharing one, a split of them pays for its reductions.
// Rows that do not start on 32-byte sectors (stride % 16 elements) or 128-byte lines (% 64) load at 0.48 and 0.8 of the
// pace (680 x 2136 x 3001: 26 us).  Measured against estimate, us, column sums included: 512 x 2048 x 4096
// 13.3 / 13.6, with 2048 x 512 19.0 / 18.4, 512 x 512 x 4096 10.1 / 10.9, four of a 256-wide transformer block 14.3 /
// 13.7, of a 512-wide one 33.6 / 34.3; the largest that is held back here comes out 12 % low, 768 x 3072 x 8192 33.2 / 29.1.
// No split beyond 128 CTAs, so that other streams' kernels find SMs.  The line hardly matters: nine of the steps in
// perf/cases.py are within 0.4 % without it (CTR with its main network 749 us, 750.5 without), and at 64 within 0.5 % but
// for the LM of d 256 on five streams (775 us, 766 at 64).
double tc_wgrad_us(const GemmArgs* gs, int n, int* splits) {
  double best = 1e30;
  for (int s = 1; s <= 8; s *= 2) {
    int ctas = 0;
    for (int i = 0; i < n; i++) ctas += (gs[i].M + BM - 1) / BM * ((gs[i].N + 127) / 128) * s;
    double blocks = 0, longest = 0;       // in units of an aligned one
    bool deep = true;
    for (int i = 0; i < n; i++) {
      const GemmArgs& g = gs[i];
      auto slow = [](long long stride) { return stride % 64 == 0 ? 1. : (stride % 16 == 0 ? 1.25 : 2.1); };
      const int nkb = (g.K + BK - 1) / BK;
      deep = deep && (s == 1 || nkb >= 4 * s);
      const double b = .5 * (slow(g.sa_k) + slow(g.sb_k)) * ((nkb + s - 1) / s);
      blocks += b * ((g.M + BM - 1) / BM) * ((g.N + 127) / 128) * s;
      longest = std::max(longest, b);
    }
    if (!deep || (s > 1 && ctas > 128)) continue;
    const int waves = (ctas + 147) / 148;
    double t = 8.5 + (s > 1 ? .3 : 0.);
    if (waves == 1) t += longest * (.125 + .00025 * ctas);
    else t += std::max(blocks / 148, longest * std::min(waves, 2)) * (waves == 2 ? .2 : .28) + (s > 1 ? .8 * waves : 0.);
    if (t < best) { best = t; *splits = s; }
  }
  return best;
}

bool tc_can_encode() {
  int n = 0;
  if (cudaGetDeviceCount(&n) != cudaSuccess || n < 1) {      // no device: sizes are asked for, as on a machine that has one
    cudaGetLastError();
    return true;
  }
  return encode_fn() != nullptr;
}

bool tc_gemm_supported(const GemmArgs& g) {
  if (g.K < 64 || g.N < 16 || g.M < 1) return false;
  auto operand_ok = [](const void* p, long long s_mn, long long s_k) {
    if (reinterpret_cast<uintptr_t>(p) & 15) return false;
    if (s_k == 1) return s_mn % 8 == 0 && s_mn > 0;
    if (s_mn == 1) return s_k % 8 == 0 && s_k > 0;
    return false;
  };
  if (!operand_ok(g.A, g.sa_m, g.sa_k) || !operand_ok(g.B, g.sb_n, g.sb_k)) return false;
  // a [1 x K] operand is ambiguous (both strides may be 1): leave such GEMVs to the SIMT kernel
  if ((g.sa_m == 1 && g.sa_k == 1) || (g.sb_n == 1 && g.sb_k == 1)) return false;
  const Epilogue& e = g.epi;
  if (e.alpha != 1.f) return false;
  if (g.splits > 1) return true;                // fp32 partials: no epilogue
  if ((e.pre_out && e.act != ACT_GELU) || (e.act == ACT_RELU && !e.bias)) return false;
  if (e.post_mul && (!e.res || e.mul || e.dact != ACT_NONE)) return false;
  if (e.act == ACT_GELU || e.mul || e.res || e.dact != ACT_NONE) {
    // fused epilogues move tiles by TMA, or rows in 16-byte pieces (GELU's two outputs), as bf16; K-major A only
    if (e.mul && e.dact != ACT_NONE) return false;
    if (g.c_f32 || g.sa_k != 1) return false;
    const long long ld = e.ld_aux ? e.ld_aux : g.N;
    if (ld % 8 != 0 || g.N % 8 != 0 || g.ldc % 8 != 0) return false;
    const void* rows[7] = {e.mul, e.res, e.dact != ACT_NONE ? e.dact_src : nullptr, e.pre_out, g.C, e.post_mul, e.post_out};
    for (const void* r : rows)
      if (reinterpret_cast<uintptr_t>(r) & 15) return false;
    if (e.act == ACT_GELU && (!e.pre_out || e.mul || e.res || e.dact != ACT_NONE || g.sb_k != 1)) return false;
    if (e.dact == ACT_GELU && (e.bias || e.act != ACT_NONE || e.mul || e.res || g.sb_n != 1)) return false;
  }
  return true;
}

// Tile of a GEMM: the CTA-pair kernel (256 x bn over two SMs) or the single-CTA kernel (128 x bn), by a model of its
// time.  Every CTA (or pair) works through ceil(tiles / units) tiles; a tile costs its 64-deep blocks at the larger of
// the issue rate and its share of the L2 (13.8 TB/s when all units pull), or its epilogue where that is longer; the
// last epilogue is not hidden; fp32 partials are written, read back and summed.  The constants are a fit to 255 GEMMs
// (the forward, dgrad and weight-gradient shapes of the models here at 512 to 32768 rows, splits 1 to 6), each timed
// with all five tiles: the model's pick is 0.6 % slower than the best one on average, "pair tiles from 56 of them
// on, else single", which it replaces, 5.3 % (3001 x 1024 x 1680: single 128 wide 22, pair 192 wide 14 us;
// 1680 x 1680 x 4096 weight gradient 42 -> 26; 8192 x 768 x 3072 pair 256 wide 37, 192 wide 33).
// (74 pairs and 148 SMs stand in it as numbers, here and in tc_wgrad_us: the constants were fitted on that device, and the
// choice must not differ between the sizing pass, which needs no device, and the building one.)
struct Tile { int pair, bn; double us; };
struct TileCost { int pair, bn; double block_us, l2_kb, epi_us; };
static const TileCost kTiles[] = {{0, 128, .200, 32, 1.20}, {0, 256, .355, 48, 1.77}, {1, 128, .154, 48, 1.66}, {1, 192, .259, 56, 1.70}, {1, 256, .297, 64, 2.22}};
// Where a pair tile of this width takes the extra column: columns of B in the last column tile where they fit in (it is at
// most 256 wide; 32 wider costs next to nothing), else in narrow tiles.
static int xcol_place(const GemmArgs& g, int bn) {
  return !g.xcol_ones && g.N - (g.N - 1) / bn * bn + 16 <= PAIR_BN ? XCOL_WIDE : XCOL_NARROW;
}
// (xcol: narrow tiles for the extra column)
static double tile_us(const GemmArgs& g, const TileCost& c, bool xcol) {
  const int tiles_m = (g.M + (c.pair ? 256 : 128) - 1) / (c.pair ? 256 : 128);
  long long ntiles = (long long)tiles_m * ((g.N + c.bn - 1) / c.bn) * g.splits;
  const int units = c.pair ? 74 : 148, kb = ((g.K + g.splits - 1) / g.splits + BK - 1) / BK;
  const bool gelu = g.splits == 1 && (g.epi.act == ACT_GELU || g.epi.dact == ACT_GELU);
  const double epi = c.epi_us * (g.splits > 1 || g.c_f32 ? 1.15 : 1.0) * (gelu ? 2.4 : 1.0);
  const double slow = 1. + .22 * ((g.sa_m == 1 ? g.sa_k : g.sa_m) % 16 != 0) + .22 * ((g.sb_n == 1 ? g.sb_k : g.sb_n) % 16 != 0);   // rows off the 32-byte sectors
  auto round_us = [&](double active) { return std::max(kb * slow * std::max(c.block_us, c.l2_kb * active / 13.76e3), epi); };
  // the extra column's narrow tiles: on idle pairs, or one (0.17 us a block) behind some pairs' full ones, or among them
  const bool last_narrow = xcol && ntiles <= units && ntiles + tiles_m > units;
  if (xcol && ntiles > units) ntiles += tiles_m;
  double t = 3.86 + (c.pair ? .75 : 0.) + epi + (ntiles / units) * round_us(units);
  if (ntiles % units) t += round_us((double)(ntiles % units));
  if (last_narrow) t += .17 * kb;
  if (g.splits > 1) t += .35 + (g.splits + 1.) * g.M * g.N * 4e-6 / 4.67;
  return t;
}
static Tile choose_tile(const GemmArgs& g, bool tma_c) {
  if (g.N <= 64) return {0, 64, tile_us(g, kTiles[0], false)};
  Tile best = {0, 128, 1e30};
  for (const TileCost& c : kTiles) {
    if (c.pair && (!tma_c || g.M < 256)) continue;
    if (g.epi.ce_ref && c.pair && c.bn != 256) continue;      // the softmax head's partial sums: 128-column groups
    if (c.bn > 128 && g.N <= 128) continue;
    const bool xcol = g.xcol_out && c.pair, narrow = xcol && xcol_place(g, c.bn) == XCOL_NARROW;
    double t = tile_us(g, c, narrow);
    if (g.xcol_out && !xcol) t += 3. + 2e-6 * g.M * g.K / 4.;  // the caller's separate column sum over A
    // 256 wide with narrow tiles against 192 wide with a wider last tile, where 256 divides the columns (measured, estimated;
    // us): 32768 x 1024 x 8192 418 / 449, 398 / 425; 1280 547 / 537, 486 / 502; 1536 621 / 597, 574 / 541; 1792 709 / 764, 618 / 695;
    // 2048 804 / 851, 706 / 772; 32768 x 1280 x 4096 269 / 269, 246 / 254; 8192 x 1280 x 8192 137 / 156, 133 / 155
    if (narrow && !g.xcol_ones) t *= 1.04;
    if (t < best.us) best = {c.pair, c.bn, t};
  }
  return best;
}

int tc_gemm_best_splits(GemmArgs g, int max_splits, int min_k, double* us) {
  g.ws = reinterpret_cast<float*>(uintptr_t(4096));           // (only its presence matters here)
  int best = 1;
  double best_us = 0;
  float* const xcol_out = g.xcol_out;
  for (int s = 1; s <= max_splits && (s == 1 || g.K / s >= min_k); s++) {
    g.splits = s;
    g.xcol_out = s == 1 ? xcol_out : nullptr;
    const double t = choose_tile(g, true).us + (s > 1 && xcol_out ? 3. + 2e-6 * g.M * g.K / 4. : 0.);
    if (s == 1 || t < best_us) { best = s; best_us = t; }
  }
  if (us) *us = best_us;
  return best;
}

static Tile pick_tile(const GemmArgs& g, bool tma_c) {
  Tile t = choose_tile(g, tma_c);
  if (const char* f = getenv("ERASE_TC_TILE")) {      // measuring aid: p128 p192 p256 (CTA pair), s64 s128 s256 (single CTA)
    const int bn = atoi(f + 1);
    if (f[0] == 'p' && tma_c && g.M >= 256 && (bn == 128 || bn == 192 || bn == 256) && !(g.epi.ce_ref && bn != 256)) t = {1, bn, 0.};
    if (f[0] == 's' && (bn == 64 || bn == 128 || bn == 256)) t = {0, bn, 0.};
  }
  return t;
}

bool tc_gemm_takes_xcol(const GemmArgs& g) {
  // Not where the narrow tiles would take longer than a pass over A: 32768-deep 4096 x 1024 (64 tiles and 16 narrow ones
  // for 74 pairs) 246 us and 73 for the pass, with them 390.
  GemmArgs h = g;
  h.xcol_out = nullptr;
  if (choose_tile(h, true).us + 3. + 2e-6 * g.M * g.K / 4. < choose_tile(g, true).us) return false;
  // (fp32 result through TMA: 16-byte aligned rows)
  return tc_gemm_supported(g) && g.sa_k != 1 && g.sb_k != 1 && g.c_f32 && g.ldc % 4 == 0 && g.N % 8 == 0 && (reinterpret_cast<uintptr_t>(g.C) & 15) == 0 &&
         pick_tile(g, true).pair;
}

bool tc_gemm_plan(const GemmArgs& g, int* status, TcPlan* plan) {
  if (!tc_gemm_supported(g)) return false;
  plan->a_mn = g.sa_k != 1;
  plan->b_mn = g.sb_k != 1;
  plan->status = status;
  plan->launches = 1;
  // outputs through TMA stores where their layout allows it (else the single-CTA kernel stores directly)
  memset(plan->map_c, 0, sizeof(plan->map_c));
  plan->tma_c = 0;
  if (g.splits > 1) {
    cuuint64_t dims[3] = {(cuuint64_t)g.N, (cuuint64_t)g.M, (cuuint64_t)g.splits};
    cuuint64_t str[2] = {(cuuint64_t)g.N * 4, (cuuint64_t)g.M * g.N * 4};
    cuuint32_t box[3] = {32u, 32u, 1u};
    plan->tma_c = g.ws && encode_map(plan->map_c, g.ws, true, 3, dims, str, box) ? 1 : 0;
  } else if (g.c_f32) {
    cuuint64_t dims[2] = {(cuuint64_t)g.N, (cuuint64_t)g.M};
    cuuint64_t str[1] = {(cuuint64_t)g.ldc * 4};
    cuuint32_t box[2] = {32u, 32u};
    plan->tma_c = encode_map(plan->map_c, g.C, true, 2, dims, str, box) ? 1 : 0;
  } else {
    cuuint64_t dims[2] = {(cuuint64_t)g.N, (cuuint64_t)g.M};
    cuuint64_t str[1] = {(cuuint64_t)g.ldc * 2};
    cuuint32_t box[2] = {64u, 32u};
    plan->tma_c = encode_map(plan->map_c, g.C, false, 2, dims, str, box) ? 1 : 0;
  }
  // fused epilogues with an auxiliary operand: its tensor map (GELU stores both of its outputs without one)
  memset(plan->map_x, 0, sizeof(plan->map_x));
  if (epi_by_tma(epi_kind(g))) {
    const void* x = aux_by_tma(g);
    cuuint64_t dims[2] = {(cuuint64_t)g.N, (cuuint64_t)g.M};
    cuuint64_t str[1] = {(cuuint64_t)(g.epi.ld_aux ? g.epi.ld_aux : g.N) * 2};
    cuuint32_t box[2] = {64u, 32u};
    if (!plan->tma_c || !encode_map(plan->map_x, x, false, 2, dims, str, box)) return false;
  }
  const Tile t = pick_tile(g, plan->tma_c != 0);
  plan->pair = t.pair;
  plan->bn = t.bn;
  static const int env_cols = getenv("ERASE_TC_PAIR_COLS") ? atoi(getenv("ERASE_TC_PAIR_COLS")) : 512;
  plan->pair_tmem_cols = env_cols == 256 ? 256 : 512;
  // extra-column product: weight-gradient layout on the pair kernel, no split (a last tile that is not full multiplies
  // the extra columns too; its store ends at N)
  plan->xcol = g.xcol_out != nullptr && plan->pair && plan->a_mn && plan->b_mn && g.splits == 1 && g.N % 8 == 0 ? xcol_place(g, plan->bn) : 0;
  if (!(plan->a_mn ? encode_2d(plan->map_a, g.A, g.M, g.K, g.sa_k, BK) : encode_2d(plan->map_a, g.A, g.K, g.M, g.sa_m, BM))) return false;
  if (plan->xcol && g.xcol_ones && !encode_2d(plan->map_x, g.xcol_ones, 16, BK, 16, BK)) return false;
  // (a CTA of a pair stages half of the tile's columns)
  return plan->b_mn ? encode_2d(plan->map_b, g.B, g.N + (plan->xcol && !g.xcol_ones ? 16 : 0), g.K, g.sb_k, BK)
                    : encode_2d(plan->map_b, g.B, g.K, g.N, g.sb_n, plan->pair ? plan->bn / 2 : plan->bn);
}

int tc_ce_group_cols(const TcPlan& plan) { return (plan.pair || plan.bn >= 128) ? plan.bn / 2 : 64; }

cudaError_t tc_gemm_launch(const GemmArgs& g, const TcPlan& plan, cudaStream_t s, int max_ctas) {
  // cross-entropy head forward: both operands K-major, bias, bf16 output through TMA
  if (g.epi.ce_ref && (plan.a_mn || plan.b_mn || !plan.tma_c || g.splits != 1 || !g.epi.bias || !g.epi.ce_psum)) return cudaErrorInvalidValue;
  if (plan.pair) return launch_pair(g, plan, s, max_ctas);
  switch (plan.bn) {
    case 64: return launch_bn<64>(g, plan, s, max_ctas);
    case 256: return launch_bn<256>(g, plan, s, max_ctas);
    default: return launch_bn<128>(g, plan, s, max_ctas);
  }
}

}  // namespace erase
