// Learned stand-in for the acoustic substeps of an advection step.
//
// A message-passing network over the frozen neighbour graph of the step predicts each
// fluid particle's velocity and density change over Dt_ad (the network is the project's
// own; the paper has none). Definition (an FP64 reference implementation of the same
// network is kept with the tests):
//   u_i  = [v_i/c0, 100 (rho_i/rho0 - 1), Dt_ad c0/h, 1]                      K = 16
//   x_ij = [r_ij/h, (v_i - v_j)/c0, 100 dev_i, 100 dev_j, wall]  (walls: v_j = 0, dev_j = 0)
//   h_i  = relu(W_enc u_i)
//   3 rounds, shared weights:
//     z_ij = relu(W_e1 [x_ij, h_j, 1])     m_ij = W_e2 [z_ij, 1]            K = 80, 80
//     a_i  = (1/NBAR) sum_j m_ij           h_i += W_n2 [relu(W_n1 [h_i, a_i, 1]), 1]   K = 144, 80
//   y_i  = W_d2 [relu(W_d1 [h_i, 1]), 1]                                     K = 80, 80
//   targets [(dv_i - g Dt_ad)/V_S, 100 drho_i/rho0], V_S = |g| Dt_ad (U_ref when g = 0),
//   loss = mean squared error.
// Every product rounds its operands to bfloat16 and accumulates in FP32 on the tensor
// cores: the layer-by-layer path (training, and inference when the fused rounds are off)
// on the fifth-generation tensor cores (tcgen05, 128-row tiles, accumulators in TMEM; see
// sph_tc.cuh), the fused inference rounds with warp-level mma.sync m16n8k16 (both sum each
// 16-wide K step in the same order, so the two paths agree bit for bit). These layers are
// skinny (64 outputs, K <= 144: ~34 FLOP per byte moved, far below the tensor-core ridge of
// ~285), so unfused they are bound by HBM, not by the MMA. Weight gradients are summed per block and then over
// blocks in a fixed order and node-embedding gradients of the neighbour gather are summed
// per node over its reverse edges in edge order, so a training step is deterministic (only
// the reported loss value is accumulated with atomics).
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <vector>

#include "sph.h"
#include "sph_handle.h"
#include "sph_kernels.h"
#include "sph_tc.cuh"

using bf16 = __nv_bfloat16;

namespace sph {
namespace learned {

constexpr int F = 64;
constexpr int ROUNDS = 3;
constexpr float S_RHO = 100.0f;
enum { L_ENC = 0, L_E1, L_E2, L_N1, L_N2, L_D1, L_D2, L_COUNT };
constexpr int kRows[L_COUNT] = {64, 64, 64, 64, 64, 64, 16};
constexpr int kCols[L_COUNT] = {16, 80, 80, 144, 80, 80, 80};
__constant__ int c_rows[L_COUNT] = {64, 64, 64, 64, 64, 64, 16};
__constant__ int c_cols[L_COUNT] = {16, 80, 80, 144, 80, 80, 80};
constexpr int kWeights = 32000;
constexpr int kTile = 64;                 // rows per tile of the weight gradient

inline int w_offset(int l) {
  int o = 0;
  for (int k = 0; k < l; ++k) o += kRows[k] * kCols[k];
  return o;
}

inline float nbar(int dim) { return dim == 2 ? 20.0f : 80.0f; }

__device__ __forceinline__ uint32_t ld_u32(const bf16* p) { return *reinterpret_cast<const uint32_t*>(p); }

__device__ __forceinline__ uint32_t pack2(bf16 lo, bf16 hi) {
  return (uint32_t)__bfloat16_as_ushort(lo) | ((uint32_t)__bfloat16_as_ushort(hi) << 16);
}

__device__ __forceinline__ void mma16816(float* c, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// ------------------------------------------------------------------ dense forward
// Y = X W^T for M rows on the fifth-generation tensor cores (sph_tc.cuh). Each CTA (one
// warpgroup of 128 threads) keeps W [NO x K] in shared memory in the core-matrix layout and
// walks 128-row tiles (grid-stride): the tile's rows are copied into the A operand, one
// thread issues the K/16 MMAs into TMEM, and each warp then reads its 32 rows' accumulators
// (TMEM lane = row) 32 columns at a time for the epilogue. Epilogue per element
// (m, n < NO): y = acc, y = max(y, 0) if relu; out_f32[m, n] = y (or += y with accum)
// for n < nf_store; out_b[m, col0 + n] = bf16(y) for n < nb_store <= 64, 0 where
// mask[m, n] <= 0 with MASK (ReLU backward; read ahead of the results). Copies are shaped
// for the memory system: a quarter-warp moves one core matrix (8 rows x 16 bytes: one
// 128-byte shared-memory wavefront, two full global sectors per row pair of pieces), and each
// warp stages 128 bytes of its 32 rows in shared memory (in the tile the tensor core has just
// read, so the staging costs no shared memory of its own) to store them as whole lines.
// What bounds it at the training sizes (a few tiles an SM) is the chain of latencies of a tile:
// W comes with the first tile, every copy is issued without a division or a wait, the MMAs are
// issued before the next tile's copies, the mask and the sums to add to are read in whole lines
// and all at once, and the epilogue has one staging round per 128 bytes of a row. With W loaded
// first, 16 columns a round in 4-byte shared accesses, the mask read row by row and a CTA a
// tile, the 28 layers of a training step of 3,200 particles (64,000 edges) took 380 us and take
// 257 us. One tile buffer and more CTAs an SM instead of two buffers was no faster.
// K is a multiple of 16, ldx, ldo, col0, nb_store and ldm multiples of 8, ldf and nf_store of 4
// (checked by the host wrapper). A wait for the tensor core that runs out sets
// ERR_TIMEOUT in *err and the CTA stops.
constexpr int kDenseStageLd = 144;          // staged row stride (bytes): 128 and a piece of padding

// shared memory of k_dense: W, then two row tiles of 128 x K, each large enough to serve as
// the four warps' staging blocks once the tensor core has read it
__host__ __device__ constexpr int dense_w_bytes(int NO, int K) { return (NO * K * 2 + 127) / 128 * 128; }
__host__ __device__ constexpr int dense_tile_bytes(int K) {
  return ((128 * K * 2 > 128 * kDenseStageLd ? 128 * K * 2 : 128 * kDenseStageLd) + 127) / 128 * 128;
}

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem, bool valid) {
  const unsigned dst = (unsigned)__cvta_generic_to_shared(smem);
  const int n = valid ? 16 : 0;                       // 0: fill the 16 bytes with zeros
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(gmem), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// 16-byte pieces of an R-row operand, [R x K] row-major in global memory (row stride ld
// elements), into the core-matrix layout: piece (row, kc) by lane (row % 8) + 8 (kc % 4) of a
// warp-sized block of 8 rows x 4 pieces. Rows at or past rows_valid are zero.
__device__ __forceinline__ void load_operand(unsigned char* dst, int R, int K, const bf16* __restrict__ src,
                                             int64_t ld, int64_t rows_valid) {
  const int KC = K / 8, KB = (KC + 3) / 4;           // pieces per row, 4-piece groups
  const int blocks = (R / 8) * KB;
  const int lane = threadIdx.x & 31;
  for (int blk = threadIdx.x >> 5; blk < blocks; blk += blockDim.x >> 5) {
    const int r = (blk / KB) * 8 + (lane & 7), kc = (blk % KB) * 4 + (lane >> 3);
    if (kc >= KC) continue;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (r < rows_valid) v = *reinterpret_cast<const uint4*>(src + (int64_t)r * ld + kc * 8);
    *reinterpret_cast<uint4*>(dst + tc::core_offset(R, r, kc * 8)) = v;
  }
}

// The same by the four warps of k_dense with the shape known when compiled, by cp.async
// (completed by the caller's cp_async_wait_all): every copy of a lane is issued without a
// division or a wait for the one before.
template <int R, int K>
__device__ __forceinline__ void load_tile(unsigned char* dst, const bf16* __restrict__ src, int ld, int rows_valid) {
  constexpr int KC = K / 8, KB = (KC + 3) / 4, kBlocks = (R / 8) * KB;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, r0 = lane & 7, k0 = lane >> 3;
#pragma unroll
  for (int q = 0; q < (kBlocks + 3) / 4; ++q) {
    const int blk = 4 * q + warp, r = blk / KB * 8 + r0, kc = blk % KB * 4 + k0;
    if (blk >= kBlocks || kc >= KC) continue;
    const bool valid = r < rows_valid;
    cp_async16(dst + tc::core_offset(R, r, kc * 8), src + (valid ? (int64_t)r * ld : 0) + kc * 8, valid);
  }
}

// all ones in the halves of a pair of bf16 that are > 0
__device__ __forceinline__ uint32_t positive2(uint32_t m) {
  return __hgt2_mask(*reinterpret_cast<const __nv_bfloat162*>(&m), __floats2bfloat162_rn(0.f, 0.f));
}

template <int NO, int K, bool MASK>
__global__ void __launch_bounds__(128)
k_dense(int64_t M, const bf16* __restrict__ X, int ldx, const bf16* __restrict__ W,
        float* __restrict__ out_f32, int ldf, int nf_store, int accum, bf16* __restrict__ out_b, int ldo,
        int col0, int nb_store, int relu, const bf16* __restrict__ mask, int ldm, int* __restrict__ err) {
  constexpr int COLS = tc::tmem_cols(NO);
  extern __shared__ __align__(128) unsigned char tc_smem[];
  __shared__ __align__(8) uint64_t bar;
  __shared__ uint32_t tmem_slot;
  unsigned char* sB = tc_smem;                        // NO x K
  constexpr int tile_bytes = dense_tile_bytes(K);
  unsigned char* sA0 = tc_smem + dense_w_bytes(NO, K);   // two 128 x K row tiles
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if ((int64_t)blockIdx.x * 128 < M) {                // the first tile and W stream in
    const int64_t m0 = (int64_t)blockIdx.x * 128;
    load_tile<128, K>(sA0, X + m0 * ldx, ldx, (int)min(M - m0, (int64_t)128));
    load_tile<NO, K>(sB, W, K, NO);
  }
  cp_async_commit();
  if (threadIdx.x == 0) tc::mbar_init(&bar);
  if (warp == 0) tc::tmem_alloc(&tmem_slot, COLS);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tmem_slot;
  const uint32_t b_addr = tc::smem_u32(sB);
  const int64_t tiles = (M + 127) / 128;
  uint32_t phase = 0;
  int buf = 0;
  for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x, buf ^= 1) {
    const int64_t m0 = tile * 128;
    unsigned char* sA = sA0 + buf * tile_bytes;
    cp_async_wait_all();
    tc::fence_to_async();
    __syncthreads();                                  // this tile in place; the other buffer free
    if (threadIdx.x == 0) {
      tc::fence_after_sync();
      tc::mma_tile<NO>(tmem, tc::smem_u32(sA), b_addr, K, false, &bar);
    }
    __syncwarp();
    const int64_t next = tile + gridDim.x;
    if (next < tiles)                                 // the next tile streams in meanwhile
      load_tile<128, K>(sA0 + (buf ^ 1) * tile_bytes, X + next * 128 * ldx, ldx,
                        (int)min(M - next * 128, (int64_t)128));
    cp_async_commit();
    const int64_t mw = m0 + warp * 32;                // this warp's first row
    // the mask of this lane's bf16 pieces (below), in flight during the MMAs
    uint4 mk[MASK ? 8 : 1];
    if (MASK)
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int64_t m = mw + 4 * q + (lane >> 3);
        mk[q] = make_uint4(0u, 0u, 0u, 0u);
        if (m < M && (lane & 7) * 8 < nb_store) mk[q] = *reinterpret_cast<const uint4*>(&mask[m * ldm + (lane & 7) * 8]);
      }
    const bool done = tc::mbar_wait(&bar, phase);
    phase ^= 1u;
    if (!__syncthreads_and(done)) {                   // the same decision in every thread
      if (threadIdx.x == 0) atomicOr(err, ERR_TIMEOUT);
      break;
    }
    tc::fence_after_sync();
    // this warp's staging block, in the tile the tensor core is done with: 32 rows of 128
    // bytes, padded so that rows of 16-byte pieces go in and lines come out without conflicts
    unsigned char* st = sA + warp * 32 * kDenseStageLd;
    unsigned char* mine = st + lane * kDenseStageLd;  // the row whose accumulators this lane reads
    if (out_f32) {
#pragma unroll
      for (int c0 = 0; c0 < NO; c0 += 32) {           // 32 (or the last 16) columns at a time
        constexpr int kW = NO % 32;
        const int w = NO - c0 < 32 ? kW : 32;
        if (c0 >= nf_store) break;
        float y[32];
        tc::tmem_ld16_async(tc::tmem_addr(tmem, warp, c0), y);
        if (w == 32) tc::tmem_ld16_async(tc::tmem_addr(tmem, warp, c0 + 16), y + 16);
        tc::tmem_wait(y);
        if (w == 32) tc::tmem_wait(y + 16);
#pragma unroll
        for (int q = 0; q < w; q += 4) {
          float4 v = make_float4(y[q], y[q + 1], y[q + 2], y[q + 3]);
          if (relu) v = make_float4(fmaxf(v.x, 0.f), fmaxf(v.y, 0.f), fmaxf(v.z, 0.f), fmaxf(v.w, 0.f));
          *reinterpret_cast<float4*>(mine + q * 4) = v;
        }
        __syncwarp();
        const int pieces = w / 4;                     // 16-byte pieces of a row
        float4 o[8];
        float4* dst[8];
        bool in[8];
#pragma unroll
        for (int q = 0; q < pieces; ++q) {
          const int r = (q * 32 + lane) / pieces, c = (q * 32 + lane) % pieces * 4;
          const int64_t m = mw + r;
          in[q] = m < M && c0 + c < nf_store;
          dst[q] = reinterpret_cast<float4*>(&out_f32[m * ldf + c0 + c]);
          o[q] = *reinterpret_cast<const float4*>(st + r * kDenseStageLd + c * 4);
        }
        if (accum) {                                  // every sum read before the first is written
          float4 p[8];
#pragma unroll
          for (int q = 0; q < pieces; ++q) p[q] = in[q] ? *dst[q] : o[q];
#pragma unroll
          for (int q = 0; q < pieces; ++q) o[q] = make_float4(p[q].x + o[q].x, p[q].y + o[q].y, p[q].z + o[q].z, p[q].w + o[q].w);
        }
#pragma unroll
        for (int q = 0; q < pieces; ++q)
          if (in[q]) *dst[q] = o[q];
        __syncwarp();                                 // the staging block is reused next
      }
    }
    if (out_b) {                                      // at most 64 columns
#pragma unroll
      for (int c0 = 0; c0 < (NO < 64 ? NO : 64); c0 += 32) {
        const int w = NO - c0 < 32 ? NO % 32 : 32;
        float y[32];
        tc::tmem_ld16_async(tc::tmem_addr(tmem, warp, c0), y);
        if (w == 32) tc::tmem_ld16_async(tc::tmem_addr(tmem, warp, c0 + 16), y + 16);
        tc::tmem_wait(y);
        if (w == 32) tc::tmem_wait(y + 16);
#pragma unroll
        for (int q = 0; q < w; q += 8) {
          uint4 o;
          uint32_t* u = reinterpret_cast<uint32_t*>(&o);
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float lo = y[q + 2 * k], hi = y[q + 2 * k + 1];
            const __nv_bfloat162 v = relu ? __floats2bfloat162_rn(fmaxf(lo, 0.f), fmaxf(hi, 0.f)) : __floats2bfloat162_rn(lo, hi);
            u[k] = *reinterpret_cast<const uint32_t*>(&v);
          }
          *reinterpret_cast<uint4*>(mine + (c0 + q) * 2) = o;
        }
      }
      __syncwarp();
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int r = 4 * q + (lane >> 3), c = (lane & 7) * 8;
        const int64_t m = mw + r;
        if (m < M && c < nb_store) {
          uint4 o = *reinterpret_cast<const uint4*>(st + r * kDenseStageLd + c * 2);
          if (MASK) {
            const uint4 k = mk[MASK ? q : 0];
            o = make_uint4(o.x & positive2(k.x), o.y & positive2(k.y), o.z & positive2(k.z), o.w & positive2(k.w));
          }
          *reinterpret_cast<uint4*>(&out_b[m * ldo + col0 + c]) = o;
        }
      }
      __syncwarp();
    }
    tc::fence_before_sync();
    __syncthreads();                                  // TMEM read and the A tile free before the next
  }
  cp_async_wait_all();                                // no copy left in flight at exit
  __syncthreads();
  if (warp == 0) tc::tmem_free(tmem, COLS);
}

// ------------------------------------------------------------------ weight gradient
// partial[block][no][k] = sum over this block's `rows` rows m of dY[m, no] X[m, k] (tensor
// cores, the row index is the MMA reduction dimension).
// A layer's operands are a few MB at the training sizes (64,000 edge rows of 288 bytes), so
// what bounds the kernel is how many SMs share the rows and how fast a block brings its
// rows in: the rows are split over up to kDwBlocks blocks (two an SM) in multiples of one
// 64-row tile, the tiles come by 16-byte cp.async into two buffers (the next one in flight
// during the MMAs), and both operands' fragments are read with ldmatrix.trans (the rows are
// the reduction dimension of both) from padded rows without bank conflicts. Eight warps:
// NO/16 row tiles of the result by 8/(NO/16) column groups, the accumulators in registers.
// With it a training step of a 3,200-particle 2D tank (64,000 edges) took 1.01 ms
// where blocks of 2048 rows with 2-byte loads took 14.7 ms, 15.9 ms of ncu time in this kernel.
// Most blocks of one weight gradient (their partial sums are kept): two for each of GB300's 152
// SMs, fixed, since a gradient's rounding follows the split.
constexpr int kDwBlocks = 304;

inline int64_t dw_rows(int64_t M) {       // rows per block
  const int64_t r = (M + kDwBlocks - 1) / kDwBlocks;
  return std::max<int64_t>(kTile, (r + kTile - 1) / kTile * kTile);
}

__device__ __forceinline__ void ldsm_x4_trans(uint32_t* r, const bf16* p) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(p);
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}

template <int NO, int K>
__global__ void __launch_bounds__(256)
k_dense_dw(int64_t M, int64_t rows, const bf16* __restrict__ dY, int ldy, const bf16* __restrict__ X, int ldx,
           float* __restrict__ partial) {
  constexpr int LDY = NO + 8, LDX = K + 8, kBuf = kTile * (LDY + LDX);
  constexpr int kMt = NO / 16, kGroups = 8 / kMt, kPairs = K / 16, kPer = (kPairs + kGroups - 1) / kGroups;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  bf16* sm = reinterpret_cast<bf16*>(smem_raw);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int mt = warp % kMt, group = warp / kMt;
  float acc[kPer][2][4];
#pragma unroll
  for (int q = 0; q < kPer; ++q)
#pragma unroll
    for (int h = 0; h < 2; ++h) acc[q][h][0] = acc[q][h][1] = acc[q][h][2] = acc[q][h][3] = 0.f;
  const int64_t r_begin = (int64_t)blockIdx.x * rows, r_end = min(r_begin + rows, M);
  auto load = [&](int buf, int64_t c0) {            // rows [c0, c0 + kTile), zeros past r_end
    bf16* d = sm + buf * kBuf;
    for (int idx = threadIdx.x; idx < kTile * (NO / 8); idx += 256) {
      const int r = idx / (NO / 8), c = idx % (NO / 8) * 8;
      const bool ok = c0 + r < r_end;
      cp_async16(d + r * LDY + c, dY + (ok ? c0 + r : r_begin) * ldy + c, ok);
    }
    d += kTile * LDY;
    for (int idx = threadIdx.x; idx < kTile * (K / 8); idx += 256) {
      const int r = idx / (K / 8), c = idx % (K / 8) * 8;
      const bool ok = c0 + r < r_end;
      cp_async16(d + r * LDX + c, X + (ok ? c0 + r : r_begin) * ldx + c, ok);
    }
    cp_async_commit();
  };
  load(0, r_begin);
  int buf = 0;
  for (int64_t c0 = r_begin; c0 < r_end; c0 += kTile, buf ^= 1) {
    cp_async_wait_all();
    __syncthreads();                                // this tile in place; the other buffer free
    if (c0 + kTile < r_end) load(buf ^ 1, c0 + kTile);
    const bf16* sY = sm + buf * kBuf;
    const bf16* sX = sY + kTile * LDY;
#pragma unroll
    for (int ks = 0; ks < kTile; ks += 16) {
      uint32_t a[4];
      ldsm_x4_trans(a, sY + (ks + (lane & 7) + (lane >> 4) * 8) * LDY + mt * 16 + ((lane >> 3) & 1) * 8);
#pragma unroll
      for (int q = 0; q < kPer; ++q) {
        const int p = group + q * kGroups;          // pair of 8-column tiles
        if (p >= kPairs) break;
        uint32_t b[4];
        ldsm_x4_trans(b, sX + (ks + (lane & 7) + ((lane >> 3) & 1) * 8) * LDX + p * 16 + (lane >> 4) * 8);
        mma16816(acc[q][0], a[0], a[1], a[2], a[3], b[0], b[1]);
        mma16816(acc[q][1], a[0], a[1], a[2], a[3], b[2], b[3]);
      }
    }
  }
  float* out = partial + (size_t)blockIdx.x * NO * K;
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    const int p = group + q * kGroups;
    if (p >= kPairs) break;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int r0 = mt * 16 + g, col = p * 16 + h * 8 + 2 * t;
      *reinterpret_cast<float2*>(&out[r0 * K + col]) = make_float2(acc[q][h][0], acc[q][h][1]);
      *reinterpret_cast<float2*>(&out[(r0 + 8) * K + col]) = make_float2(acc[q][h][2], acc[q][h][3]);
    }
  }
}

// grad[dst + o] += sum over blocks of partial[src + block count + o] for the weight gradients
// of several layers in one launch, each in a fixed order: eight warps take every eighth block
// of 32 consecutive outputs, then their sums are added in warp order. Counts are multiples of 32.
// A launch of its own for each layer left most of the chip idle (160 blocks) fifteen times a
// training step; the layers of a round share one.
struct DwSum {
  int blocks, count, dst;
  size_t src;
};
constexpr int kDwSums = 6;                // layers in one launch, at most
struct DwSums {
  DwSum job[kDwSums];
};
__global__ void __launch_bounds__(256)
k_reduce_partials(DwSums S, int jobs, const float* __restrict__ partial, float* __restrict__ grad) {
  __shared__ float red[8][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int at = blockIdx.x * 32, q = 0;
  while (q + 1 < jobs && at >= S.job[q].count) at -= S.job[q++].count;
  const DwSum j = S.job[q];
  const int o = at + lane;
  const float* p = partial + j.src;
  float s = 0.f;
#pragma unroll 8
  for (int b = warp; b < j.blocks; b += 8) s += p[(size_t)b * j.count + o];
  red[warp][lane] = s;
  __syncthreads();
  if (warp == 0) {
#pragma unroll
    for (int w = 1; w < 8; ++w) s += red[w][lane];
    grad[j.dst + o] += s;
  }
}

// ------------------------------------------------------------------ graph and features
// Edge CSR of the frozen neighbour table: node i owns edges [off[i], off[i+1]), fluid
// neighbours first, then walls; nbr >= 0 is a fluid slot, nbr < 0 encodes wall -1 - w.
__global__ void k_edge_count(int64_t n, const uint32_t* __restrict__ nbc, uint32_t* __restrict__ cnt) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) cnt[i] = (nbc[i] & 0xffffu) + (nbc[i] >> 16);
}

// Node features (one 32-byte row per particle).
template <int D>
__global__ void k_node_features(int64_t n, const int4* __restrict__ P, const float4* __restrict__ V,
                                const int* __restrict__ inst_of, const Inst* __restrict__ inst,
                                const Ctrl* __restrict__ ctrl, bf16* __restrict__ U) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int k = inst_of ? inst_of[i] : 0;
  const Inst& I = inst[k];
  const int4 pi = P[i];
  const float4 vi = V[i];
  const float inv_c0 = 1.0f / I.c0;
  const float uv[3] = {vi.x, vi.y, vi.z};
  __align__(16) bf16 u[16];
  for (int c = 0; c < 16; ++c) u[c] = __float2bfloat16_rn(0.f);
  for (int a = 0; a < D; ++a) u[a] = __float2bfloat16_rn(uv[a] * inv_c0);
  u[D] = __float2bfloat16_rn(S_RHO * (i2f(pi.w) / I.rho0));
  u[D + 1] = __float2bfloat16_rn((float)ctrl[k].dt_ad * I.c0 * I.inv_h);
  u[D + 2] = __float2bfloat16_rn(1.0f);
  uint4* dst = reinterpret_cast<uint4*>(U + i * 16);
  dst[0] = reinterpret_cast<const uint4*>(u)[0];
  dst[1] = reinterpret_cast<const uint4*>(u)[1];
}

// The edge list of the frozen table and each edge's static features, 16 bf16 per edge:
// [r_ij/h, (v_i - v_j)/c0, 100 dev_i, 100 dev_j, is_wall, 0...]; the rounds' input rows are
// assembled from them by k_edge_rows. A warp takes kEdgeNodes consecutive nodes, whose edges
// are consecutive, and its lanes take 32 of them at a time: the lists and rows are written
// in whole lines (a thread per node that walked its edges, and a second pass over the edges
// for the features, took 25 + 20 us for 2.7 M edges where this takes 27 us).
constexpr int kEdgeNodes = 4;
template <int D>
__global__ void k_edge_features(int64_t n, const int4* __restrict__ P, const float4* __restrict__ V,
                                const int* __restrict__ inst_of, const Inst* __restrict__ inst,
                                const int* __restrict__ nbr, const uint32_t* __restrict__ nbc,
                                const uint32_t* __restrict__ off, const int4* __restrict__ WP, int* __restrict__ esrc,
                                int* __restrict__ enbr, bf16* __restrict__ XS) {
  const int64_t i0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * kEdgeNodes;
  if (i0 >= n) return;
  uint32_t o[kEdgeNodes + 1];
#pragma unroll
  for (int k = 0; k <= kEdgeNodes; ++k) o[k] = off[min(i0 + k, n)];
  for (uint32_t e = o[0] + (threadIdx.x & 31); e < o[kEdgeNodes]; e += 32) {
    int k = 0;                                          // the last node whose edges begin at or before e
#pragma unroll
    for (int q = 1; q < kEdgeNodes; ++q) k += o[q] <= e;
    uint32_t first = o[0];
#pragma unroll
    for (int q = 1; q < kEdgeNodes; ++q) first = k == q ? o[q] : first;
    const int64_t i = i0 + k;
    const int s = (int)(e - first), nf = (int)(nbc[i] & 0xffffu);
    const bool wall = s >= nf;
    const int j = nbr[slot_index(n, i, wall ? wall_slot0(nf) + (s - nf) : s)];
    esrc[e] = (int)i;
    enbr[e] = wall ? -1 - j : j;
    const Inst& I = inst[inst_of ? inst_of[i] : 0];
    const int4 pi = P[i];
    const float4 vi = V[i];
    const int4 pj = wall ? WP[j] : P[j];
    float4 vj = make_float4(0.f, 0.f, 0.f, 0.f);
    float dev_j = 0.f;
    if (!wall) {
      vj = V[j];
      dev_j = i2f(pj.w) / I.rho0;
    }
    const float inv_c0 = 1.0f / I.c0;
    const int qi[3] = {pi.x, pi.y, pi.z}, qj[3] = {pj.x, pj.y, pj.z};
    const float ui[3] = {vi.x, vi.y, vi.z}, uj[3] = {vj.x, vj.y, vj.z};
    __align__(16) bf16 row[16];
    for (int c = 0; c < 16; ++c) row[c] = __float2bfloat16_rn(0.f);
    for (int a = 0; a < D; ++a) {
      row[a] = __float2bfloat16_rn((float)wrap_diff(qi[a] - qj[a], I.period[a]) * I.dq * I.inv_h);
      row[D + a] = __float2bfloat16_rn((ui[a] - uj[a]) * inv_c0);
    }
    row[2 * D] = __float2bfloat16_rn(S_RHO * (i2f(pi.w) / I.rho0));
    row[2 * D + 1] = __float2bfloat16_rn(S_RHO * dev_j);
    row[2 * D + 2] = __float2bfloat16_rn(wall ? 1.0f : 0.0f);
    uint4* dst = reinterpret_cast<uint4*>(XS + e * 16);
    dst[0] = reinterpret_cast<const uint4*>(row)[0];
    dst[1] = reinterpret_cast<const uint4*>(row)[1];
  }
}

// Round input row of edge e: XE[e] = [static features (fe) | bf16(h_j) (64, zero for a
// wall) | 1 | 0...] (80 columns). One thread per 16-byte piece: consecutive threads write
// consecutive pieces.
__global__ void k_edge_rows(int64_t E, int fe, const bf16* __restrict__ XS, const int* __restrict__ enbr,
                            const float* __restrict__ H, bf16* __restrict__ XE) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= E * 10) return;
  const int64_t e = idx / 10;
  const int c0 = (int)(idx - e * 10) * 8;
  const int j = enbr[e];
  __align__(16) bf16 v[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int c = c0 + k;
    float x = 0.f;
    if (c < fe) x = __bfloat162float(XS[e * 16 + c]);
    else if (c < fe + F) x = j >= 0 ? H[(int64_t)j * F + (c - fe)] : 0.f;
    else if (c == fe + F) x = 1.0f;
    v[k] = __float2bfloat16_rn(x);
  }
  *reinterpret_cast<uint4*>(XE + e * 80 + c0) = *reinterpret_cast<const uint4*>(v);
}

// XN[i] = [bf16(h_i), bf16(a_i), 1], a_i = (1/nbar) sum over node i's edges of M
__global__ void k_segsum(int64_t n, const uint32_t* __restrict__ off, const float* __restrict__ Mm,
                         const float* __restrict__ H, float inv_nbar, bf16* __restrict__ XN) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n * F) return;
  const int64_t i = idx / F;
  const int f = (int)(idx % F);
  float s = 0.f;
  const uint32_t end = off[i + 1];
  for (uint32_t e = off[i]; e < end; e += 8) {        // eight rows in flight; +0 changes no sum
    float v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = e + k < end ? Mm[(int64_t)(e + k) * F + f] : 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) s += v[k];
  }
  XN[i * 144 + f] = __float2bfloat16_rn(H[i * F + f]);
  XN[i * 144 + F + f] = __float2bfloat16_rn(s * inv_nbar);
}

// Edge network of one round, fused for inference. Each warp takes a run of nodes and walks
// their edges in 32-row tiles. A tile's rows are assembled as k_edge_rows lays a round input
// row out (static features, bf16(h_j) or zero for a wall, the bias 1, zero padding) in one
// of the warp's two buffers: 16-byte pieces of the neighbours' row templates (see
// k_node_templates) by cp.async, and the one piece that holds static features and node state
// merged in registers, all one tile ahead of the products, the neighbour indices two. Both
// edge layers run on the tensor cores (mma.sync m16n8k16, k-steps in k_dense's order; the
// first layer's accumulators become the second layer's A fragments after k_dense's ReLU
// and bfloat16 rounding), and the messages are added per node in edge order as k_segsum
// does. After its edges, the run's node rows go through the node network (both node
// layers, the update added to h) into the other node-state buffer and, as the next round's
// templates (after the last round the decoder's input rows), into Tout. The new node states
// are therefore bit-identical to the unfused path's, and no per-edge row, activation or
// message goes to memory.
// What bounds it: the shared-memory pipe. A warp reads 20 KB of weight fragments per tile,
// so a tile has 32 rows, whose two m16 halves share them, and the operands are read by
// ldmatrix from bf16 rows; with 16-row tiles of FP32 node states, converted element by
// element, the pipe moved about twice the bytes for a row and took 263 us a round
// at 100,128 particles (2.7 M edges) against 154 us now, at 68 % of the pipe and 49 % of the
// mma.sync rate; 12 warps with 168 registers 170 us, 14 that spill 181 us.
constexpr int kFuseWarps = 16;                // one block an SM, 128 registers a thread
constexpr int kFuseRun = 64;                  // nodes in a run, at most (their edge offsets stay in two registers)
constexpr int kFuseRunMin = 4;
constexpr int kFuseBuf = 32 * 80;             // bf16 elements of one tile buffer
constexpr int kMsgLd = 40;                    // message row stride: 32 columns + pad, conflict-free float2 stores

static_assert(32 * kMsgLd * sizeof(float) <= kFuseBuf * sizeof(bf16), "32 columns of messages must fit a tile buffer");

inline size_t fused_smem() {
  return (size_t)(3 * 64 * 80 + 64 * 144 + kFuseWarps * 2 * kFuseBuf) * sizeof(bf16);
}

// Column c of row r in a row-major operand of 80 or 144 columns: pieces of 8 columns trade
// places in pairs in every second group of four rows, so that the eight rows of an ldmatrix
// (10 or 18 pieces apart) lie in different banks without padding.
__device__ __forceinline__ int fuse_at(int ld, int r, int c) { return r * ld + (c ^ ((r & 4) << 1)); }

__device__ __forceinline__ void ldsm_x4(uint32_t a, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(a)
               : "memory");
}

// This lane's ldmatrix address in an [n][ld] weight copy, and the B fragments of two n-tiles
// (nt, nt + 1) at k-step k0 read with it: lane i addresses row i % 8 of 8x8 matrix i / 8
// (matrices: (nt, k0), (nt, k0 + 8), (nt + 1, k0), (nt + 1, k0 + 8)), and receives row
// lane / 4, columns 2 (lane % 4), +1 of each, which is the m16n8k16 B fragment.
__device__ __forceinline__ uint32_t b_lane(const bf16* W, int ld, int lane) {
  return tc::smem_u32(W + fuse_at(ld, (lane >> 4) * 8 + (lane & 7), ((lane >> 3) & 1) * 8));
}
template <int LD = 80>
__device__ __forceinline__ void ldsm_b4(uint32_t base, int nt, int k0, uint32_t& b0, uint32_t& b1, uint32_t& c0,
                                        uint32_t& c1) {
  ldsm_x4(base + (nt * 8 * LD + k0) * 2, b0, b1, c0, c1);
}

// The same for the A fragments of rows r0 .. r0 + 15 of an [.][80] tile: matrices (rows 0..7,
// k0), (rows 8..15, k0), (rows 0..7, k0 + 8), (rows 8..15, k0 + 8)
__device__ __forceinline__ uint32_t a_lane(const bf16* X, int lane) {
  return tc::smem_u32(X + fuse_at(80, lane & 15, (lane >> 4) * 8));
}
__device__ __forceinline__ void ldsm_a4(uint32_t base, int r0, int k0, uint32_t* r) {
  ldsm_x4(base + (r0 * 80 + k0) * 2, r[0], r[1], r[2], r[3]);
}

// bf16(relu(lo)), bf16(relu(hi)): rounded by one packed conversion, then clamped (rounding
// keeps the sign; a NaN becomes 0 as under fmaxf)
__device__ __forceinline__ uint32_t relu2(float lo, float hi) {
  const __nv_bfloat162 v = __hmax2(__floats2bfloat162_rn(lo, hi), __floats2bfloat162_rn(0.f, 0.f));
  return *reinterpret_cast<const uint32_t*>(&v);
}

// A fragments of the layer after a 64-wide one, from its accumulators: [bf16(relu(z)), 1, 0...]
__device__ __forceinline__ void relu_frags(const float (*acc)[4], uint32_t (*A)[4]) {
#pragma unroll
  for (int kk = 0; kk < 4; ++kk) {
    const float* lo = acc[2 * kk];
    const float* hi = acc[2 * kk + 1];
    A[kk][0] = relu2(lo[0], lo[1]);
    A[kk][1] = relu2(lo[2], lo[3]);
    A[kk][2] = relu2(hi[0], hi[1]);
    A[kk][3] = relu2(hi[2], hi[3]);
  }
}

// read-only loads that stay where they are written: issued a tile before their use, and not
// moved down to it
__device__ __forceinline__ uint4 ld_early(const uint4* p) {
  uint4 v;
  asm volatile("ld.global.nc.v4.u32 {%0,%1,%2,%3}, [%4];\n" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}
__device__ __forceinline__ uint32_t ld_early(const uint16_t* p) {
  uint32_t v;
  asm volatile("ld.global.nc.u16 %0, [%1];\n" : "=r"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ int ld_early(const int* p) {
  int v;
  asm volatile("ld.global.nc.s32 %0, [%1];\n" : "=r"(v) : "l"(p));
  return v;
}

// Templates T: row 0 serves wall neighbours, row j + 1 fluid node j. Tout: row i at
// 80 i, its 64 node-state columns at ocol (then the bias 1, zeros elsewhere); with ocol > 0
// it is the next round's templates, whose row 0 (at -80) is written too.
template <int FE>
__global__ void __launch_bounds__(kFuseWarps * 32, 1)
k_edge_round_fused(int64_t n, int run, const uint32_t* __restrict__ off, const bf16* __restrict__ XS,
                   const int* __restrict__ enbr, const float* __restrict__ H, const bf16* __restrict__ T,
                   const bf16* __restrict__ W1, const bf16* __restrict__ W2, const bf16* __restrict__ Wn1,
                   const bf16* __restrict__ Wn2, float inv_nbar, bf16* __restrict__ XN, float* __restrict__ Hout,
                   bf16* __restrict__ Tout, int ocol) {
  constexpr int MP = FE / 8;                  // the piece of static features and node state
  static_assert((FE == 7 || FE == 9) && FE + F + 1 <= 8 * (MP + 9), "pieces MP + 1 .. MP + 8 hold the rest of a row");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  bf16* sW1 = reinterpret_cast<bf16*>(smem_raw);
  bf16* sW2 = sW1 + 64 * 80;
  bf16* sN2 = sW2 + 64 * 80;                  // node layer 2
  bf16* sN1 = sN2 + 64 * 80;                  // node layer 1, 144 columns
  bf16* buf = sN1 + 64 * 144 + warp * 2 * kFuseBuf;
  for (int idx = threadIdx.x; idx < 64 * 10; idx += blockDim.x) {
    const int r = idx / 10, c = (idx % 10) * 8, o = fuse_at(80, r, c);
    *reinterpret_cast<uint4*>(&sW1[o]) = *reinterpret_cast<const uint4*>(&W1[r * 80 + c]);
    *reinterpret_cast<uint4*>(&sW2[o]) = *reinterpret_cast<const uint4*>(&W2[r * 80 + c]);
    *reinterpret_cast<uint4*>(&sN2[o]) = *reinterpret_cast<const uint4*>(&Wn2[r * 80 + c]);
  }
  for (int idx = threadIdx.x; idx < 64 * 18; idx += blockDim.x) {
    const int r = idx / 18, c = (idx % 18) * 8;
    *reinterpret_cast<uint4*>(&sN1[fuse_at(144, r, c)]) = *reinterpret_cast<const uint4*>(&Wn1[r * 144 + c]);
  }
  __syncthreads();
  if (ocol > 0 && blockIdx.x == 0 && threadIdx.x < 80)   // the wall template of the next round
    Tout[(int)threadIdx.x - 80] = __float2bfloat16_rn((int)threadIdx.x == ocol + F ? 1.0f : 0.f);
  const uint32_t w1_base = b_lane(sW1, 80, lane), n1_base = b_lane(sN1, 144, lane), a_base = a_lane(buf, lane);
  const uint32_t bias = t == 0 ? pack2(__float2bfloat16_rn(1.0f), __float2bfloat16_rn(0.f)) : 0u;
  const int64_t runs = (n + run - 1) / run;
  // few runs: over the blocks first, then over a block's warps
  for (int64_t rr = (int64_t)warp * gridDim.x + blockIdx.x; rr < runs; rr += (int64_t)gridDim.x * kFuseWarps) {
    const int64_t i0 = rr * run, i1 = min(i0 + (int64_t)run, n);
    const int nodes = (int)(i1 - i0);
    const uint32_t e_begin = off[i0], e_end = off[i1];
    // ends of the run's nodes: node k in lane k % 32 of register k / 32
    const uint32_t endA = off[min(i0 + lane + 1, i1)], endB = off[min(i0 + lane + 33, i1)];
    auto end_of = [&](int k) {
      const uint32_t a = __shfl_sync(0xffffffffu, endA, k & 31), b = __shfl_sync(0xffffffffu, endB, k & 31);
      return k < 32 ? a : b;
    };
    // The open node and, per half of the 64 columns, its sum in column 32 half + lane. Nodes
    // that end at or before edge e are closed (edgeless ones included); both halves pass the
    // same nodes, so the second returns to where the first began.
    int cur = 0;
    uint32_t cur_end = end_of(0);
    float sum[2] = {0.f, 0.f};
    auto close_until = [&](uint32_t e, int half) {
      while (cur < nodes && cur_end <= e) {
        XN[(i0 + cur) * 144 + F + 32 * half + lane] = __float2bfloat16_rn(sum[half] * inv_nbar);
        sum[half] = 0.f;
        ++cur;
        cur_end = end_of(cur & 63);           // past the run's last node: not used
      }
    };
    // neighbour of edge t0 + lane (not worked on until its use, a tile later); rows past the
    // end repeat the last edge
    auto idx_of = [&](uint32_t t0) { return ld_early(&enbr[min(t0 + lane, e_end - 1)]); };
    // this lane's row: piece MP and the one element of it that comes from the other source
    // (7 static features: XS and element 7 of T; 9: T and element 0 of XS)
    uint4 mq;
    uint32_t me;
    auto load_tile = [&](uint32_t t0, int nb, bf16* dst) {
      const int jrow = max(nb, -1) + 1;       // template row
#pragma unroll
      for (int p = 0; p < 8; ++p) {
        const int row = 4 * p + (lane >> 3), c = (MP + 1 + (lane & 7)) * 8;
        const int j = __shfl_sync(0xffffffffu, jrow, row);
        cp_async16(dst + fuse_at(80, row, c), T + (int64_t)j * 80 + c, true);
      }
      const bf16* x = XS + (int64_t)min(t0 + lane, e_end - 1) * 16;
      if (MP) cp_async16(dst + fuse_at(80, lane, 0), x, true);
      cp_async_commit();
      const bf16* tj = T + (int64_t)jrow * 80 + MP * 8;
      mq = ld_early(reinterpret_cast<const uint4*>(MP ? tj : x));
      me = ld_early(reinterpret_cast<const uint16_t*>(MP ? x + 8 : tj + 7));
    };
    int jn = 0;
    if (e_begin < e_end) {
      load_tile(e_begin, idx_of(e_begin), buf);
      jn = idx_of(e_begin + 32);
    }
    int par = 0;
    for (uint32_t t0 = e_begin; t0 < e_end; t0 += 32, par ^= 1) {
      bf16* tile = buf + par * kFuseBuf;
      if (MP) mq.x = (mq.x & 0xffff0000u) | me;
      else mq.w = (mq.w & 0x0000ffffu) | (me << 16);
      *reinterpret_cast<uint4*>(&tile[fuse_at(80, lane, MP * 8)]) = mq;
      if (MP == 0) *reinterpret_cast<uint4*>(&tile[fuse_at(80, lane, 72)]) = make_uint4(0u, 0u, 0u, 0u);
      cp_async_wait_all();
      __syncwarp();
      // next tile's rows in flight during this tile's products
      if (t0 + 32 < e_end) {
        load_tile(t0 + 32, jn, buf + (par ^ 1) * kFuseBuf);
        jn = idx_of(t0 + 64);
      }
      const uint32_t at = a_base + par * kFuseBuf * 2;
      float acc[2][8][4];
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) acc[q][nt][0] = acc[q][nt][1] = acc[q][nt][2] = acc[q][nt][3] = 0.f;
#pragma unroll
      for (int kk = 0; kk < 5; ++kk) {
        uint32_t A0[4], A1[4];
        ldsm_a4(at, 0, kk * 16, A0);
        ldsm_a4(at, 16, kk * 16, A1);
#pragma unroll
        for (int nt = 0; nt < 8; nt += 2) {
          uint32_t b0, b1, c0, c1;
          ldsm_b4(w1_base, nt, kk * 16, b0, b1, c0, c1);
          mma16816(acc[0][nt], A0[0], A0[1], A0[2], A0[3], b0, b1);
          mma16816(acc[0][nt + 1], A0[0], A0[1], A0[2], A0[3], c0, c1);
          mma16816(acc[1][nt], A1[0], A1[1], A1[2], A1[3], b0, b1);
          mma16816(acc[1][nt + 1], A1[0], A1[1], A1[2], A1[3], c0, c1);
        }
      }
      uint32_t Z[2][4][4];
      relu_frags(acc[0], Z[0]);
      relu_frags(acc[1], Z[1]);
      // second layer and the messages, 32 columns at a time, through the tile's buffer
      float* sM = reinterpret_cast<float*>(tile);
      const int cur0 = cur;
      const uint32_t cur_end0 = cur_end;
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        float out[2][4][4];
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
          for (int nt = 0; nt < 4; ++nt) out[q][nt][0] = out[q][nt][1] = out[q][nt][2] = out[q][nt][3] = 0.f;
#pragma unroll
        for (int kk = 0; kk < 5; ++kk)
#pragma unroll
          for (int nt = 0; nt < 4; nt += 2) {
            uint32_t b0, b1, c0, c1;
            ldsm_b4(w1_base + 64 * 80 * 2, 4 * half + nt, kk * 16, b0, b1, c0, c1);
#pragma unroll
            for (int q = 0; q < 2; ++q) {
              const uint32_t a0 = kk < 4 ? Z[q][kk & 3][0] : bias, a1 = kk < 4 ? Z[q][kk & 3][1] : bias;
              const uint32_t a2 = kk < 4 ? Z[q][kk & 3][2] : 0u, a3 = kk < 4 ? Z[q][kk & 3][3] : 0u;
              mma16816(out[q][nt], a0, a1, a2, a3, b0, b1);
              mma16816(out[q][nt + 1], a0, a1, a2, a3, c0, c1);
            }
          }
        __syncwarp();                         // layer 1's rows, or the first half's messages, read
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
          for (int nt = 0; nt < 4; ++nt) {
            float* m = &sM[(16 * q + g) * kMsgLd + nt * 8 + 2 * t];
            *reinterpret_cast<float2*>(m) = make_float2(out[q][nt][0], out[q][nt][1]);
            *reinterpret_cast<float2*>(m + 8 * kMsgLd) = make_float2(out[q][nt][2], out[q][nt][3]);
          }
        __syncwarp();
        cur = cur0;
        cur_end = cur_end0;
        const int rows = (int)min(32u, e_end - t0);
        for (int r = 0; r < rows;) {
          close_until(t0 + (uint32_t)r, half);
          // rows r .. r1 - 1 belong to the open node
          const int r1 = (int)min((uint32_t)rows, cur_end - t0);
          for (; r + 8 <= r1; r += 8) {
            float v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = sM[(r + k) * kMsgLd + lane];
#pragma unroll
            for (int k = 0; k < 8; ++k) sum[half] += v[k];
          }
          if (r < r1) {                       // +0 leaves a sum that started at +0 unchanged, bit for bit
            float v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = sM[min(r + k, 31) * kMsgLd + lane];
#pragma unroll
            for (int k = 0; k < 8; ++k) sum[half] += r + k < r1 ? v[k] : 0.f;
            r = r1;
          }
        }
      }
      __syncwarp();                           // the buffer is free for the tile after the next
    }
    {
      const int cur0 = cur;
      const uint32_t cur_end0 = cur_end;
      close_until(e_end, 0);
      cur = cur0;
      cur_end = cur_end0;
      close_until(e_end, 1);
    }
    __syncwarp();                             // the run's sums in XN, written above, visible
    // node network of the run, 16 nodes at a time, as the unfused node layers compute it:
    // z = relu(W_n1 [h, a, 1]), h_out = h + W_n2 [z, 1]
    for (int m0 = 0; m0 < nodes; m0 += 16) {
      const int64_t ib = i0 + m0;
      const int left = nodes - m0;
      const bool vg = g < left, vh = g + 8 < left;
      const float* hg = H + (ib + (vg ? g : 0)) * F;
      const float* hh = H + (ib + (vh ? g + 8 : 0)) * F;
      const bf16* xg = XN + (ib + (vg ? g : 0)) * 144;
      const bf16* xh = XN + (ib + (vh ? g + 8 : 0)) * 144;
      auto state = [&](const float* p) {
        const float2 v = *reinterpret_cast<const float2*>(p);
        return pack2(__float2bfloat16_rn(v.x), __float2bfloat16_rn(v.y));
      };
      uint32_t A[9][4];
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        const int c = kk * 16 + 2 * t;
        A[kk][0] = state(hg + c);
        A[kk][1] = state(hh + c);
        A[kk][2] = state(hg + c + 8);
        A[kk][3] = state(hh + c + 8);
        A[kk + 4][0] = ld_u32(xg + F + c);
        A[kk + 4][1] = ld_u32(xh + F + c);
        A[kk + 4][2] = ld_u32(xg + F + c + 8);
        A[kk + 4][3] = ld_u32(xh + F + c + 8);
      }
      A[8][0] = A[8][1] = bias;
      A[8][2] = A[8][3] = 0u;
      float acc[8][4];
#pragma unroll
      for (int nt = 0; nt < 8; ++nt) acc[nt][0] = acc[nt][1] = acc[nt][2] = acc[nt][3] = 0.f;
#pragma unroll
      for (int kk = 0; kk < 9; ++kk)
#pragma unroll
        for (int nt = 0; nt < 8; nt += 2) {
          uint32_t b0, b1, c0, c1;
          ldsm_b4<144>(n1_base, nt, kk * 16, b0, b1, c0, c1);
          mma16816(acc[nt], A[kk][0], A[kk][1], A[kk][2], A[kk][3], b0, b1);
          mma16816(acc[nt + 1], A[kk][0], A[kk][1], A[kk][2], A[kk][3], c0, c1);
        }
      uint32_t Z[4][4];
      relu_frags(acc, Z);
      float out[8][4];
#pragma unroll
      for (int nt = 0; nt < 8; ++nt) out[nt][0] = out[nt][1] = out[nt][2] = out[nt][3] = 0.f;
#pragma unroll
      for (int kk = 0; kk < 5; ++kk) {
        const uint32_t a0 = kk < 4 ? Z[kk & 3][0] : bias, a1 = kk < 4 ? Z[kk & 3][1] : bias;
        const uint32_t a2 = kk < 4 ? Z[kk & 3][2] : 0u, a3 = kk < 4 ? Z[kk & 3][3] : 0u;
#pragma unroll
        for (int nt = 0; nt < 8; nt += 2) {
          uint32_t b0, b1, c0, c1;
          ldsm_b4(w1_base + 2 * 64 * 80 * 2, nt, kk * 16, b0, b1, c0, c1);
          mma16816(out[nt], a0, a1, a2, a3, b0, b1);
          mma16816(out[nt + 1], a0, a1, a2, a3, c0, c1);
        }
      }
      // new states out; their rows of Tout through the buffer
#pragma unroll
      for (int nt = 0; nt < 8; ++nt) {
        const int c = nt * 8 + 2 * t;
        const float2 ha = *reinterpret_cast<const float2*>(hg + c), hb = *reinterpret_cast<const float2*>(hh + c);
        const float2 na = make_float2(ha.x + out[nt][0], ha.y + out[nt][1]);
        const float2 nb = make_float2(hb.x + out[nt][2], hb.y + out[nt][3]);
        if (vg) *reinterpret_cast<float2*>(&Hout[(ib + g) * F + c]) = na;
        if (vh) *reinterpret_cast<float2*>(&Hout[(ib + g + 8) * F + c]) = nb;
        buf[fuse_at(80, g, ocol + c)] = __float2bfloat16_rn(na.x);
        buf[fuse_at(80, g, ocol + c + 1)] = __float2bfloat16_rn(na.y);
        buf[fuse_at(80, g + 8, ocol + c)] = __float2bfloat16_rn(nb.x);
        buf[fuse_at(80, g + 8, ocol + c + 1)] = __float2bfloat16_rn(nb.y);
      }
      // the 16 other columns: static features (zero), bias, padding
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int r = 2 * k + (lane >> 4), q = lane & 15, c = q < ocol ? q : F + q;
        buf[fuse_at(80, r, c)] = __float2bfloat16_rn(c == ocol + F ? 1.0f : 0.f);
      }
      __syncwarp();
      for (int idx = lane; idx < min(left, 16) * 10; idx += 32) {
        const int r = idx / 10, c = (idx - r * 10) * 8;
        *reinterpret_cast<uint4*>(&Tout[(ib + r) * 80 + c]) = *reinterpret_cast<const uint4*>(&buf[fuse_at(80, r, c)]);
      }
      __syncwarp();
    }
  }
}

// ------------------------------------------------------------------ fused edge round, pipelined (tcgen05)
// Round input row templates: row j + 1 is edge row [XS | bf16(h_j) | 1 | 0...] of any edge
// whose neighbour is fluid node j, with zeros where the static features go; row 0 serves
// wall neighbours (h = 0). An edge row is its neighbour's template with the static features
// merged into the first one or two 16-byte pieces. Threads past the templates (the pipelined
// form launches them) write the h part of the round's node rows, XN[i][0, 64) = bf16(h_i).
// One thread per 16-byte piece.
template <int FE>
__global__ void k_node_templates(int64_t n, const float* __restrict__ H, bf16* __restrict__ T,
                                 bf16* __restrict__ XN) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  __align__(16) bf16 v[8];
  if (idx < (n + 1) * 10) {
    const int64_t row = idx / 10, j = row - 1;
    const int c0 = (int)(idx - row * 10) * 8;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int c = c0 + k;
      float x = 0.f;
      if (c >= FE && c < FE + F) x = j >= 0 ? H[j * F + (c - FE)] : 0.f;
      else if (c == FE + F) x = 1.0f;
      v[k] = __float2bfloat16_rn(x);
    }
    *reinterpret_cast<uint4*>(T + row * 80 + c0) = *reinterpret_cast<const uint4*>(v);
  } else if (idx < (n + 1) * 10 + n * 8) {
    const int64_t q = idx - (n + 1) * 10, i = q / 8;
    const int c0 = (int)(q - i * 8) * 8;
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = __float2bfloat16_rn(H[i * F + c0 + k]);
    *reinterpret_cast<uint4*>(XN + i * 144 + c0) = *reinterpret_cast<const uint4*>(v);
  }
}

// Edge network of one round for inference on the fifth-generation tensor cores, as a
// warp-specialised pipeline. Each CTA takes runs of at most kWsRun consecutive nodes and
// walks their edges in 128-row tiles through a ring of kWsStages tile buffers:
//   warp 4 + p (producer p) assembles the tiles t with t % kWsStages == p in buffer p:
//     pieces of the neighbours' templates by cp.async, the static features merged into
//     the first pieces by plain stores; it signals a tile as soon as its copies have landed;
//   warp 4 + kWsStages (one issuing lane) runs layer 1 of tile t + 1 into TMEM accumulator set
//     (t + 1) % 2 before layer 2 of tile t, each as K/16 tcgen05.mma (M = 128, N = 64)
//     committed to an mbarrier; layer 2's commit also frees the tile buffer;
//   warps 0-3 (epilogue, one TMEM lane = one edge row per thread) turn layer 1's
//     accumulators of tile t into bf16(relu(z)) and the constant columns, written over the
//     tile's own buffer as layer 2's A operand; then, while layer 2 of tile t runs, they
//     stage the messages of tile t - 1 32 columns at a time and add them per node in edge
//     order (a node whose edges continue into the next tile carries its partial sums);
//     closed nodes write XN[i][64, 128) = bf16(a_i).
// Every product, rounding and sum is the layer-by-layer path's, so XN is bit-identical to
// it; the node layers then run as that path's dense layers. Every wait is bounded: one that
// runs out sets ERR_TIMEOUT in *err and makes every role stop. On GB300 this pipeline ran
// the 100,128-particle learned step in 1.17 ms against 1.15 ms for the warp-level MMA rounds
// (k_edge_round_fused) of 16-row tiles, since 0.80 ms with tiles of 32: the epilogue warpgroup's per-node sums and operand conversion,
// not the tensor core, bound it, so inference keeps the warp-level rounds by default.
constexpr int kWsStages = 3;
constexpr int kWsThreads = 128 + 32 * kWsStages + 32;   // warps 0-3 epilogue, one producer per buffer, MMA
constexpr int kWsMmaWarp = 4 + kWsStages;
constexpr int kWsRun = 128;                   // nodes in a run, at most
constexpr int kWsTile = 128 * 80 * 2;         // bytes of one 128-row tile of edge rows
constexpr int kWsMsgLd = 36;                  // staged message row: 32 floats + pad (16-byte rows, conflict-free)

inline size_t ws_smem() {
  // at least a third of an SM's shared memory, so that no more than two CTAs (256 TMEM
  // columns each) share an SM and a TMEM allocation never waits
  const size_t need = (size_t)2 * 64 * 80 * 2 + (size_t)kWsStages * kWsTile + 128 * kWsMsgLd * sizeof(float) +
                      2 * 64 * sizeof(float) + (kWsRun + 1) * sizeof(uint32_t);
  return std::max(need, (size_t)233472 / 3 + 1);
}

struct WsSync {
  uint64_t full[kWsStages], empty[kWsStages];   // tile buffer written / free again
  uint64_t a1_full[2], a1_empty[2];             // layer-1 accumulators ready / read
  uint64_t a2_ready[2];                         // layer 2's operand written
  uint64_t a2_full[2], a2_empty[2];             // layer-2 accumulators ready / read
  uint64_t fin;                                 // every MMA of the CTA complete
  int abort;
};

__device__ __forceinline__ void ws_bar_init(uint64_t* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(tc::smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void ws_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(tc::smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void ws_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(tc::smem_u32(bar))
               : "memory");
}
// Bounded wait for the phase of parity `parity`; gives up when another role has aborted,
// and aborts every role when it runs out itself.
__device__ __forceinline__ bool ws_wait(uint64_t* bar, uint32_t parity, volatile int* abort, int* err) {
  for (unsigned spin = 0; spin < tc::kWaitLimit; ++spin) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done)
        : "r"(tc::smem_u32(bar)), "r"(parity)
        : "memory");
    if (done) return true;
    if (*abort) return false;
  }
  *abort = 1;
  atomicOr(err, ERR_TIMEOUT);
  return false;
}
// AND of a flag over the epilogue warpgroup (named barrier 1, 128 threads): the same
// decision in every epilogue thread
__device__ __forceinline__ bool epi_all(bool v) {
  int r;
  asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\tbar.red.and.pred q, 1, 128, p;\n\t"
               "selp.s32 %0, 1, 0, q;\n\t}\n"
               : "=r"(r)
               : "r"((int)v)
               : "memory");
  return r != 0;
}
__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, 128;\n" ::: "memory"); }
__device__ __forceinline__ float ld_shared_f32(uint32_t addr) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];\n" : "=f"(v) : "r"(addr) : "memory");
  return v;
}
// number of epilogue threads whose flag is set (named barrier 1, 128 threads)
__device__ __forceinline__ int epi_count(bool v) {
  int r;
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %1, 0;\n\tbar.red.popc.u32 %0, 1, 128, p;\n\t}\n"
               : "=r"(r)
               : "r"((int)v)
               : "memory");
  return r;
}

template <int FE>
__global__ void __launch_bounds__(kWsThreads, 2)
k_edge_round_ws(int64_t n, int run, const uint32_t* __restrict__ off, const bf16* __restrict__ XS,
                const int* __restrict__ enbr, const bf16* __restrict__ T, const bf16* __restrict__ W1,
                const bf16* __restrict__ W2, float inv_nbar, bf16* __restrict__ XN, int* __restrict__ err) {
  constexpr int MP = (FE + 7) / 8;                    // leading pieces that hold static features
  extern __shared__ __align__(128) unsigned char tc_smem[];
  __shared__ WsSync S;
  __shared__ uint32_t tmem_slot;
  __shared__ int carry_open;
  unsigned char* sW1 = tc_smem;                       // 64 x 80
  unsigned char* sW2 = sW1 + 64 * 80 * 2;             // 64 x 80
  unsigned char* sTiles = sW2 + 64 * 80 * 2;          // kWsStages x (128 x 80)
  float* stage = reinterpret_cast<float*>(sTiles + kWsStages * kWsTile);   // 128 x 32 messages
  float* carry_in = stage + 128 * kWsMsgLd;           // partial sums of the node carried into the tile
  float* carry_out = carry_in + 64;                   // ... and of the node it leaves open
  uint32_t* soff = reinterpret_cast<uint32_t*>(carry_out + 64);   // the run's edge offsets
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tid = threadIdx.x;
  load_operand(sW1, 64, 80, W1, 80, 64);
  load_operand(sW2, 64, 80, W2, 80, 64);
  if (tid == 0) {
    for (int s = 0; s < kWsStages; ++s) {
      ws_bar_init(&S.full[s], 1);
      ws_bar_init(&S.empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      ws_bar_init(&S.a1_full[b], 1);
      ws_bar_init(&S.a1_empty[b], 4);             // one arrival per epilogue warp
      ws_bar_init(&S.a2_ready[b], 4);
      ws_bar_init(&S.a2_full[b], 1);
      ws_bar_init(&S.a2_empty[b], 4);
    }
    ws_bar_init(&S.fin, 1);
    S.abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 0) tc::tmem_alloc(&tmem_slot, 256);
  tc::fence_to_async();                               // the weights, for the tensor core
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tmem_slot;                    // acc1[b] at 64 b, acc2[b] at 128 + 64 b
  volatile int* abort = &S.abort;
  const int64_t runs = (n + run - 1) / run;

  if (warp >= 4 && warp < kWsMmaWarp) {
    // ---------------- producers: warp 4 + p assembles the tiles t with t % kWsStages == p,
    // always into buffer p, and signals each as soon as its copies have landed
    const int p = warp - 4;
    uint32_t t = 0;
    bool ok = true;
    for (int64_t rr = blockIdx.x; rr < runs && ok; rr += gridDim.x) {
      const int64_t i0 = rr * run, i1 = min(i0 + (int64_t)run, n);
      const uint32_t E0 = __ldg(&off[i0]), E1 = __ldg(&off[i1]);
      for (uint32_t e0 = E0; e0 < E1; e0 += 128, ++t) {
        if ((int)(t % kWsStages) != p) continue;
        const bool got = ws_wait(&S.empty[p], ((t / kWsStages) & 1u) ^ 1u, abort, err);
        if (!__all_sync(0xffffffffu, got)) {
          ok = false;
          break;
        }
        const uint32_t te = min(e0 + 128u, E1);
        unsigned char* A = sTiles + p * kWsTile;
        // rows lane + 32 k: every load of the tile issued before any is used
        int jr[4];
        bool vr[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const uint32_t e = e0 + (uint32_t)(lane + 32 * k);
          vr[k] = e < te;
          const int j = vr[k] ? __ldg(&enbr[e]) : 0;
          jr[k] = max(j, -1) + 1;                     // row 0: the walls' template
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const bf16* tj = T + (int64_t)jr[k] * 80;
#pragma unroll
          for (int q = MP; q < 10; ++q)
            cp_async16(A + tc::core_offset(128, lane + 32 * k, q * 8), vr[k] ? tj + q * 8 : T, vr[k]);
        }
        uint4 q[4][MP], x[4][MP];
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
          for (int c = 0; c < MP; ++c) {
            q[k][c] = x[k][c] = make_uint4(0u, 0u, 0u, 0u);
            if (vr[k]) {
              q[k][c] = __ldg(reinterpret_cast<const uint4*>(T + (int64_t)jr[k] * 80) + c);
              x[k][c] = __ldg(reinterpret_cast<const uint4*>(XS + (int64_t)(e0 + lane + 32 * k) * 16) + c);
            }
          }
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
          for (int c = 0; c < MP; ++c) {
            bf16* a = reinterpret_cast<bf16*>(&q[k][c]);
            const bf16* xa = reinterpret_cast<const bf16*>(&x[k][c]);
#pragma unroll
            for (int m = 0; m < 8; ++m)
              if (c * 8 + m < FE) a[m] = xa[m];
            *reinterpret_cast<uint4*>(A + tc::core_offset(128, lane + 32 * k, c * 8)) = q[k][c];
          }
        cp_async_commit();
        cp_async_wait_all();
        tc::fence_to_async();
        __syncwarp();                                 // the warp's copies and stores, then one arrival
        if (lane == 0) ws_arrive(&S.full[p]);
      }
    }
    cp_async_wait_all();
  } else if (warp == kWsMmaWarp) {
    // ---------------- MMA issue (all lanes wait, lane 0 issues)
    uint32_t TT = 0;
    for (int64_t rr = blockIdx.x; rr < runs; rr += gridDim.x) {
      const int64_t i0 = rr * run, i1 = min(i0 + (int64_t)run, n);
      const uint32_t E0 = __ldg(&off[i0]), E1 = __ldg(&off[i1]);
      TT += (E1 - E0 + 127u) / 128u;
    }
    const uint32_t w1 = tc::smem_u32(sW1), w2 = tc::smem_u32(sW2);
    auto layer1 = [&](uint32_t t) -> bool {
      const int s = (int)(t % kWsStages), b = (int)(t & 1u);
      bool g = ws_wait(&S.full[s], (t / kWsStages) & 1u, abort, err);
      g = g && ws_wait(&S.a1_empty[b], ((t >> 1) & 1u) ^ 1u, abort, err);
      if (!__all_sync(0xffffffffu, g)) return false;
      tc::fence_after_sync();
      if (lane == 0) tc::mma_tile<64>(tmem + 64 * b, tc::smem_u32(sTiles + s * kWsTile), w1, 80, false, &S.a1_full[b]);
      __syncwarp();
      return true;
    };
    bool ok = TT == 0 || layer1(0);
    for (uint32_t t = 0; t < TT && ok; ++t) {
      if (t + 1 < TT && !layer1(t + 1)) break;
      const int s = (int)(t % kWsStages), b = (int)(t & 1u);
      bool g = ws_wait(&S.a2_ready[b], (t >> 1) & 1u, abort, err);
      g = g && ws_wait(&S.a2_empty[b], ((t >> 1) & 1u) ^ 1u, abort, err);
      if (!__all_sync(0xffffffffu, g)) break;
      tc::fence_after_sync();
      if (lane == 0) {
        tc::mma_tile<64>(tmem + 128 + 64 * b, tc::smem_u32(sTiles + s * kWsTile), w2, 80, false, &S.a2_full[b]);
        ws_commit(&S.empty[s]);                       // the tile buffer is free once layer 2 has read it
      }
      __syncwarp();
    }
    if (lane == 0) ws_commit(&S.fin);                 // every MMA issued above, complete
    __syncwarp();
    if (!tc::mbar_wait(&S.fin, 0) && lane == 0) atomicOr(err, ERR_TIMEOUT);
  } else {
    // ---------------- epilogue (warps 0-3): the messages of tile t - 1 are summed while
    // layer 2 of tile t runs (within a run; its last tile is summed before the next run)
    __align__(16) bf16 one[8];                        // layer 2's constant columns: 1 at 64, 0 after
#pragma unroll
    for (int k = 0; k < 8; ++k) one[k] = __float2bfloat16_rn(k == 0 ? 1.0f : 0.0f);
    uint32_t t = 0;
    bool ok = true;
    int cur = 0;                                      // first node of the run not yet closed
    int64_t i0 = 0;
    int nodes = 0;
    // messages of tile u = [e0, te) of the current run, summed per node in edge order. The
    // tile's nodes are cur, cur + 1, ... while their first edge lies before te (soff never
    // decreases, so they are the nodes cur + k with soff[cur + k] < te; an edgeless node
    // closes where it sits in edge order, those after the run's last edge close after its
    // last tile); a node whose edges run past te stays open and carries its sums.
    auto messages = [&](uint32_t u, uint32_t e0, uint32_t te) -> bool {
      const int b = (int)(u & 1u);
      const int k = cur + tid;
      const int len = epi_count(k < nodes && soff[k] < te);
      if (!epi_all(ws_wait(&S.a2_full[b], (u >> 1) & 1u, abort, err))) return false;
      tc::fence_after_sync();
#pragma unroll 1
      for (int c0 = 0; c0 < 64; c0 += 32) {
        float m[16];
        tc::tmem_ld16(tc::tmem_addr(tmem + 128 + 64 * b, warp, c0), m);
#pragma unroll
        for (int q = 0; q < 16; q += 4)
          *reinterpret_cast<float4*>(&stage[tid * kWsMsgLd + q]) = make_float4(m[q], m[q + 1], m[q + 2], m[q + 3]);
        tc::tmem_ld16(tc::tmem_addr(tmem + 128 + 64 * b, warp, c0 + 16), m);
#pragma unroll
        for (int q = 0; q < 16; q += 4)
          *reinterpret_cast<float4*>(&stage[tid * kWsMsgLd + 16 + q]) = make_float4(m[q], m[q + 1], m[q + 2], m[q + 3]);
        epi_sync();
        // two (node, column) sums a thread at a time, each over its rows in edge order, eight
        // rows' loads in flight (+0 past a node's last row leaves a sum that started at +0
        // unchanged, bit for bit)
        for (int p0 = tid; p0 < len * 32; p0 += 256) {
          const int p1 = p0 + 128;
          const bool two = p1 < len * 32;
          const int li0 = p0 >> 5, li1 = two ? p1 >> 5 : li0, q = p0 & 31;
          const uint32_t kb0 = soff[cur + li0], ke0 = soff[cur + li0 + 1];
          const uint32_t kb1 = soff[cur + li1], ke1 = soff[cur + li1 + 1];
          const int rb0 = (int)(max(kb0, e0) - e0), re0 = (int)(min(ke0, te) - e0);
          const int rb1 = (int)(max(kb1, e0) - e0), re1 = two ? (int)(min(ke1, te) - e0) : rb1;
          float s0 = (li0 == 0 && carry_open) ? carry_in[c0 + q] : 0.f;
          float s1 = (li1 == 0 && carry_open) ? carry_in[c0 + q] : 0.f;
          const uint32_t col = tc::smem_u32(stage + q);
          for (int r = 0; r < re0 - rb0 || r < re1 - rb1; r += 8) {
            float v[8], w[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) {
              v[c] = ld_shared_f32(col + 4u * (uint32_t)(min(rb0 + r + c, 127) * kWsMsgLd));
              w[c] = ld_shared_f32(col + 4u * (uint32_t)(min(rb1 + r + c, 127) * kWsMsgLd));
            }
#pragma unroll
            for (int c = 0; c < 8; ++c) {
              s0 += rb0 + r + c < re0 ? v[c] : 0.f;
              s1 += rb1 + r + c < re1 ? w[c] : 0.f;
            }
          }
          if (ke0 <= te) XN[(i0 + cur + li0) * 144 + F + c0 + q] = __float2bfloat16_rn(s0 * inv_nbar);
          else carry_out[c0 + q] = s0;
          if (two) {
            if (ke1 <= te) XN[(i0 + cur + li1) * 144 + F + c0 + q] = __float2bfloat16_rn(s1 * inv_nbar);
            else carry_out[c0 + q] = s1;
          }
        }
        epi_sync();
      }
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) ws_arrive(&S.a2_empty[b]);
      const bool open = len > 0 && soff[cur + len] > te;   // the tile's last node continues
      if (tid < 64) carry_in[tid] = carry_out[tid];   // read only after the barrier below
      if (tid == 0) carry_open = open ? 1 : 0;
      cur += open ? len - 1 : len;
      epi_sync();
      return true;
    };
    for (int64_t rr = blockIdx.x; rr < runs && ok; rr += gridDim.x) {
      i0 = rr * run;
      const int64_t i1 = min(i0 + (int64_t)run, n);
      nodes = (int)(i1 - i0);
      for (int k = tid; k <= nodes; k += 128) soff[k] = off[i0 + k];
      if (tid == 0) carry_open = 0;
      epi_sync();
      const uint32_t E0 = soff[0], E1 = soff[nodes];
      cur = 0;
      bool pending = false;                           // a tile whose messages are not summed yet
      uint32_t pu = 0, pe0 = 0, pte = 0;
      for (uint32_t e0 = E0; e0 < E1; e0 += 128, ++t) {
        const uint32_t te = min(e0 + 128u, E1);
        const int s = (int)(t % kWsStages), b = (int)(t & 1u);
        unsigned char* A = sTiles + s * kWsTile;
        // layer 2's A over the tile's rows: bf16(relu(z)) of this thread's row, 1, 0...
        if (!epi_all(ws_wait(&S.a1_full[b], (t >> 1) & 1u, abort, err))) {
          ok = false;
          break;
        }
        tc::fence_after_sync();
#pragma unroll 1
        for (int c0 = 0; c0 < 64; c0 += 16) {
          float z[16];
          tc::tmem_ld16(tc::tmem_addr(tmem + 64 * b, warp, c0), z);
          __align__(16) __nv_bfloat162 v[8];         // pairs rounded by one packed conversion each
#pragma unroll
          for (int q = 0; q < 8; ++q) v[q] = __floats2bfloat162_rn(fmaxf(z[2 * q], 0.f), fmaxf(z[2 * q + 1], 0.f));
          *reinterpret_cast<uint4*>(A + tc::core_offset(128, tid, c0)) = *reinterpret_cast<const uint4*>(v);
          *reinterpret_cast<uint4*>(A + tc::core_offset(128, tid, c0 + 8)) = *reinterpret_cast<const uint4*>(v + 4);
        }
        *reinterpret_cast<uint4*>(A + tc::core_offset(128, tid, 64)) = *reinterpret_cast<const uint4*>(one);
        *reinterpret_cast<uint4*>(A + tc::core_offset(128, tid, 72)) = make_uint4(0u, 0u, 0u, 0u);
        tc::fence_to_async();
        tc::fence_before_sync();
        __syncwarp();                                 // the warp's TMEM reads and stores, then one arrival
        if (lane == 0) {
          ws_arrive(&S.a1_empty[b]);
          ws_arrive(&S.a2_ready[b]);
        }
        if (pending && !messages(pu, pe0, pte)) {
          ok = false;
          break;
        }
        pending = true;
        pu = t;
        pe0 = e0;
        pte = te;
      }
      if (ok && pending && !messages(pu, pe0, pte)) ok = false;
      if (!ok) break;
      // nodes left (edgeless ones after the run's last edge): a = 0
      for (int k = cur + tid / 64; k < nodes; k += 2)
        XN[(i0 + k) * 144 + F + (tid & 63)] = __float2bfloat16_rn(0.f * inv_nbar);
      epi_sync();
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) {
    tc::fence_after_sync();
    tc::tmem_free(tmem, 256);
  }
}

__global__ void k_rows_bf16(int64_t n, int cols, const float* __restrict__ src, int lds, bf16* __restrict__ dst,
                            int ldd) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n * cols) return;
  const int64_t r = idx / cols;
  const int c = (int)(idx % cols);
  dst[r * ldd + c] = __float2bfloat16_rn(src[r * lds + c]);
}

// constant columns of an activation buffer: column `one` = 1, [pad_from, ld) = 0
__global__ void k_const_cols(int64_t rows, int ld, int one, int pad_from, bf16* __restrict__ A) {
  const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= rows) return;
  A[r * ld + one] = __float2bfloat16_rn(1.0f);
  for (int c = pad_from; c < ld; ++c) A[r * ld + c] = __float2bfloat16_rn(0.f);
}

// loss and its gradient: dY = 2 (y - target) / (n (d+1)) on the first d+1 columns
__global__ void k_loss(int64_t n, int dout, const float* __restrict__ Y, const double* __restrict__ T,
                       const int* __restrict__ id, bf16* __restrict__ dY, double* __restrict__ loss) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  double l = 0.0;
  if (i < n) {
    const int64_t row = id[i];
    const double scale = 2.0 / ((double)n * dout);
    for (int c = 0; c < 16; ++c) {
      float gval = 0.f;
      if (c < dout) {
        const double d = (double)Y[i * 16 + c] - T[row * dout + c];
        l += d * d;
        gval = (float)(scale * d);
      }
      dY[i * 16 + c] = __float2bfloat16_rn(gval);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
  if ((threadIdx.x & 31) == 0) atomicAdd(loss, l / ((double)n * dout));
}

// dM[e] = bf16(dXN[src(e), F + f] / nbar), 8 columns a thread
__global__ void k_edge_back(int64_t E, const int* __restrict__ esrc, const float* __restrict__ dXN, float inv_nbar,
                            bf16* __restrict__ dM) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= E * (F / 8)) return;
  const int64_t e = idx / (F / 8);
  const int f = (int)(idx % (F / 8)) * 8;
  const float4* x = reinterpret_cast<const float4*>(&dXN[(int64_t)esrc[e] * 144 + F + f]);
  const float4 a = x[0], b = x[1];
  uint4 o;
  o.x = pack2(__float2bfloat16_rn(a.x * inv_nbar), __float2bfloat16_rn(a.y * inv_nbar));
  o.y = pack2(__float2bfloat16_rn(a.z * inv_nbar), __float2bfloat16_rn(a.w * inv_nbar));
  o.z = pack2(__float2bfloat16_rn(b.x * inv_nbar), __float2bfloat16_rn(b.y * inv_nbar));
  o.w = pack2(__float2bfloat16_rn(b.z * inv_nbar), __float2bfloat16_rn(b.w * inv_nbar));
  *reinterpret_cast<uint4*>(&dM[e * F + f]) = o;
}

// Reverse of each fluid edge: erev[e] for e = (i -> j) is the edge (j -> i) (the frozen
// fluid neighbour relation is symmetric: |r_i - r_j| < 2h either way); -1 for walls.
__global__ void k_reverse_edges(int64_t E, const int* __restrict__ esrc, const int* __restrict__ enbr,
                                const uint32_t* __restrict__ off, int* __restrict__ erev) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= E) return;
  const int i = esrc[e], j = enbr[e];
  int r = -1;
  if (j >= 0)
    for (uint32_t e2 = off[j]; e2 < off[j + 1]; ++e2)
      if (enbr[e2] == i) {
        r = (int)e2;
        break;
      }
  erev[e] = r;
}

// Node-state gradient of a round: dh[j] = (dh[j] + dXN[j, :F]) + sum over edges (i -> j) of
// dXE[e, fe + f], the transpose of the gather h_j -> x_ij, taken over j's own fluid edges
// (j -> i) through their reverses, in edge order. dZ = bf16(dh), the next round's operand, or
// with H0 (the encoder's ReLU) bf16(dh) where h0 > 0 and 0 elsewhere. A warp per node: the
// reverses of 32 edges come in one load, and eight edges' rows are in flight at a time (a
// thread per element that followed enbr, erev and the row edge by edge took twice the time).
__global__ void k_gather_dh(int64_t n, int fe, const uint32_t* __restrict__ off, const int* __restrict__ enbr,
                            const int* __restrict__ erev, const float* __restrict__ dXE,
                            const float* __restrict__ dXN, const float* __restrict__ H0, float* __restrict__ dH,
                            bf16* __restrict__ dZ) {
  const int64_t j = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (j >= n) return;
  const uint32_t end = off[j + 1];
  float a0 = 0.f, a1 = 0.f;
  for (uint32_t e0 = off[j]; e0 < end; e0 += 32) {
    const uint32_t e = e0 + lane;
    const bool fluid = e < end && enbr[e] >= 0;       // fluid edges come first
    const int rev = fluid ? erev[e] : -1;
    const int cnt = __popc(__ballot_sync(0xffffffffu, fluid));
    for (int k0 = 0; k0 < cnt; k0 += 8) {
      float v0[8], v1[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int r = __shfl_sync(0xffffffffu, rev, (k0 + k) & 31);
        const bool use = k0 + k < cnt && r >= 0;
        const float* x = dXE + (int64_t)(use ? r : 0) * 80 + fe + lane;
        v0[k] = use ? x[0] : 0.f;
        v1[k] = use ? x[32] : 0.f;
      }
#pragma unroll
      for (int k = 0; k < 8; ++k) {                   // +0 leaves a sum that started at +0 unchanged
        a0 += v0[k];
        a1 += v1[k];
      }
    }
  }
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    const int64_t o = j * F + 32 * half + lane;
    const float h = dH[o] + dXN[j * 144 + 32 * half + lane] + (half ? a1 : a0);
    dH[o] = h;
    dZ[o] = __float2bfloat16_rn(!H0 || H0[o] > 0.f ? h : 0.f);
  }
}

// Adam (beta1 0.9, beta2 0.999, eps 1e-8); b1pow = beta1^t, b2pow = beta2^t
__global__ void k_adam(int count, float* __restrict__ w, float* __restrict__ m, float* __restrict__ v,
                       const float* __restrict__ g, float lr, float b1pow, float b2pow) {
  const int o = blockIdx.x * blockDim.x + threadIdx.x;
  if (o >= count) return;
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  m[o] = b1 * m[o] + (1.f - b1) * g[o];
  v[o] = b2 * v[o] + (1.f - b2) * g[o] * g[o];
  const float mh = m[o] / (1.f - b1pow), vh = v[o] / (1.f - b2pow);
  w[o] -= lr * mh / (sqrtf(vh) + eps);
}

// bf16 copies of the weights: row-major and, per matrix, transposed
__global__ void k_weights_bf16(const float* __restrict__ w, bf16* __restrict__ wb, bf16* __restrict__ wbt) {
  const int o = blockIdx.x * blockDim.x + threadIdx.x;
  if (o >= kWeights) return;
  int base = 0, l = 0;
  while (l < L_COUNT - 1 && o >= base + c_rows[l] * c_cols[l]) {
    base += c_rows[l] * c_cols[l];
    ++l;
  }
  const int r = (o - base) / c_cols[l], c = (o - base) % c_cols[l];
  const bf16 b = __float2bfloat16_rn(w[o]);
  wb[o] = b;
  wbt[base + c * c_rows[l] + r] = b;
}

// Apply a prediction: v' = v + g Dt_ad + V_S y_v, rho' = rho + rho0 y_rho / 100,
// r' = r + Dt_ad (v + v')/2, d rho/dt = (rho' - rho)/Dt_ad; the tank's clock advances by Dt_ad.
template <int D>
__global__ void k_apply(int64_t n, int4* __restrict__ P, float4* __restrict__ V, const int* __restrict__ inst_of,
                        const Inst* __restrict__ inst, const Ctrl* __restrict__ ctrl, const float* __restrict__ Y,
                        Global* g) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int k = inst_of ? inst_of[i] : 0;
  const Inst& I = inst[k];
  const float dt = (float)ctrl[k].dt_ad;
  const float gmag = sqrtf(I.g[0] * I.g[0] + I.g[1] * I.g[1] + I.g[2] * I.g[2]);
  const float vs = gmag > 0.f ? gmag * dt : (float)I.u_ref;
  int4 p = P[i];
  const float4 v = V[i];
  const float* y = Y + i * 16;
  const float vn[3] = {v.x + I.g[0] * dt + vs * y[0], v.y + I.g[1] * dt + vs * y[1],
                       D == 3 ? v.z + I.g[2] * dt + vs * y[2] : 0.f};
  const float drho = I.rho0 * y[D] / S_RHO;
  const float dev = i2f(p.w) + drho;
  const float vo[3] = {v.x, v.y, v.z};
  int q[3] = {p.x, p.y, p.z};
  for (int a = 0; a < D; ++a) q[a] = wrap_coord(q[a] + __float2int_rn(0.5f * dt * (vo[a] + vn[a]) * I.inv_dq), I.period[a]);
  if (!isfinite(dev) || !isfinite(vn[0]) || !isfinite(vn[1])) atomicOr(&g->err, ERR_NAN);
  P[i] = make_int4(q[0], q[1], q[2], f2i(dev));
  V[i] = make_float4(vn[0], vn[1], vn[2], dt > 0.f ? drho / dt : 0.f);
}

__global__ void k_learned_clock(int n_inst, Ctrl* ctrl) {
  for (int k = threadIdx.x; k < n_inst; k += blockDim.x) {
    ctrl[k].t += ctrl[k].dt_ad;
    ctrl[k].tau = ctrl[k].dt_ad;
    ctrl[k].done = 1;
    ctrl[k].dt = 0.0;
  }
}

template <int NO>
size_t dense_smem(int K) {
  // W and two A tiles; at least enough that no more CTAs share an SM than its 512 TMEM
  // columns hold, so a TMEM allocation never waits
  const size_t need = (size_t)dense_w_bytes(NO, K) + 2 * (size_t)dense_tile_bytes(K);
  const size_t per_sm = 233472;                               // shared memory of an SM
  const size_t floor = per_sm / (size_t)(512 / tc::tmem_cols(NO) + 1) + 1;
  return std::max(need, floor);
}

template <int NO, int K>
constexpr int dw_smem() { return 2 * kTile * ((NO + 8) + (K + 8)) * (int)sizeof(bf16); }

template <int NO, int K, bool MASK = false>
void set_smem_attrs() {
  cudaFuncSetAttribute(k_dense<NO, K, MASK>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dense_smem<NO>(K));
}

template <int NO, int K>
void set_dw_attrs() {
  cudaFuncSetAttribute(k_dense_dw<NO, K>, cudaFuncAttributeMaxDynamicSharedMemorySize, dw_smem<NO, K>());
}

}  // namespace learned
}  // namespace sph

using namespace sph::learned;

struct sph_learned {
  int dim = 2;
  float* w32 = nullptr;
  float* m = nullptr;
  float* v = nullptr;
  float* grad = nullptr;
  bf16* wb = nullptr;
  bf16* wbt = nullptr;
  int64_t adam_t = 0;
  int fused = 1;                             // inference rounds: 0 layer by layer, 1 warp MMA, 2 tcgen05 pipeline
  int* tc_err = nullptr;                     // the handle's device error word (tensor-core waits)
  int n_sm = 1;                              // SMs of the device
  // workspace
  int64_t cap_n = 0, cap_e = 0;
  uint32_t* cnt = nullptr;
  uint32_t* off = nullptr;
  uint32_t* scan_tmp = nullptr;
  int* esrc = nullptr;
  int* enbr = nullptr;
  bf16* U = nullptr;
  bf16* XS = nullptr;                        // [E][16] static edge features
  bf16* T = nullptr;                         // [n + 1][80] round input row templates
  bf16* T2 = nullptr;                        // ... of every second fused round
  int* erev = nullptr;                       // [E] reverse of each fluid edge, -1 for walls
  bf16* XE[ROUNDS] = {nullptr};
  bf16* A1[ROUNDS] = {nullptr};
  bf16* XN[ROUNDS] = {nullptr};
  bf16* A2[ROUNDS] = {nullptr};
  float* Mbuf = nullptr;
  float* H = nullptr;
  float* H0 = nullptr;
  bf16* XD = nullptr;
  bf16* A3 = nullptr;
  float* Y = nullptr;
  float* dH = nullptr;
  float* dXN = nullptr;
  bf16* dYb = nullptr;
  bf16* dZn = nullptr;
  bf16* dM = nullptr;
  bf16* dZe = nullptr;
  float* dXE = nullptr;
  float* partial = nullptr;
  size_t partial_elems = 0;
  double* loss = nullptr;
  int64_t E = 0;
  // saved state for the fallback
  int4* saveP = nullptr;
  float4* saveV = nullptr;
  sph::Ctrl* saveC = nullptr;
  std::vector<void*> allocs;
  std::string err;
};

namespace {

template <typename T>
bool nalloc(sph_learned* L, T** p, size_t count) {
  if (count == 0) count = 1;
  if (cudaMalloc((void**)p, sizeof(T) * count) != cudaSuccess) {
    cudaGetLastError();
    *p = nullptr;
    return false;
  }
  L->allocs.push_back((void*)*p);
  return true;
}

inline unsigned blocks_for(int64_t n, int b = 256) { return (unsigned)((n + b - 1) / b); }

int ensure_workspace(sph_learned* L, int64_t n, int64_t E) {
  if (n <= L->cap_n && E <= L->cap_e) return SPH_OK;
  // grow: free the old workspace (not the weights) and allocate anew
  void* keep[6] = {L->w32, L->m, L->v, L->grad, L->wb, L->wbt};
  std::vector<void*> rest;
  for (void* p : L->allocs) {
    bool k = false;
    for (void* q : keep) k |= (p == q);
    if (k) rest.push_back(p);
    else cudaFree(p);
  }
  L->allocs = rest;
  L->saveC = nullptr;                        // freed above with the rest of the workspace
  n = std::max<int64_t>(n, L->cap_n);
  E = std::max<int64_t>(E, L->cap_e);
  bool ok = nalloc(L, &L->cnt, n) && nalloc(L, &L->off, n + 1) &&
            nalloc(L, &L->scan_tmp, sph::scan_tmp_elems(n)) && nalloc(L, &L->esrc, E) && nalloc(L, &L->enbr, E) && nalloc(L, &L->XS, E * 16) && nalloc(L, &L->erev, E) &&
            nalloc(L, &L->U, n * 16) && nalloc(L, &L->Mbuf, E * F) && nalloc(L, &L->H, n * F) &&
            nalloc(L, &L->H0, n * F) && nalloc(L, &L->XD, n * 80) && nalloc(L, &L->A3, n * 80) &&
            nalloc(L, &L->Y, n * 16) && nalloc(L, &L->dH, n * F) && nalloc(L, &L->dXN, n * 144) &&
            nalloc(L, &L->dYb, n * 16) && nalloc(L, &L->dZn, n * F) && nalloc(L, &L->dM, E * F) &&
            nalloc(L, &L->dZe, std::max(E, n) * F) && nalloc(L, &L->dXE, E * 80) && nalloc(L, &L->loss, 1) &&
            nalloc(L, &L->saveP, n) && nalloc(L, &L->saveV, n) && nalloc(L, &L->T, (n + 1) * 80) && nalloc(L, &L->T2, (n + 1) * 80);
  for (int r = 0; r < ROUNDS && ok; ++r)
    ok = nalloc(L, &L->XE[r], E * 80) && nalloc(L, &L->A1[r], E * 80) && nalloc(L, &L->XN[r], n * 144) &&
         nalloc(L, &L->A2[r], n * 80);
  // one round's layers and the decoder's or the encoder's
  L->partial_elems = (size_t)kDwBlocks * (64 * 144 + 4 * 64 * 80 + 16 * 80);
  ok = ok && nalloc(L, &L->partial, L->partial_elems);
  if (!ok) {
    L->err = "device allocation of the network workspace failed";
    return SPH_E_OOM;
  }
  L->cap_n = n;
  L->cap_e = E;
  // constant columns of the activation buffers (bias 1 and zero padding): no kernel writes
  // them afterwards, so they are set once for every row the workspace holds
  auto consts = [](int64_t rows, int ld, int one, int pad_from, bf16* A) {
    if (rows > 0) k_const_cols<<<blocks_for(rows), 256>>>(rows, ld, one, pad_from, A);
  };
  for (int r = 0; r < ROUNDS; ++r) {
    consts(E, 80, F, F + 1, L->A1[r]);
    consts(n, 144, 2 * F, 2 * F + 1, L->XN[r]);
    consts(n, 80, F, F + 1, L->A2[r]);
  }
  consts(n, 80, F, F + 1, L->XD);
  consts(n, 80, F, F + 1, L->A3);
  if (cudaDeviceSynchronize() != cudaSuccess) {   // before work on the caller's stream uses them
    L->err = "initialising the network workspace failed";
    return SPH_E_CUDA;
  }
  return SPH_OK;
}

template <int NO, int K, bool MASK = false>
void dense(int64_t M, const bf16* X, int ldx, const bf16* W, float* of, int ldf, int nf, int accum,
           bf16* ob, int ldo, int col0, int nb, int relu, const bf16* mask, int ldm, const sph_learned* L, cudaStream_t s) {
  static_assert(K % 16 == 0, "K in MMA steps of 16");
  if (M == 0) return;
  // rows move as 16-byte pieces, results as 16-byte pieces: strides and column ranges must
  // allow it; a mask applies to the bfloat16 results
  if (ldx % 8 || (of && (ldf % 4 || nf % 4)) || (ob && (ldo % 8 || col0 % 8 || nb % 8 || nb > 64)) ||
      (mask != nullptr) != MASK || (MASK && (ldm % 8 || of || !ob))) {
    std::fprintf(stderr, "sph_learned: dense layer with unaligned shape\n");
    return;
  }
  // One CTA an SM up to eight tiles an SM, then two: a CTA's start takes 2 us (its TMEM, its
  // first copies), and the CTAs of an SM start one after the other, so a CTA a tile only pays
  // where an SM has no second one (64 outputs, K = 80: 498 tiles 12.4 us with one CTA an SM, 13.6
  // with two, 14.5 with four; 784 tiles 16.5, 16.5, 18.6; 5,000 tiles 69, 58, 62; 21,094 tiles 264, 219, 220).
  const int64_t tiles = (M + 127) / 128;
  const int64_t sms = L->n_sm;
  const unsigned grid = (unsigned)std::min<int64_t>(tiles, tiles <= 8 * sms ? sms : 2 * sms);
  k_dense<NO, K, MASK><<<grid, 128, dense_smem<NO>(K), s>>>(M, X, ldx, W, of, ldf, nf, accum, ob, ldo, col0, nb, relu,
                                                            mask, ldm, L->tc_err);
}

// The weight gradients pending for one launch of k_reduce_partials
struct DwPending {
  DwSums S;
  int jobs = 0, outputs = 0;
  size_t used = 0;
};

// grad[layer] += dY^T X over M rows, complete after flush_dw
template <int NO, int K>
void dense_dw(sph_learned* L, DwPending& p, int layer, int64_t M, const bf16* dY, int ldy, const bf16* X, int ldx,
              cudaStream_t s) {
  if (M == 0) return;
  const int64_t rows = dw_rows(M);
  const int blocks = (int)((M + rows - 1) / rows);
  k_dense_dw<NO, K><<<blocks, 256, dw_smem<NO, K>(), s>>>(M, rows, dY, ldy, X, ldx, L->partial + p.used);
  p.S.job[p.jobs++] = {blocks, NO * K, w_offset(layer), p.used};
  p.used += (size_t)blocks * NO * K;
  p.outputs += NO * K;
}
void flush_dw(sph_learned* L, DwPending& p, cudaStream_t s) {
  if (p.jobs) k_reduce_partials<<<p.outputs / 32, 256, 0, s>>>(p.S, p.jobs, L->partial, L->grad);
  p = DwPending();
}

const bf16* Wl(const sph_learned* L, int l) { return L->wb + w_offset(l); }
const bf16* WTl(const sph_learned* L, int l) { return L->wbt + w_offset(l); }

// Graph and features of the handle's current (post density re-initialisation) state.
int build_inputs(sph_handle* h, sph_learned* L, cudaStream_t s) {
  const sph::Buffers& b = h->b;
  const int64_t n = b.n;
  // edge count first (host needs E to size the workspace)
  if (ensure_workspace(L, n, std::max<int64_t>(L->cap_e, 1)) != SPH_OK) return SPH_E_OOM;
  k_edge_count<<<blocks_for(n), 256, 0, s>>>(n, b.nbc, L->cnt);
  int64_t dummy = 0;
  sph::scan_exclusive(L->cnt, L->off, n, L->scan_tmp, s, &dummy);
  uint32_t E32 = 0;
  if (cudaMemcpyAsync(&E32, L->off + n, sizeof(uint32_t), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess) {
    cudaGetLastError();
    return SPH_E_CUDA;
  }
  const int64_t E = E32;
  if (E > L->cap_e) {
    if (ensure_workspace(L, n, E) != SPH_OK) return SPH_E_OOM;
    k_edge_count<<<blocks_for(n), 256, 0, s>>>(n, b.nbc, L->cnt);
    sph::scan_exclusive(L->cnt, L->off, n, L->scan_tmp, s, &dummy);
  }
  L->E = E;
  auto nodes = b.dim == 2 ? k_node_features<2> : k_node_features<3>;
  nodes<<<blocks_for(n), 256, 0, s>>>(n, b.PS, b.VS, b.inst_of, b.inst, b.ctrl, L->U);
  auto edges = b.dim == 2 ? k_edge_features<2> : k_edge_features<3>;
  edges<<<blocks_for((n + kEdgeNodes - 1) / kEdgeNodes * 32), 256, 0, s>>>(
      n, b.PS, b.VS, b.inst_of, b.inst, b.nbr, b.nbc, L->off, b.WP, L->esrc, L->enbr, L->XS);
  return cudaGetLastError() == cudaSuccess ? SPH_OK : SPH_E_CUDA;
}

// train: keep every round's edge rows and activations for the backward pass; otherwise
// (inference) the edge network of each round runs fused when the network allows it.
void forward(sph_handle* h, sph_learned* L, cudaStream_t s, bool train) {
  L->tc_err = &h->b.glob->err;
  const int64_t n = h->b.n, E = L->E;
  const int d = h->b.dim, fe = 2 * d + 3;
  const float inv_nbar = 1.0f / nbar(d);
  const bool fused = L->fused == 1 && !train;
  const bool piped = L->fused == 2 && !train;
  // encoder: H = relu(U W_enc^T); H0 keeps h0 for the encoder's backward
  dense<64, 16>(n, L->U, 16, Wl(L, L_ENC), L->H, F, F, 0, nullptr, 0, 0, 0, 1, nullptr, 0, L, s);
  if (train) cudaMemcpyAsync(L->H0, L->H, sizeof(float) * n * F, cudaMemcpyDeviceToDevice, s);
  for (int r = 0; r < ROUNDS; ++r) {
    if (fused) {
      if (n == 0) continue;
      // runs of equal node counts, a whole number of them per warp where possible; short runs
      // where the warps would outnumber them, down to a half tile of edges
      const int64_t slots = (int64_t)L->n_sm * kFuseWarps;
      const int64_t per = (n + slots * kFuseRun - 1) / (slots * kFuseRun);
      const int run = (int)std::max<int64_t>(kFuseRunMin, (n + slots * per - 1) / (slots * per));
      const unsigned grid = (unsigned)std::min<int64_t>((n + run - 1) / run, L->n_sm);
      // node states ping-pong between H and H0 (H0 is only kept for training's backward), the
      // templates between T and T2; the last round leaves the decoder's input rows instead
      const float* hin = (r & 1) ? L->H0 : L->H;
      float* hout = (r & 1) ? L->H : L->H0;
      const bf16* tin = (r & 1) ? L->T2 : L->T;
      const bool last = r == ROUNDS - 1;
      bf16* tout = last ? L->XD : ((r & 1) ? L->T : L->T2) + 80;
      if (r == 0) {
        auto tmpl = d == 2 ? k_node_templates<7> : k_node_templates<9>;
        tmpl<<<blocks_for((n + 1) * 10), 256, 0, s>>>(n, hin, L->T, L->XN[r]);
      }
      auto kern = d == 2 ? k_edge_round_fused<7> : k_edge_round_fused<9>;
      kern<<<grid, kFuseWarps * 32, fused_smem(), s>>>(n, run, L->off, L->XS, L->enbr, hin, tin, Wl(L, L_E1),
                                                       Wl(L, L_E2), Wl(L, L_N1), Wl(L, L_N2), inv_nbar, L->XN[r], hout,
                                                       tout, last ? 0 : fe);
    } else if (piped) {
      auto tmpl = d == 2 ? k_node_templates<7> : k_node_templates<9>;
      tmpl<<<blocks_for((n + 1) * 10 + n * 8), 256, 0, s>>>(n, L->H, L->T, L->XN[r]);
      if (n > 0) {
        // runs of equal node counts, a whole number of them per CTA where possible
        const int64_t slots = 2 * (int64_t)L->n_sm;
        const int64_t per = (n + slots * kWsRun - 1) / (slots * kWsRun);
        const int run = (int)std::max<int64_t>(1, (n + slots * per - 1) / (slots * per));
        const int64_t runs = (n + run - 1) / run;
        const unsigned grid = (unsigned)std::min<int64_t>(runs, slots);
        auto kern = d == 2 ? k_edge_round_ws<7> : k_edge_round_ws<9>;
        kern<<<grid, kWsThreads, ws_smem(), s>>>(n, run, L->off, L->XS, L->enbr, L->T, Wl(L, L_E1), Wl(L, L_E2),
                                                 inv_nbar, L->XN[r], L->tc_err);
      }
      dense<64, 144>(n, L->XN[r], 144, Wl(L, L_N1), nullptr, 0, 0, 0, L->A2[r], 80, 0, F, 1, nullptr, 0, L, s);
      dense<64, 80>(n, L->A2[r], 80, Wl(L, L_N2), L->H, F, F, 1, nullptr, 0, 0, 0, 0, nullptr, 0, L, s);
    } else {
      if (E > 0) k_edge_rows<<<blocks_for(E * 10), 256, 0, s>>>(E, fe, L->XS, L->enbr, L->H, L->XE[r]);
      dense<64, 80>(E, L->XE[r], 80, Wl(L, L_E1), nullptr, 0, 0, 0, L->A1[r], 80, 0, F, 1, nullptr, 0, L, s);
      dense<64, 80>(E, L->A1[r], 80, Wl(L, L_E2), L->Mbuf, F, F, 0, nullptr, 0, 0, 0, 0, nullptr, 0, L, s);
      k_segsum<<<blocks_for(n * F), 256, 0, s>>>(n, L->off, L->Mbuf, L->H, inv_nbar, L->XN[r]);
      dense<64, 144>(n, L->XN[r], 144, Wl(L, L_N1), nullptr, 0, 0, 0, L->A2[r], 80, 0, F, 1, nullptr, 0, L, s);
      dense<64, 80>(n, L->A2[r], 80, Wl(L, L_N2), L->H, F, F, 1, nullptr, 0, 0, 0, 0, nullptr, 0, L, s);
    }
  }
  // the fused rounds leave the decoder's input rows
  if (!fused) k_rows_bf16<<<blocks_for(n * F), 256, 0, s>>>(n, F, L->H, F, L->XD, 80);
  dense<64, 80>(n, L->XD, 80, Wl(L, L_D1), nullptr, 0, 0, 0, L->A3, 80, 0, F, 1, nullptr, 0, L, s);
  dense<16, 80>(n, L->A3, 80, Wl(L, L_D2), L->Y, 16, 16, 0, nullptr, 0, 0, 0, 0, nullptr, 0, L, s);
}

void backward(sph_handle* h, sph_learned* L, cudaStream_t s) {
  L->tc_err = &h->b.glob->err;
  const int64_t n = h->b.n, E = L->E;
  const int d = h->b.dim, fe = 2 * d + 3;
  const float inv_nbar = 1.0f / nbar(d);
  cudaMemsetAsync(L->grad, 0, sizeof(float) * kWeights, s);
  if (E > 0) k_reverse_edges<<<blocks_for(E), 256, 0, s>>>(E, L->esrc, L->enbr, L->off, L->erev);
  DwPending p;
  // decoder; dZe is the edge buffer (at least n rows)
  dense_dw<16, 80>(L, p, L_D2, n, L->dYb, 16, L->A3, 80, s);
  dense<80, 16, true>(n, L->dYb, 16, WTl(L, L_D2), nullptr, 0, 0, 0, L->dZe, F, 0, F, 0, L->A3, 80, L, s);
  dense_dw<64, 80>(L, p, L_D1, n, L->dZe, F, L->XD, 80, s);
  dense<80, 64>(n, L->dZe, F, WTl(L, L_D1), L->dH, F, F, 0, L->dZn, F, 0, F, 0, nullptr, 0, L, s);
  for (int r = ROUNDS - 1; r >= 0; --r) {
    // h_new = h + W_n2 [relu(W_n1 XN), 1]; dZn = bf16(dh)
    dense_dw<64, 80>(L, p, L_N2, n, L->dZn, F, L->A2[r], 80, s);
    bf16* dZ2 = L->dZe;
    dense<80, 64, true>(n, L->dZn, F, WTl(L, L_N2), nullptr, 0, 0, 0, dZ2, F, 0, F, 0, L->A2[r], 80, L, s);
    dense_dw<64, 144>(L, p, L_N1, n, dZ2, F, L->XN[r], 144, s);
    dense<144, 64>(n, dZ2, F, WTl(L, L_N1), L->dXN, 144, 144, 0, nullptr, 0, 0, 0, 0, nullptr, 0, L, s);
    if (E > 0) k_edge_back<<<blocks_for(E * (F / 8)), 256, 0, s>>>(E, L->esrc, L->dXN, inv_nbar, L->dM);
    dense_dw<64, 80>(L, p, L_E2, E, L->dM, F, L->A1[r], 80, s);
    dense<80, 64, true>(E, L->dM, F, WTl(L, L_E2), nullptr, 0, 0, 0, L->dZe, F, 0, F, 0, L->A1[r], 80, L, s);
    dense_dw<64, 80>(L, p, L_E1, E, L->dZe, F, L->XE[r], 80, s);
    dense<80, 64>(E, L->dZe, F, WTl(L, L_E1), L->dXE, 80, 80, 0, nullptr, 0, 0, 0, 0, nullptr, 0, L, s);
    k_gather_dh<<<blocks_for(n * 32), 256, 0, s>>>(n, fe, L->off, L->enbr, L->erev, L->dXE, L->dXN,
                                                   r == 0 ? L->H0 : nullptr, L->dH, L->dZn);
    if (r > 0) flush_dw(L, p, s);
  }
  dense_dw<64, 16>(L, p, L_ENC, n, L->dZn, F, L->U, 16, s);
  flush_dw(L, p, s);
}

}  // namespace

// ------------------------------------------------------------------ C ABI
namespace {

__global__ void k_export_y(int64_t n, int dout, const float* __restrict__ Y, const int* __restrict__ id,
                           double* __restrict__ y) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int64_t row = id[i];
  for (int c = 0; c < dout; ++c) y[row * dout + c] = (double)Y[i * 16 + c];
}

// Memory the current device can address directly (its own or managed); device memory
// of another GPU counts as not addressable (see foreign_ptr).
bool device_ptr(const void* p) {
  cudaPointerAttributes at;
  if (!p || cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  if (at.type == cudaMemoryTypeManaged) return true;
  int cur = -1;
  if (at.type != cudaMemoryTypeDevice || cudaGetDevice(&cur) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return at.device == cur;
}

// Device memory of a GPU other than the current one: rejected by the entry points, since
// the kernels run on the current device.
bool foreign_ptr(const void* p) {
  cudaPointerAttributes at;
  if (!p || cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  int cur = -1;
  if (at.type != cudaMemoryTypeDevice || cudaGetDevice(&cur) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return at.device != cur;
}

int lfail(sph_learned* L, int code, const char* msg) {
  if (L) L->err = msg;
  return code;
}

void upload_weights_bf16(sph_learned* L, cudaStream_t s) {
  k_weights_bf16<<<blocks_for(kWeights), 256, 0, s>>>(L->w32, L->wb, L->wbt);
}

int ready(sph_handle* h, sph_learned* L, void* stream) {
  if (!h || !L) return SPH_E_INVALID;
  if (h->b.dim != L->dim) return lfail(L, SPH_E_INVALID, "network and handle dimensions differ");
  if (!h->cells_valid) return lfail(L, SPH_E_INVALID, "run sph_build_cells and sph_advection_step first");
  const int r = sph_debug_check(h, (cudaStream_t)stream);
  if (r != SPH_OK) return lfail(L, r, "neighbour table check failed (SPH_FLAG_DEBUG_BOUNDS)");
  return SPH_OK;
}

}  // namespace

extern "C" {

int sph_learned_weight_count(int64_t* count) {
  if (!count) return SPH_E_INVALID;
  *count = kWeights;
  return SPH_OK;
}

const char* sph_learned_last_error(const sph_learned* L) { return L ? L->err.c_str() : "null network"; }

void sph_learned_destroy(sph_learned* L) {
  if (!L) return;
  for (void* p : L->allocs) cudaFree(p);
  delete L;
}

int sph_learned_create(int32_t dim, const float* weights, sph_learned** out) {
  if (!out || (dim != 2 && dim != 3)) return SPH_E_INVALID;
  sph_learned* L = new sph_learned();
  *out = L;
  L->dim = dim;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&L->n_sm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    cudaGetLastError();
    return lfail(L, SPH_E_CUDA, "no CUDA device");
  }
  if (!nalloc(L, &L->w32, kWeights) || !nalloc(L, &L->m, kWeights) || !nalloc(L, &L->v, kWeights) ||
      !nalloc(L, &L->grad, kWeights) || !nalloc(L, &L->wb, kWeights) || !nalloc(L, &L->wbt, kWeights))
    return lfail(L, SPH_E_OOM, "device allocation of the weights failed");
  cudaFuncSetAttribute(k_edge_round_fused<7>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fused_smem());
  cudaFuncSetAttribute(k_edge_round_fused<9>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fused_smem());
  cudaFuncSetAttribute(k_edge_round_ws<7>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ws_smem());
  cudaFuncSetAttribute(k_edge_round_ws<9>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ws_smem());
  set_smem_attrs<64, 16>();
  set_smem_attrs<64, 80>();
  set_smem_attrs<64, 144>();
  set_smem_attrs<16, 80>();
  set_smem_attrs<80, 16, true>();
  set_smem_attrs<80, 64>();
  set_smem_attrs<80, 64, true>();
  set_smem_attrs<144, 64>();
  set_dw_attrs<16, 80>();
  set_dw_attrs<64, 16>();
  set_dw_attrs<64, 80>();
  set_dw_attrs<64, 144>();
  cudaMemset(L->m, 0, sizeof(float) * kWeights);
  cudaMemset(L->v, 0, sizeof(float) * kWeights);
  cudaMemset(L->w32, 0, sizeof(float) * kWeights);
  if (weights && cudaMemcpy(L->w32, weights, sizeof(float) * kWeights, cudaMemcpyDefault) != cudaSuccess) {
    cudaGetLastError();
    return lfail(L, SPH_E_CUDA, "copy of the weights failed");
  }
  upload_weights_bf16(L, 0);
  if (cudaDeviceSynchronize() != cudaSuccess) {
    cudaGetLastError();
    return lfail(L, SPH_E_CUDA, "network set-up failed");
  }
  return SPH_OK;
}

int sph_learned_set_weights(sph_learned* L, const float* w) {
  if (!L || !w) return SPH_E_INVALID;
  if (cudaMemcpy(L->w32, w, sizeof(float) * kWeights, cudaMemcpyDefault) != cudaSuccess) {
    cudaGetLastError();
    return lfail(L, SPH_E_CUDA, "copy of the weights failed");
  }
  cudaMemset(L->m, 0, sizeof(float) * kWeights);
  cudaMemset(L->v, 0, sizeof(float) * kWeights);
  L->adam_t = 0;
  upload_weights_bf16(L, 0);
  return cudaDeviceSynchronize() == cudaSuccess ? SPH_OK : SPH_E_CUDA;
}

int sph_learned_get_weights(sph_learned* L, float* w) {
  if (!L || !w) return SPH_E_INVALID;
  if (cudaMemcpy(w, L->w32, sizeof(float) * kWeights, cudaMemcpyDefault) != cudaSuccess) {
    cudaGetLastError();
    return lfail(L, SPH_E_CUDA, "copy of the weights failed");
  }
  return SPH_OK;
}

int sph_learned_set_fused(sph_learned* L, int32_t enabled) {
  if (!L) return SPH_E_INVALID;
  if (enabled < 0 || enabled > 2) return SPH_E_INVALID;
  L->fused = enabled;
  return SPH_OK;
}

int sph_learned_predict(sph_handle* h, sph_learned* L, double* y, void* stream) {
  int r = ready(h, L, stream);
  if (r != SPH_OK) return r;
  cudaStream_t s = (cudaStream_t)stream;
  r = build_inputs(h, L, s);
  if (r != SPH_OK) return lfail(L, r, "building the network inputs failed");
  if (foreign_ptr(y)) return lfail(L, SPH_E_INVALID, "y lives on another device");
  forward(h, L, s, false);
  if (y) {
    const int dout = h->b.dim + 1;
    const bool dev = device_ptr(y);
    double* tgt = dev ? y : h->stage;
    k_export_y<<<blocks_for(h->b.n), 256, 0, s>>>(h->b.n, dout, L->Y, h->b.id, tgt);
    if (!dev && cudaMemcpyAsync(y, tgt, sizeof(double) * h->b.n * dout, cudaMemcpyDeviceToHost, s) != cudaSuccess) {
      cudaGetLastError();
      return lfail(L, SPH_E_CUDA, "copy of the prediction failed");
    }
  }
  if (cudaStreamSynchronize(s) != cudaSuccess) {
    cudaGetLastError();
    return lfail(L, SPH_E_CUDA, "network forward pass failed");
  }
  return SPH_OK;
}

int sph_learned_train_step(sph_handle* h, sph_learned* L, const double* target, double lr, double* loss_out,
                           float* grad_out, void* stream) {
  int r = ready(h, L, stream);
  if (r != SPH_OK) return r;
  if (!target) return lfail(L, SPH_E_INVALID, "target is required");
  if (foreign_ptr(target)) return lfail(L, SPH_E_INVALID, "target lives on another device");
  cudaStream_t s = (cudaStream_t)stream;
  r = build_inputs(h, L, s);
  if (r != SPH_OK) return lfail(L, r, "building the network inputs failed");
  forward(h, L, s, true);
  const int64_t n = h->b.n;
  const int dout = h->b.dim + 1;
  const double* T = target;
  if (!device_ptr(target)) {
    if (cudaMemcpyAsync(h->stage, target, sizeof(double) * n * dout, cudaMemcpyHostToDevice, s) != cudaSuccess) {
      cudaGetLastError();
      return lfail(L, SPH_E_CUDA, "copy of the target failed");
    }
    T = h->stage;
  }
  cudaMemsetAsync(L->loss, 0, sizeof(double), s);
  k_loss<<<blocks_for(n), 256, 0, s>>>(n, dout, L->Y, T, h->b.id, L->dYb, L->loss);
  backward(h, L, s);
  if (lr > 0.0) {
    ++L->adam_t;
    const float b1pow = (float)std::pow(0.9, (double)L->adam_t), b2pow = (float)std::pow(0.999, (double)L->adam_t);
    k_adam<<<blocks_for(kWeights), 256, 0, s>>>(kWeights, L->w32, L->m, L->v, L->grad, (float)lr, b1pow, b2pow);
    upload_weights_bf16(L, s);
  }
  double loss = 0.0;
  cudaMemcpyAsync(&loss, L->loss, sizeof(double), cudaMemcpyDeviceToHost, s);
  if (grad_out) cudaMemcpyAsync(grad_out, L->grad, sizeof(float) * kWeights, cudaMemcpyDefault, s);
  if (cudaStreamSynchronize(s) != cudaSuccess) {
    cudaGetLastError();
    return lfail(L, SPH_E_CUDA, "training step failed");
  }
  if (loss_out) *loss_out = loss;
  return SPH_OK;
}

int sph_learned_step(sph_handle* h, sph_learned* L, double max_mean_rho_dev, double max_energy_drift,
                     int32_t* used_learned, void* stream) {
  if (!h || !L) return SPH_E_INVALID;
  if (h->b.dim != L->dim) return lfail(L, SPH_E_INVALID, "network and handle dimensions differ");
  cudaStream_t s = (cudaStream_t)stream;
  int r = sph_build_cells(h, stream);
  if (r == SPH_OK) r = sph_advection_step(h, nullptr, stream);
  if (r != SPH_OK) return r;
  const int K = h->b.n_inst;
  std::vector<sph_diag> d0(K), d1(K);
  r = sph_diagnostics(h, d0.data(), stream);
  if (r != SPH_OK) return r;
  const int64_t n = h->b.n;
  r = build_inputs(h, L, s);
  if (r != SPH_OK) return lfail(L, r, "building the network inputs failed");
  if (!L->saveC && !nalloc(L, &L->saveC, K)) return lfail(L, SPH_E_OOM, "allocation failed");
  cudaMemcpyAsync(L->saveP, h->b.PS, sizeof(int4) * n, cudaMemcpyDeviceToDevice, s);
  cudaMemcpyAsync(L->saveV, h->b.VS, sizeof(float4) * n, cudaMemcpyDeviceToDevice, s);
  cudaMemcpyAsync(L->saveC, h->b.ctrl, sizeof(sph::Ctrl) * K, cudaMemcpyDeviceToDevice, s);
  forward(h, L, s, false);
  if (h->b.dim == 2)
    k_apply<2><<<blocks_for(n), 256, 0, s>>>(n, h->b.PS, h->b.VS, h->b.inst_of, h->b.inst, h->b.ctrl, L->Y, h->b.glob);
  else
    k_apply<3><<<blocks_for(n), 256, 0, s>>>(n, h->b.PS, h->b.VS, h->b.inst_of, h->b.inst, h->b.ctrl, L->Y, h->b.glob);
  k_learned_clock<<<1, 256, 0, s>>>(K, h->b.ctrl);
  sph::launch_vmax(h->b, s, &h->launches);
  h->cells_valid = false;
  r = sph_diagnostics(h, d1.data(), stream);
  bool ok = (r == SPH_OK);
  for (int k = 0; k < K && ok; ++k) {
    const double drift = std::fabs(d1[k].energy - d0[k].energy) / std::max(std::fabs(d0[k].energy), 1e-300);
    if (!(d1[k].mean_rho_dev <= max_mean_rho_dev) || !(drift <= max_energy_drift)) ok = false;
  }
  if (used_learned) *used_learned = ok ? 1 : 0;
  if (ok) return SPH_OK;
  // fall back: restore the step's start and run the acoustic substeps
  h->err.clear();
  cudaMemsetAsync(h->b.glob, 0, sizeof(int), s);                    // clear error bits of the trial
  cudaMemcpyAsync(h->b.PS, L->saveP, sizeof(int4) * n, cudaMemcpyDeviceToDevice, s);
  cudaMemcpyAsync(h->b.VS, L->saveV, sizeof(float4) * n, cudaMemcpyDeviceToDevice, s);
  cudaMemcpyAsync(h->b.ctrl, L->saveC, sizeof(sph::Ctrl) * K, cudaMemcpyDeviceToDevice, s);
  h->cells_valid = true;
  for (int guard = 0;; ++guard) {
    int32_t done = 0;
    r = sph_acoustic_substep(h, &done, nullptr, stream);
    if (r != SPH_OK) return r;
    if (done) break;
    if (guard > 1000000) return SPH_E_UNSTABLE;
  }
  return SPH_OK;
}

}  // extern "C"

