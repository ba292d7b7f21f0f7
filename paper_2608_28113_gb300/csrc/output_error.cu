// output_error.cu -- the layer-output error ||X dW^T||_F^2 of an NVFP4 quantization (Eq. 3)
// on the tcgen05 tensor cores of sm_103a.
//
//   residual_kernel       dW = W - W_hat with W_hat = s_g * E4M3(code) * E2M1(nibble), as a
//                         bf16 pair hi = bf16(dW), lo = bf16(dW - hi), written as one matrix
//                         [hi | lo] per row (each half zero-padded to n_pad = 64 * ceil(n/64))
//   output_error_kernel   C = [X | X] [hi | lo]^T = X (hi + lo)^T on the tensor cores (bf16
//                         operands, fp32 accumulation in tensor memory), fused with the sum of
//                         squares of C: one fp64 partial per 128 x 256 tile of C
//   reduce_kernel         the partials summed in tile order, added to the caller's scalar
//   gemm_kernel<3>        H += X^T X, the full Hessian of Algorithm 3, with the same tensor-
//                         core pipeline over K = tokens, reading X as it is (both operands
//                         MN-major), and an epilogue that adds each 128 x 256 tile of the
//                         product into H; tiles wholly below the diagonal are skipped (the
//                         factor reads the upper triangle only).  K runs in segments of 2048
//                         tokens, each accumulated from zero and folded into a running sum
//                         in tensor memory
//   (hessian_cluster.cu)  the same for widths with few tiles: a cluster per tile splits K
//   transpose_kernel,     the same for X whose rows are not 16-byte aligned (no TMA): X is
//   gemm_kernel<1>        transposed into the workspace (tokens contiguous per channel)
//                         and both operands are K-major
//
// The residual is rounded once (one FMA of the exact w - s_g * (l q)), and hi + lo carries
// it to a relative 2^-17, so the GEMM sees dW, not a difference of two large products.
//
// GEMM tile: 128 tokens x 256 outputs, K in steps of 64 bf16 (one 128-byte swizzle atom
// per row), a 4-stage ring of TMA loads (48 KB per stage).  Warp 0 issues the loads, warp 1
// owns the tensor memory and issues the MMAs (M = 128, N = 256, K = 16 each), warps 2-9
// read the 128 x 256 fp32 accumulator back (each warp half the columns of its 32-lane
// quarter) and square and sum it.  Every wait is bounded; one that runs out sets the error flag and the
// tile's partial becomes NaN, and the CTA's loads and MMAs in flight finish before it ends.
#include <algorithm>
#include <cuda_bf16.h>

#include "hscale_device.cuh"
#include "hscale_internal.h"
#include "tcgen05.cuh"
#include "tma.cuh"

namespace hscale {
namespace {

constexpr int kBM = 128, kBN = 256, kBK = 64, kStages = 4;
constexpr int kGemmThreads = 320;  // TMA warp, MMA warp, 8 epilogue warps
constexpr uint32_t kTileABytes = kBM * kBK * 2;  // 16 KB
constexpr uint32_t kTileBBytes = kBN * kBK * 2;  // 32 KB
constexpr uint32_t kStageBytes = kTileABytes + kTileBBytes;
// Full Hessian (modes 1, 3) and output error (mode 0): the tensor cores accumulate in fp32
// with an error that grows with the accumulation length (the Hessian's diagonal comes out
// low by about 0.9 u per K = 16 step, measured), so each tile's K loop is cut into
// segments of kSegBlocks K blocks (2048 tokens, or 2048 of the 2 n channels of [X | X]).
// Each segment accumulates from zero in TMEM columns [0, 256); the epilogue warps add it in
// fp32 round-to-nearest into a running sum kept in TMEM columns [256, 512) and, after the
// last segment, add the running sum into H (or square and sum it).  With H = 0 before the
// call the Hessian is bit for bit that of successive calls of 2048 tokens, whatever the
// call size.
constexpr int kSegBlocks = 32;
constexpr uint32_t kTmemColsSeg = 2 * kBN;
constexpr uint32_t kGemmSmemBytes = kStages * kStageBytes + 1024 /* alignment */ + 256 /* barriers */;
constexpr uint32_t kIdesc = idesc_bf16_f32(kBM, kBN);
constexpr uint32_t kIdescMN = idesc_bf16_f32_mn(kBM, kBN);
constexpr uint32_t kBoxBytes = 64 * kBK * 2;  // mode 3: one 64-channel x 64-token TMA box

__device__ uint32_t g_output_error_flags = 0;

// ---------------------------------------------------------------- residual
__device__ __forceinline__ uint32_t bf16x2_pack(__nv_bfloat16 lo, __nv_bfloat16 hi) {
  return (uint32_t)__bfloat16_as_ushort(lo) | ((uint32_t)__bfloat16_as_ushort(hi) << 16);
}

// One thread per 16-element slot of a [hi | lo] row: slots below ng hold a group, the rest
// of the padded half is written with zeros.
// kWide: w and every row of dw2 are 32-byte aligned.
// 4096 x 4096: 23.0 us with 16-byte accesses and a 64-bit division per slot, 17.1 now (110 MB).
template <bool kWide>
__global__ void __launch_bounds__(256) residual_kernel(const uint4* __restrict__ w, int64_t m, int ng,
                                                       int ng_pad, const float* __restrict__ global_scale,
                                                       const uint8_t* __restrict__ codes,
                                                       const uint2* __restrict__ packed,
                                                       uint4* __restrict__ dw2, int64_t ld_dw2) {
  const float sg = *global_scale;
  const int64_t slots = m * ng_pad;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < slots;
       t += (int64_t)gridDim.x * blockDim.x) {
    // 32-bit arithmetic where it reaches: a 64-bit division is a call of some 70 instructions
    const int64_t r = slots <= UINT32_MAX ? (int64_t)((uint32_t)t / (uint32_t)ng_pad) : t / ng_pad;
    const int i = (int)(t - r * ng_pad);
    uint4* hi_dst = dw2 + (r * ld_dw2 + (int64_t)i * 16) / 8;
    uint4* lo_dst = dw2 + (r * ld_dw2 + (int64_t)(ng_pad + i) * 16) / 8;
    if (i >= ng) {
      const uint4 z = make_uint4(0u, 0u, 0u, 0u);
      st_32<kWide>(hi_dst, z, z);
      st_32<kWide>(lo_dst, z, z);
      continue;
    }
    const int64_t g = r * ng + i;
    uint4 p0, p1;
    ld_stream_32<kWide>(w + 2 * g, p0, p1);
    const uint32_t wb[8] = {p0.x, p0.y, p0.z, p0.w, p1.x, p1.y, p1.z, p1.w};
    uint32_t c = codes[g] & 0x7Fu;
    c = c < 1u ? 1u : (c > kE4M3MaxCode ? kE4M3MaxCode : c);
    const float l = e4m3_mag(c);
    const uint2 nib = packed[g];
    uint32_t hw[8], lw[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      __nv_bfloat16 h2[2], l2[2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int j = 2 * k + e;
        const uint32_t nb = ((j < 8 ? nib.x : nib.y) >> (4 * (j & 7))) & 0xFu;
        float lq = __fmul_rn(l, e2m1_from_raw((nb & 7u) << 22));  // exact: <= 6 significant bits
        if (nb & 8u) lq = -lq;
        const float wv = e ? bf16_hi(wb[k]) : bf16_lo(wb[k]);
        const float d = __fmaf_rn(-sg, lq, wv);  // w - s_g * l * q, rounded once
        h2[e] = __float2bfloat16_rn(d);
        l2[e] = __float2bfloat16_rn(__fsub_rn(d, __bfloat162float(h2[e])));
      }
      hw[k] = bf16x2_pack(h2[0], h2[1]);
      lw[k] = bf16x2_pack(l2[0], l2[1]);
    }
    st_32<kWide>(hi_dst, make_uint4(hw[0], hw[1], hw[2], hw[3]), make_uint4(hw[4], hw[5], hw[6], hw[7]));
    st_32<kWide>(lo_dst, make_uint4(lw[0], lw[1], lw[2], lw[3]), make_uint4(lw[4], lw[5], lw[6], lw[7]));
  }
}

// ---------------------------------------------------------------- GEMM + sum of squares
__device__ __forceinline__ float sum_squares32(const uint32_t (&r)[32]) {
  float t[16];
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const float a = __uint_as_float(r[2 * j]), b = __uint_as_float(r[2 * j + 1]);
    t[j] = __fmaf_rn(a, a, __fmul_rn(b, b));
  }
#pragma unroll
  for (int step = 1; step < 16; step <<= 1)
#pragma unroll
    for (int j = 0; j + step < 16; j += 2 * step) t[j] = __fadd_rn(t[j], t[j + step]);
  return t[0];
}

// kMode 0: the sum-of-squares GEMM of the output error (K runs over [X | X], kb_half
// blocks per half).  kMode 1: H[rows, cols] += A B^T over kb_half K blocks, both operands
// rows of X^T, tiles wholly below the diagonal skipped.  kMode 3: kMode 1 read from X itself
// ([tokens, n], channels contiguous): each stage loads 64-channel x 64-token boxes and
// the MMAs take both operands MN-major, so no transpose is needed.
// Tile t of a persistent GEMM's sequence (tiles_n column tiles per row of tiles) in groups of
// kRasterRows rows of tiles, column-major within a group: the tiles in flight at once (about
// one per SM) then cover a few row strips of A and a part of B's column strips, rather than
// every column strip of B for one or two row strips, so their operands stay in L2.
constexpr int kRasterRows = 8;
__device__ __forceinline__ void raster_tile(int t, int tiles_n, int tiles_total, int& tm, int& tn) {
  const int tiles_m = tiles_total / tiles_n;
  const int first = t / (kRasterRows * tiles_n) * kRasterRows;
  const int rows = min(kRasterRows, tiles_m - first);
  const int within = t - first * tiles_n;
  tm = first + within % rows;
  tn = within / rows;
}

template <int kMode>
__global__ void __launch_bounds__(kGemmThreads, 1)
gemm_kernel(const __grid_constant__ CUtensorMap xmap, const __grid_constant__ CUtensorMap wmap,
            int kb_half, int tiles_n, int tiles_total,
            double* __restrict__ partials, float* __restrict__ H, int64_t h_rows, int64_t h_cols, int64_t ld_h,
            int grouped) {
  extern __shared__ __align__(16) uint8_t dynamic_smem[];
  uint8_t* smem = dynamic_smem + ((1024u - (smem_addr(dynamic_smem) & 1023u)) & 1023u);
  uint8_t* tile_a = smem;
  uint8_t* tile_b = smem + kStages * kTileABytes;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + kStages * kStageBytes);
  uint64_t* empty = full + kStages;
  uint64_t* seg_full = empty + kStages;  // a segment's partial is complete
  uint64_t* seg_empty = seg_full + 1;    // the partial has been read out
  uint64_t* mma_done = seg_empty + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mma_done + 1);
  uint32_t* failed = tmem_slot + 1;
  double* warp_sum = reinterpret_cast<double*>(smem + kStages * kStageBytes + 128);
  constexpr bool kHessian = kMode == 1 || kMode == 3;
  // The output error is persistent: a CTA takes tiles blockIdx.x, + gridDim.x, ...  Its segments
  // run on across its tiles (one segment counter), so the MMAs of a tile's first segment start
  // as soon as the previous tile's last partial has been read out, alongside that tile's sum of
  // squares.  The Hessian modes take one tile per CTA.
  constexpr bool kPersistent = kMode == 0;

  const int warp = (int)warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int ntiles = kPersistent ? (tiles_total - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x : 1;
  const int tile_m = blockIdx.x / tiles_n, tile_n = blockIdx.x - tile_m * tiles_n;
  constexpr bool kAccum = kMode != 0;
  const int kb_total = kAccum ? kb_half : 2 * kb_half;
  // H is symmetric and only its upper triangle is used: a tile wholly below the diagonal
  // (every column index below every row index) is skipped, uniformly for the whole CTA
  if (kHessian && (int64_t)(tile_n + 1) * kBN <= (int64_t)tile_m * kBM) return;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(seg_full, 1);
    mbar_init(seg_empty, 256);  // every epilogue thread arrives
    mbar_init(mma_done, 1);
    *failed = 0u;
    mbar_fence_init();
    prefetch_tensormap(&xmap);
    prefetch_tensormap(&wmap);
  }
  if (warp == 1) {
    tmem_alloc(smem_addr(tmem_slot), kTmemColsSeg);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_d = warp_uniform(*tmem_slot);
  if (warp == 0) {
    uint64_t policy;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(policy));
    uint32_t s = 0, parity = 1;  // the ring's position, over all of the CTA's tiles
    bool go = true;
    for (int i = 0; i < ntiles && go; ++i) {
      const int t = (int)blockIdx.x + i * (int)gridDim.x;
      int tm = t / tiles_n, tn = t - tm * tiles_n;
      if (kMode == 0) raster_tile(t, tiles_n, tiles_total, tm, tn);
      for (int kb = 0; kb < kb_total; ++kb) {
        if (!mbar_wait_warp(&empty[s], parity)) {
          if (lane == 0) atomicOr(failed, 1u);
          go = false;
          break;
        }
        if (elect_one()) {
          mbar_arrive_expect_tx(&full[s], kStageBytes);
          uint8_t* a = tile_a + s * kTileABytes;
          uint8_t* b = tile_b + s * kTileBBytes;
          if (kMode == 3 && grouped) {
            // boxes of two and four 64-channel groups
            tma_load_3d(a, &xmap, 0, kb * kBK, tm * (kBM / 64), &full[s], policy);
            tma_load_3d(b, &wmap, 0, kb * kBK, tn * (kBN / 64), &full[s], policy);
          } else if (kMode == 3) {
#pragma unroll
            for (int j = 0; j < kBM / 64; ++j)
              tma_load_2d(a + j * kBoxBytes, &xmap, tm * kBM + 64 * j, kb * kBK, &full[s], policy);
#pragma unroll
            for (int j = 0; j < kBN / 64; ++j)
              tma_load_2d(b + j * kBoxBytes, &wmap, tn * kBN + 64 * j, kb * kBK, &full[s], policy);
          } else {
            const int xk = (kAccum || kb < kb_half ? kb : kb - kb_half) * kBK;
            tma_load_2d(a, &xmap, xk, tm * kBM, &full[s], policy);
            tma_load_2d(b, &wmap, kb * kBK, tn * kBN, &full[s], policy);
          }
        }
        __syncwarp();
        if (++s == kStages) {
          s = 0;
          parity ^= 1u;
        }
      }
    }
    ring_drain(full, kStages, s, parity);
  } else if (warp == 1) {
    // segments of kSegBlocks K blocks, each accumulated from zero
    const int nseg = (kb_total + kSegBlocks - 1) / kSegBlocks;
    uint32_t s = 0, parity = 0, gs = 0;  // gs counts the segments over all of the CTA's tiles
    bool ok = true;
    for (int i = 0; i < ntiles && ok; ++i) {
      for (int seg = 0; seg < nseg && ok; ++seg, ++gs) {
        // the previous segment's partial (of this tile or the one before) must have been
        // read out of TMEM
        if (gs >= 1 && !mbar_wait_warp(seg_empty, (gs - 1) & 1u)) {
          ok = false;
          break;
        }
        tc_fence_after_sync();
        const int kb0 = seg * kSegBlocks, kb1 = min(kb_total, kb0 + kSegBlocks);
        for (int kb = kb0; kb < kb1; ++kb) {
          if (!mbar_wait_warp(&full[s], parity)) {
            ok = false;
            break;
          }
          tc_fence_after_sync();
          if (elect_one()) {
            const uint32_t a = smem_addr(tile_a + s * kTileABytes), b = smem_addr(tile_b + s * kTileBBytes);
            if (kMode == 3) {
              // MN-major: 16 K rows are two 1024-byte swizzle atoms further
              const uint64_t ad = smem_desc_mn_sw128(a, kBoxBytes), bd = smem_desc_mn_sw128(b, kBoxBytes);
#pragma unroll
              for (int kk = 0; kk < kBK / 16; ++kk)
                umma_bf16(tmem_d, ad + 128 * kk, bd + 128 * kk, kIdescMN, (uint32_t)(kb > kb0 || kk > 0));
            } else {
              const uint64_t ad = smem_desc_k_sw128(a), bd = smem_desc_k_sw128(b);
#pragma unroll
              for (int kk = 0; kk < kBK / 16; ++kk)
                umma_bf16(tmem_d, ad + 2 * kk, bd + 2 * kk, kIdesc, (uint32_t)(kb > kb0 || kk > 0));
            }
            umma_commit(smem_addr(&empty[s]));
            // fires once every MMA issued above has completed
            if (kb + 1 == kb1) umma_commit(smem_addr(seg_full));
          }
          __syncwarp();
          if (++s == kStages) {
            s = 0;
            parity ^= 1u;
          }
        }
      }
    }
    if (!ok && lane == 0) atomicOr(failed, 1u);
    __syncwarp();
    umma_drain(mma_done);
  } else {
    // epilogue warps 2-9: TMEM lane quarter warp % 4 (a warp may only touch that quarter),
    // column half (warp - 2) / 4; each thread holds one tile row's half of the partial
    constexpr int kHalf = kBN / 2;
    const uint32_t quarter = (uint32_t)(warp & 3);
    const uint32_t cbase = (uint32_t)((warp - 2) >> 2) * kHalf;
    const uint32_t lane_base = (quarter * 32u) << 16;
    const int nseg = (kb_total + kSegBlocks - 1) / kSegBlocks;
    double acc = 0.0;
    bool alive = true;
    for (int i = 0; i < ntiles && alive; ++i) {
      const int t = (int)blockIdx.x + i * (int)gridDim.x;
      const int tm = t / tiles_n, tn = t - tm * tiles_n;
      const int64_t row = (int64_t)tm * kBM + quarter * 32 + lane;
      const int64_t col0 = (int64_t)tn * kBN + cbase;
      for (int seg = 0; seg < nseg; ++seg) {
        if (!mbar_wait_acc(seg_full, (uint32_t)(i * nseg + seg) & 1u)) {
          atomicOr(failed, 1u);
          alive = false;
          break;
        }
        tc_fence_after_sync();
        const bool last = seg + 1 == nseg;
        uint32_t p[kHalf];
#pragma unroll
        for (int c = 0; c < kHalf; c += 32)
          tmem_ld_32x32b_x32(tmem_d + lane_base + cbase + (uint32_t)c,
                             *reinterpret_cast<uint32_t(*)[32]>(p + c));
        tmem_ld_wait();
        if (!last || kPersistent) {
          // the partial is in registers: the MMAs may go on with the next segment (of this
          // tile or the next)
          tc_fence_before_sync();
          mbar_arrive(seg_empty);
        }
        if (seg > 0) {
          // fold into the running sum (TMEM columns [256, 512)), fp32 round-to-nearest
#pragma unroll
          for (int c = 0; c < kHalf; c += 32) {
            uint32_t q[32];
            tmem_ld_32x32b_x32(tmem_d + lane_base + kBN + cbase + (uint32_t)c, q);
            tmem_ld_wait();
#pragma unroll
            for (int j = 0; j < 32; ++j)
              p[c + j] = __float_as_uint(__fadd_rn(__uint_as_float(q[j]), __uint_as_float(p[c + j])));
          }
        }
        if (!last) {
#pragma unroll
          for (int c = 0; c < kHalf; c += 32)
            tmem_st_32x32b_x32(tmem_d + lane_base + kBN + cbase + (uint32_t)c, *reinterpret_cast<uint32_t(*)[32]>(p + c));
          tmem_st_wait();
          continue;
        }
        if (!kAccum) {
          // the output error: the sum of squares of the complete tile
#pragma unroll
          for (int c = 0; c < kHalf; c += 32) acc += (double)sum_squares32(*reinterpret_cast<uint32_t(*)[32]>(p + c));
          continue;
        }
        // the Hessian: the tile row added into H
        if (row < h_rows) {
          float* dst = H + row * ld_h + col0;
          if (col0 + kHalf <= h_cols && ((ld_h | col0) & 3) == 0 && (reinterpret_cast<uintptr_t>(H) & 15) == 0) {
#pragma unroll
            for (int q = 0; q < kHalf / 4; ++q) {
              float4 v = reinterpret_cast<float4*>(dst)[q];
              v.x += __uint_as_float(p[4 * q]);
              v.y += __uint_as_float(p[4 * q + 1]);
              v.z += __uint_as_float(p[4 * q + 2]);
              v.w += __uint_as_float(p[4 * q + 3]);
              reinterpret_cast<float4*>(dst)[q] = v;
            }
          } else {
#pragma unroll
            for (int q = 0; q < kHalf; ++q)
              if (col0 + q < h_cols) dst[q] += __uint_as_float(p[q]);
          }
        }
      }
    }
    if (!kAccum) {
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, off);
      if (lane == 0) warp_sum[warp - 2] = acc;
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  if (kAccum) {
    // a wait that ran out makes the whole tile NaN (written after the partial sums above)
    if (*failed && warp >= 2) {
      const uint32_t quarter = (uint32_t)(warp & 3);
      for (int i = 0; i < ntiles; ++i) {
        const int t = (int)blockIdx.x + i * (int)gridDim.x;
        const int tm = t / tiles_n, tn = t - tm * tiles_n;
        const int64_t row = (int64_t)tm * kBM + quarter * 32 + lane;
        const int64_t c0 = (int64_t)tn * kBN + ((warp - 2) >> 2) * (kBN / 2);
        if (row < h_rows)
          for (int64_t c = c0; c < c0 + kBN / 2 && c < h_cols; ++c) H[row * ld_h + c] = __int_as_float(0x7FC00000);
      }
      if (threadIdx.x == 64) atomicOr(&g_output_error_flags, kErrMbarTimeout);
    }
  } else if (threadIdx.x == 0) {
    double total = ((warp_sum[0] + warp_sum[1]) + (warp_sum[2] + warp_sum[3])) +
                   ((warp_sum[4] + warp_sum[5]) + (warp_sum[6] + warp_sum[7]));
    if (*failed) {
      atomicOr(&g_output_error_flags, kErrMbarTimeout);
      total = __longlong_as_double(0x7FF8000000000000ll);
    }
    partials[blockIdx.x] = total;
  }
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc(tmem_d, kTmemColsSeg);
  }
}

// X [tokens, n] (row stride ld_x, 2-byte aligned) -> Xt [n, tokens] (row stride ld_t, a multiple of
// 8), 64 x 64 tiles through shared memory: the reads run along channels, two bytes a lane (rows
// may start anywhere), the writes along tokens, eight bytes a thread (32 x 32 tiles with two-byte
// writes took 130 us for 16384 x 4095, now 57).
__global__ void __launch_bounds__(256) transpose_kernel(const uint16_t* __restrict__ x, int64_t tokens, int64_t n,
                                                        int64_t ld_x, uint16_t* __restrict__ xt, int64_t ld_t) {
  __shared__ uint16_t tile[64][66];
  const int64_t t0 = (int64_t)blockIdx.x * 64, c0 = (int64_t)blockIdx.y * 64;
  const int tx = threadIdx.x & 63, ty = threadIdx.x >> 6;  // 4 rows of 64 per pass
  uint16_t v[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const int64_t t = t0 + ty + 4 * k, c = c0 + tx;
    v[k] = (t < tokens && c < n) ? x[t * ld_x + c] : (uint16_t)0;
  }
#pragma unroll
  for (int k = 0; k < 16; ++k) tile[ty + 4 * k][tx] = v[k];
  __syncthreads();
  // four tokens of one channel each; rows of Xt reach ld_t >= tokens (its padding takes zeros)
  const int q = 4 * (threadIdx.x & 15), cy = threadIdx.x >> 4;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int cc = cy + 16 * k;
    if (c0 + cc >= n || t0 + q >= ld_t) continue;
    *reinterpret_cast<uint2*>(xt + (c0 + cc) * ld_t + t0 + q) =
        make_uint2((uint32_t)tile[q][cc] | ((uint32_t)tile[q + 1][cc] << 16),
                   (uint32_t)tile[q + 2][cc] | ((uint32_t)tile[q + 3][cc] << 16));
  }
}

// The partials summed in index order by one block (fixed tree), added to *out.
__global__ void __launch_bounds__(256) reduce_kernel(const double* __restrict__ partials, int64_t count,
                                                     double* __restrict__ out) {
  __shared__ double part[256];
  double s = 0.0;
  for (int64_t i = threadIdx.x; i < count; i += blockDim.x) s += partials[i];
  part[threadIdx.x] = s;
  __syncthreads();
  for (int step = 128; step > 0; step >>= 1) {
    if ((int)threadIdx.x < step) part[threadIdx.x] += part[threadIdx.x + step];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out += part[0];
}

}  // namespace

cudaError_t launch_residual(const void* w, int64_t m, int64_t n, const float* global_scale,
                            const uint8_t* codes, const uint8_t* packed, void* dw2, int64_t ld_dw2,
                            cudaStream_t stream) {
  DeviceInfo info;
  cudaError_t err = current_device_info(&info);
  if (err != cudaSuccess) return err;
  const int ng = (int)(n / 16);
  const int ng_pad = (int)((n + 63) / 64 * 4);
  const int64_t slots = m * ng_pad;
  const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((slots + 255) / 256, (int64_t)info.sm_count * 8));
  const bool wide = ((reinterpret_cast<uintptr_t>(w) | reinterpret_cast<uintptr_t>(dw2)) & 31) == 0 && ld_dw2 % 16 == 0;
  auto kernel = wide ? residual_kernel<true> : residual_kernel<false>;
  kernel<<<(unsigned)blocks, 256, 0, stream>>>(static_cast<const uint4*>(w), m, ng, ng_pad, global_scale, codes,
                                               reinterpret_cast<const uint2*>(packed), static_cast<uint4*>(dw2), ld_dw2);
  return cudaGetLastError();
}

int64_t output_error_tiles(int64_t tokens, int64_t m) {
  return ((tokens + kBM - 1) / kBM) * ((m + kBN - 1) / kBN);
}

cudaError_t launch_output_error(const void* x, int64_t tokens, int64_t n, int64_t ld_x, const void* dw2,
                                int64_t ld_dw2, int64_t m, double* out, double* partials,
                                cudaStream_t stream) {
  EncodeTiledFn encode = nullptr;
  cudaError_t err = encode_tiled_fn(&encode);
  if (err != cudaSuccess) return err;
  const int64_t n_pad = (n + kBK - 1) / kBK * kBK;
  CUtensorMap xmap, wmap;
  {
    const cuuint64_t dims[2] = {(cuuint64_t)n, (cuuint64_t)tokens};
    const cuuint64_t strides[1] = {(cuuint64_t)ld_x * 2};
    const cuuint32_t box[2] = {(cuuint32_t)kBK, (cuuint32_t)kBM};
    const cuuint32_t estr[2] = {1, 1};
    if (encode(&xmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(x), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return cudaErrorInvalidValue;
  }
  {
    const cuuint64_t dims[2] = {(cuuint64_t)(2 * n_pad), (cuuint64_t)m};
    const cuuint64_t strides[1] = {(cuuint64_t)ld_dw2 * 2};
    const cuuint32_t box[2] = {(cuuint32_t)kBK, (cuuint32_t)kBN};
    const cuuint32_t estr[2] = {1, 1};
    if (encode(&wmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(dw2), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return cudaErrorInvalidValue;
  }
  const cudaError_t attr_status =
      ensure_dynamic_smem(reinterpret_cast<const void*>(gemm_kernel<0>), (int)kGemmSmemBytes);
  if (attr_status != cudaSuccess) return attr_status;
  const int64_t tiles_n = (m + kBN - 1) / kBN;
  const int64_t tiles = output_error_tiles(tokens, m);
  // persistent: one CTA per SM (the shared-memory ring and the 512 TMEM columns allow no
  // more), tiles strided; one partial per CTA
  DeviceInfo info;
  if ((err = current_device_info(&info)) != cudaSuccess) return err;
  const int64_t grid = std::max<int64_t>(1, std::min<int64_t>(tiles, info.sm_count));
  gemm_kernel<0><<<(unsigned)grid, kGemmThreads, kGemmSmemBytes, stream>>>(
      xmap, wmap, (int)(n_pad / kBK), (int)tiles_n, (int)tiles, partials, nullptr, 0, 0, 0, 0);
  err = cudaGetLastError();
  if (err != cudaSuccess) return err;
  reduce_kernel<<<1, 256, 0, stream>>>(partials, grid, out);
  return cudaGetLastError();
}

int64_t hessian_full_ld(int64_t tokens) { return (tokens + 7) / 8 * 8; }

cudaError_t launch_hessian_full(const void* x, int64_t tokens, int64_t n, int64_t ld_x, float* H, int64_t ld_h,
                                void* xt, cudaStream_t stream) {
  EncodeTiledFn encode = nullptr;
  cudaError_t err = encode_tiled_fn(&encode);
  if (err != cudaSuccess) return err;
  const int64_t tiles_n = (n + kBN - 1) / kBN;
  const int64_t tiles = ((n + kBM - 1) / kBM) * tiles_n;
  DeviceInfo info;
  if ((err = current_device_info(&info)) != cudaSuccess) return err;
  const bool h_aligned = (reinterpret_cast<uintptr_t>(H) & 15) == 0 && ld_h % 4 == 0;
  const int cluster = hessian_cluster_size(tokens, n, h_aligned, info.sm_count);
  if ((reinterpret_cast<uintptr_t>(x) & 15) == 0 && ld_x % 8 == 0) {
    // X read as it is: 64-channel x 64-token boxes, MN-major operands (kMode 3).  Where n is whole
    // 64-channel groups, X is mapped as [n / 64][tokens][64] and one load takes an operand's two or
    // four boxes, instead of six loads a stage; otherwise a last group would reach past the rows'
    // ends, and each box is a load of its own, bounded by n.
    const bool grouped = n % 64 == 0;
    CUtensorMap map, bmap;
    const cuuint64_t dims2[2] = {(cuuint64_t)n, (cuuint64_t)tokens};
    const cuuint64_t strides2[1] = {(cuuint64_t)ld_x * 2};
    const cuuint64_t dims3[3] = {64, (cuuint64_t)tokens, (cuuint64_t)(n / 64)};
    const cuuint64_t strides3[2] = {(cuuint64_t)ld_x * 2, 128};
    const cuuint32_t estr[3] = {1, 1, 1};
    auto encode_x = [&](CUtensorMap* out, cuuint32_t groups) {
      const cuuint32_t box[3] = {64, (cuuint32_t)kBK, groups};
      return encode(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, grouped ? 3 : 2, const_cast<void*>(x), grouped ? dims3 : dims2,
                    grouped ? strides3 : strides2, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                    CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    };
    if (encode_x(&map, kBM / 64) != CUDA_SUCCESS || encode_x(&bmap, kBN / 64) != CUDA_SUCCESS)
      return cudaErrorInvalidValue;
    if (cluster > 1) return launch_hessian_cluster(cluster, map, bmap, true, grouped, tokens, n, H, ld_h, stream);
    err = ensure_dynamic_smem(reinterpret_cast<const void*>(gemm_kernel<3>), (int)kGemmSmemBytes);
    if (err != cudaSuccess) return err;
    gemm_kernel<3><<<(unsigned)tiles, kGemmThreads, kGemmSmemBytes, stream>>>(
        map, bmap, (int)((tokens + kBK - 1) / kBK), (int)tiles_n, (int)tiles, nullptr, H, n, n, ld_h, grouped ? 1 : 0);
    return cudaGetLastError();
  }
  // X with rows that are not 16-byte aligned: transposed first (tokens contiguous per
  // channel), then both operands K-major (kMode 1)
  const int64_t ld_t = hessian_full_ld(tokens);
  const dim3 tgrid((unsigned)((tokens + 63) / 64), (unsigned)((n + 63) / 64));
  transpose_kernel<<<tgrid, 256, 0, stream>>>(static_cast<const uint16_t*>(x), tokens, n, ld_x,
                                              static_cast<uint16_t*>(xt), ld_t);
  err = cudaGetLastError();
  if (err != cudaSuccess) return err;
  CUtensorMap amap, bmap;
  const cuuint64_t dims[2] = {(cuuint64_t)tokens, (cuuint64_t)n};
  const cuuint64_t strides[1] = {(cuuint64_t)ld_t * 2};
  const cuuint32_t estr[2] = {1, 1};
  const cuuint32_t abox[2] = {(cuuint32_t)kBK, (cuuint32_t)kBM};
  const cuuint32_t bbox[2] = {(cuuint32_t)kBK, (cuuint32_t)kBN};
  if (encode(&amap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, xt, dims, strides, abox, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
             CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS ||
      encode(&bmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, xt, dims, strides, bbox, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
             CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return cudaErrorInvalidValue;
  if (cluster > 1) return launch_hessian_cluster(cluster, amap, bmap, false, false, tokens, n, H, ld_h, stream);
  const cudaError_t attr_status =
      ensure_dynamic_smem(reinterpret_cast<const void*>(gemm_kernel<1>), (int)kGemmSmemBytes);
  if (attr_status != cudaSuccess) return attr_status;
  gemm_kernel<1><<<(unsigned)tiles, kGemmThreads, kGemmSmemBytes, stream>>>(
      amap, bmap, (int)((tokens + kBK - 1) / kBK), (int)tiles_n, (int)tiles, nullptr, H, n, n, ld_h, 0);
  return cudaGetLastError();
}

cudaError_t read_output_error_device_error(uint32_t* flags) {
  uint32_t v = 0;
  cudaError_t err = cudaMemcpyFromSymbol(&v, g_output_error_flags, sizeof v);
  if (err != cudaSuccess) return err;
  *flags = v;
  if (v) {
    const uint32_t zero = 0;
    err = cudaMemcpyToSymbol(g_output_error_flags, &zero, sizeof zero);
  }
  return err;
}

}  // namespace hscale
