// update.cu -- the fp32-accurate updates C -= A B^T of GPTQ's block loop and of the factor's
// sweep, on the tcgen05 tensor cores of sm_103a.
//
// A [rows, K] and B [cols, K] are fp32 matrices given as three bf16 parts each, x = x1 + x2 + x3
// (split3: the parts carry x to about 2^-24 relative), stored once: row r holds its parts side
// by side, three segments of K.  The six products whose weight is above 2^-24, A1 B3, A3 B1,
// A2 B2, A1 B2, A2 B1 and A1 B1, are accumulated in fp32 in tensor memory, the small ones over
// all of K first: the tensor cores' accumulation loses up to about a unit in the last place of
// the running sum per 16 of K, so only the K / 16 steps of A1 B1 add to the error, not the
// 6 K / 16 of all six.  The tile is subtracted from C in a TMA reduce-add, which the L2 applies
// in fp32 round-to-nearest without the SM reading C.
//
// Persistent: one CTA per SM takes 128 x 256 tiles in a strided loop.  Warp 0 loads (a ring of
// four 48 KB stages, 64 of K each), warp 1 owns the tensor memory and issues the MMAs, warps
// 2-9 are the epilogue.  Two 256-column accumulators alternate, so a tile's epilogue runs
// beside the next one's loads and MMAs.  Every wait is bounded; one that runs out sets the error
// flag and turns the CTA's tiles into NaN, and the CTA's loads and MMAs in flight finish before it ends.
//
// The factor's form (kFactor) updates the rows below diagonal block j (rows, relative to the
// first row below it) with A = L_:j and B = [L_:j ; X_j,:^T], one operand array Bo:
//   * the trailing square, only its 128 x 256 tiles on and below the diagonal (and of a tile
//     crossing it only the columns up to the diagonal block's end): half the products and half
//     the traffic, so what is live of both halves stays in L2;
//   * the inverse's columns 0 .. xcols - 1;
//   * CTA 0 takes only the next diagonal block: its update goes from tensor memory to shared
//     memory, where the CTA factors and inverts it (factor_block128) and writes the inverse
//     Z_j+1, while the other CTAs run the rest of the update.  So the serial diagonal block
//     runs beside the update and not after it.  It is the step's critical path, so nothing of it
//     goes through the ring: the operand (A and B are the same rows) is loaded once, whole, and the
//     block by TMA too.  One GB300: 4.0 us to the tile in shared memory, of which the MMAs take 2.0,
//     against 5.5 through the ring with the block's rows read by the epilogue's threads (n = 4096
//     factor 847 -> 802 us in a graph).
//
// One GB300: the K = 512 update of 4096 x 3584 takes 56 us with the operands' first touch from
// HBM (the tensor pipe 73 % busy); what it cannot hide are the ends of the last round of tiles
// (448 tiles over 152 SMs), the ring's first loads and the last tile's reduce-add.
#include <algorithm>

#include "factor_block.cuh"
#include "hscale_internal.h"
#include "tcgen05.cuh"
#include "tma.cuh"

namespace hscale {
namespace {

constexpr int kBM = 128, kBN = 256, kBK = 64, kStages = 4;
constexpr uint32_t kHalfTileBytes = 128 * kBK * 2;         // 128 rows of one operand: 16 KB
constexpr uint32_t kStageBytes = 3 * kHalfTileBytes;       // A's 128 rows and B's 256
constexpr int kProducts = 6;
constexpr int kEpiWarps = 8;
constexpr uint32_t kBoxCols = 32, kBoxRows = 32;           // one reduce-add box per warp
constexpr uint32_t kBoxBytes = kBoxCols * kBoxRows * 4;
// the ring, barriers in a 1 KB block (keeping the boxes 1 KB aligned for the 128-byte swizzle),
// the epilogue's boxes
constexpr uint32_t kUpdateSmemBytes = 1024 /* alignment */ + kStages * kStageBytes + 1024 + kEpiWarps * kBoxBytes;
constexpr uint32_t kDiagOperandBytes = 6 * kHalfTileBytes;  // the next diagonal block's
constexpr int kLoopThreads = 320;  // TMA warp, MMA warp, 8 epilogue warps
static_assert(kDiagSmemBytes <= (int)(kStages * kStageBytes), "the diagonal block is factored in the ring");
static_assert(kDiagOperandBytes + kNb * kNb * 4 <= kStages * kStageBytes, "its operands and itself are loaded into the ring");
static_assert(kNb * kLd * 4 <= (int)kDiagOperandBytes, "it takes the operands' place");

__device__ uint32_t g_update_flags = 0;

__device__ __forceinline__ void tma_reduce_add_2d(const CUtensorMap* map, const void* src, int32_t c0, int32_t c1) {
  asm volatile("cp.reduce.async.bulk.tensor.2d.global.shared::cta.add.tile.bulk_group [%0, {%1, %2}], [%3];" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(c0), "r"(c1), "r"(smem_addr(src))
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// every committed bulk operation has finished reading shared memory
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
// every committed bulk operation has completed
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

struct UpdateArgs {
  int K;            // columns of A and B
  int rows, cols;   // of C; kFactor: the trailing square's size (twice)
  int tiles;
  int whole;        // tiles from here on are 128 columns wide, two to a 128 x 256 tile (!kFactor)
  // kFactor
  int xcols;        // columns of the inverse
  float* C;         // [rows, cols] (kFactor: the trailing square)
  float* X;         // the inverse's rows
  int64_t ld;       // of C and X
  int32_t order0;   // order of the next diagonal block's first pivot
  int32_t* info;
};

// The tiles of one CTA in turn: rows from 128 tm, columns [col0, col_end), and whether the tile
// belongs to the inverse (kFactor).
template <bool kFactor>
struct Tiles {
  const UpdateArgs& s;
  int t, step, tiles_n, first;
  int tm, col0, col_end;
  bool inverse;
  __device__ explicit Tiles(const UpdateArgs& args) : s(args), first(0), tm(0) {
    tiles_n = ((kFactor ? s.xcols : s.cols) + kBN - 1) / kBN;
    step = kFactor ? (int)gridDim.x - 1 : (int)gridDim.x;
    t = (int)blockIdx.x;
    // kFactor: tile 0 is the next diagonal block, CTA 0's only one
    if (kFactor && t == 0) step = s.tiles;
    locate();
  }
  __device__ bool valid() const { return t < s.tiles; }
  __device__ void next() {
    t += step;
    locate();
  }
  __device__ void locate() {
    if (!valid()) return;
    if (kFactor) {
      // row tm has tm / 2 + 1 tiles of the trailing square, then the inverse's
      while (t >= first + tm / 2 + 1 + tiles_n) {
        first += tm / 2 + 1 + tiles_n;
        ++tm;
      }
      const int k = t - first;
      inverse = k > tm / 2;
      col0 = (inverse ? k - (tm / 2 + 1) : k) * kBN;
      col_end = inverse ? s.xcols : (tm + 1) * kBM;
    } else {
      const bool half = t >= s.whole;
      const int tile = half ? s.whole + (t - s.whole) / 2 : t;
      tm = tile / tiles_n;
      col0 = (tile - tm * tiles_n) * kBN + (half ? ((t - s.whole) & 1) * (kBN / 2) : 0);
      col_end = half ? min(s.cols, col0 + kBN / 2) : s.cols;
      inverse = false;
    }
  }
  __device__ bool narrow() const { return col_end - col0 <= 128; }
  __device__ int b_row() const { return (kFactor && inverse ? s.rows : 0) + col0; }
};

// The parts of product p, the small products first.
__device__ __forceinline__ int part_a(int p) { return p == 1 ? 2 : (p == 2 || p == 4 ? 1 : 0); }
__device__ __forceinline__ int part_b(int p) { return p == 0 ? 2 : (p == 2 || p == 3 ? 1 : 0); }

template <bool kFactor>
__global__ void __launch_bounds__(kFactor ? kDiagThreads : kLoopThreads, 1)
update_kernel(const __grid_constant__ CUtensorMap amap, const __grid_constant__ CUtensorMap bmap,
              const __grid_constant__ CUtensorMap cmap, const __grid_constant__ CUtensorMap xmap, UpdateArgs args) {
  extern __shared__ __align__(16) uint8_t dynamic_smem[];
  const uint32_t offset = (1024u - (smem_addr(dynamic_smem) & 1023u)) & 1023u;
  uint8_t* smem = dynamic_smem + offset;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + kStages * kStageBytes);
  uint64_t* empty = full + kStages;
  uint64_t* acc_full = empty + kStages;  // accumulator a holds a finished tile
  uint64_t* acc_empty = acc_full + 2;    // accumulator a has been read out
  uint64_t* mma_done = acc_empty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mma_done + 1);
  uint32_t* failed = tmem_slot + 1;
  const int warp = (int)warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
  const bool diagonal = kFactor && blockIdx.x == 0;
  const int chunks = (args.K + kBK - 1) / kBK;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&acc_full[a], 1);
      mbar_init(&acc_empty[a], kEpiWarps * 32);
    }
    mbar_init(mma_done, 1);
    *failed = 0u;
    mbar_fence_init();
    prefetch_tensormap(&amap);
    prefetch_tensormap(&bmap);
  }
  if (warp == 1) {
    tmem_alloc(smem_addr(tmem_slot), 2 * kBN);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_d = warp_uniform(*tmem_slot);
  // launched with programmatic dependent launch: the next kernel may be scheduled (after the TMEM
  // allocation), and the previous one's writes must be visible before the first load
  pdl_launch_dependents();
  pdl_wait_primary();

  if (warp == 0) {
    uint64_t policy;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(policy));
    uint32_t s = 0, parity = 1;  // position in the ring, over all of the CTA's tiles
    bool go = true;
    if (diagonal) {
      if (elect_one()) {
        // A and B are the same rows: three parts of two K steps, then the block itself in the
        // reduce-add's boxes
        mbar_arrive_expect_tx(&full[0], kDiagOperandBytes);
        for (int e = 0; e < 6; ++e)
          tma_load_3d(smem + e * kHalfTileBytes, &amap, (e & 1) * kBK, e >> 1, 0, &full[0], policy);
        mbar_arrive_expect_tx(&full[1], kNb * kNb * 4);
        for (int e = 0; e < 16; ++e)
          tma_load_2d(smem + kDiagOperandBytes + e * kBoxBytes, &cmap, (e & 3) * (int)kBoxCols,
                      (e >> 2) * (int)kBoxRows, &full[1], policy);
      }
      __syncwarp();
    }
    for (Tiles<kFactor> T(args); !diagonal && go && T.valid(); T.next()) {
      // B's boxes of 128 rows: amap's in kFactor, where A and B are one array, otherwise xmap's
      const bool narrow = T.narrow();
      const int a_row = T.tm * kBM, b_row = T.b_row();
      for (int p = 0; p < kProducts && go; ++p) {
        for (int c = 0; c < chunks; ++c) {
          if (!mbar_wait_warp(&empty[s], parity)) {
            go = false;
            break;
          }
          if (elect_one()) {
            uint8_t* st = smem + s * kStageBytes;
            mbar_arrive_expect_tx(&full[s], narrow ? 2 * kHalfTileBytes : kStageBytes);
            tma_load_3d(st, &amap, c * kBK, part_a(p), a_row, &full[s], policy);
            tma_load_3d(st + kHalfTileBytes, narrow ? (kFactor ? &amap : &xmap) : &bmap, c * kBK, part_b(p), b_row, &full[s], policy);
          }
          __syncwarp();
          if (++s == kStages) {
            s = 0;
            parity ^= 1u;
          }
        }
      }
    }
    if (!go && lane == 0) atomicOr(failed, 1u);
    __syncwarp();
    if (diagonal) {
      mbar_wait(&full[0], 0u);
      mbar_wait(&full[1], 0u);
    } else {
      ring_drain(full, kStages, s, parity);
    }
  } else if (warp == 1) {
    uint32_t s = 0, parity = 0, i = 0;  // i counts the CTA's tiles
    bool ok = true;
    if (diagonal) {
      ok = mbar_wait_warp(&full[0], 0u);
      tc_fence_after_sync();
      if (ok && elect_one()) {
        for (int p = 0; p < kProducts; ++p)
          for (int c = 0; c < 2; ++c)
            umma_bf16_block(tmem_d, smem_desc_k_sw128(smem_addr(smem + (2 * part_a(p) + c) * kHalfTileBytes)),
                            smem_desc_k_sw128(smem_addr(smem + (2 * part_b(p) + c) * kHalfTileBytes)),
                            idesc_bf16_f32(kBM, kNb), kBK / 16, (uint32_t)(p > 0 || c > 0));
        umma_commit(smem_addr(&acc_full[0]));
      }
      __syncwarp();
    }
    for (Tiles<kFactor> T(args); !diagonal && ok && T.valid(); T.next(), ++i) {
      const uint32_t idesc = T.narrow() ? idesc_bf16_f32(kBM, 128) : idesc_bf16_f32(kBM, kBN);
      const uint32_t a = i & 1u, d = tmem_d + a * kBN;
      // the accumulator's previous tile (two back) must have been read out of TMEM
      if (i >= 2 && !mbar_wait_warp(&acc_empty[a], ((i >> 1) - 1) & 1u)) {
        ok = false;
        break;
      }
      tc_fence_after_sync();
      for (int p = 0; p < kProducts && ok; ++p) {
        for (int c = 0; c < chunks; ++c) {
          if (!mbar_wait_warp(&full[s], parity)) {
            ok = false;
            break;
          }
          tc_fence_after_sync();
          if (elect_one()) {
            const uint32_t st = smem_addr(smem + s * kStageBytes);
            // a ragged last block of K is zero-filled by TMA: its 16-wide steps past K are left out
            umma_bf16_block(d, smem_desc_k_sw128(st), smem_desc_k_sw128(st + kHalfTileBytes), idesc,
                            min(kBK / 16, (args.K - c * kBK + 15) / 16), (uint32_t)(p > 0 || c > 0));
            umma_commit(smem_addr(&empty[s]));
            // fires once every MMA issued above has completed
            if (p + 1 == kProducts && c + 1 == chunks) umma_commit(smem_addr(&acc_full[a]));
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
  } else if (warp < 2 + kEpiWarps) {
    // epilogue: TMEM lane quarter warp % 4 (a warp may only touch that quarter), column half
    const uint32_t quarter = (uint32_t)(warp & 3), half = (uint32_t)((warp - 2) >> 2);
    const uint32_t lane_base = (quarter * 32u) << 16;
    uint8_t* box = smem + kStages * kStageBytes + 1024 + (uint32_t)(warp - 2) * kBoxBytes;
    if (diagonal) {
      // the next diagonal block: this thread's row, 64 columns, less the tile
      const int row = (int)quarter * 32 + lane;
      if (mbar_wait(&full[1], 0u) && mbar_wait_acc(&acc_full[0], 0u)) {
        tc_fence_after_sync();
        float* S = reinterpret_cast<float*>(smem) + row * kLd + 64 * half;  // over the operands
#pragma unroll
        for (int c = 0; c < 64; c += 32) {
          const uint8_t* src = smem + kDiagOperandBytes + (4 * quarter + 2 * half + c / 32) * kBoxBytes + lane * 128;
          uint32_t p[32];
          tmem_ld_32x32b_x32(tmem_d + lane_base + 64 * half + (uint32_t)c, p);
          tmem_ld_wait();
#pragma unroll
          for (int k = 0; k < 32; k += 4) {
            // the 128-byte swizzle holds 16-byte chunk i of a row at i ^ (row & 7)
            const float4 b = *reinterpret_cast<const float4*>(src + ((k / 4) ^ (lane & 7)) * 16);
            *reinterpret_cast<float4*>(S + c + k) =
                make_float4(__fsub_rn(b.x, __uint_as_float(p[k])), __fsub_rn(b.y, __uint_as_float(p[k + 1])),
                            __fsub_rn(b.z, __uint_as_float(p[k + 2])), __fsub_rn(b.w, __uint_as_float(p[k + 3])));
          }
        }
      } else {
        atomicOr(failed, 1u);
      }
    } else {
      uint32_t i = 0;
      bool alive = true;
      for (Tiles<kFactor> T(args); T.valid(); T.next(), ++i) {
        const uint32_t a = i & 1u;
        const CUtensorMap* map = kFactor && T.inverse ? &xmap : &cmap;
        const int row0 = T.tm * kBM + (int)quarter * 32, col0 = T.col0 + (int)half * 128, col_end = T.col_end;
        // subtract 32 columns of the tile (values p) from C
        auto subtract = [&](const uint32_t (&p)[32], int c) {
          // the previous box must have been read out of the buffer
          if (lane == 0) bulk_wait_read();
          __syncwarp();
          // row `lane` of the box holds 128 bytes; the 128-byte swizzle puts its 16-byte chunk k
          // at k ^ (lane & 7), so a warp's stores hit every bank once
          float4* rowp = reinterpret_cast<float4*>(box + lane * 128);
#pragma unroll
          for (int k = 0; k < 8; ++k)
            rowp[k ^ (lane & 7)] = make_float4(-__uint_as_float(p[4 * k]), -__uint_as_float(p[4 * k + 1]),
                                               -__uint_as_float(p[4 * k + 2]), -__uint_as_float(p[4 * k + 3]));
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0 && row0 < args.rows) {
            tma_reduce_add_2d(map, box, col0 + c, row0);
            bulk_commit();
          }
        };
        if (!mbar_wait_acc(&acc_full[a], (i >> 1) & 1u)) {
          alive = false;
          break;
        }
        tc_fence_after_sync();
        const uint32_t src = tmem_d + a * kBN + lane_base + half * 128;
        if (kFactor) {
          // 128 registers a thread: 32 columns at a time
#pragma unroll 1
          for (int c = 0; c < 128 && col0 + c < col_end; c += 32) {
            uint32_t p[32];
            tmem_ld_32x32b_x32(src + (uint32_t)c, p);
            tmem_ld_wait();
            subtract(p, c);
          }
          tc_fence_before_sync();
          mbar_arrive(&acc_empty[a]);
        } else {
          uint32_t p[128];
#pragma unroll
          for (int c = 0; c < 128; c += 32)
            tmem_ld_32x32b_x32(src + (uint32_t)c, *reinterpret_cast<uint32_t(*)[32]>(p + c));
          tmem_ld_wait();
          tc_fence_before_sync();
          mbar_arrive(&acc_empty[a]);
#pragma unroll
          for (int c = 0; c < 128; c += 32)
            if (col0 + c < col_end) subtract(*reinterpret_cast<uint32_t(*)[32]>(p + c), c);
        }
      }
      if (!alive) atomicOr(failed, 1u);
      // the reduce-adds complete before the CTA ends
      if (lane == 0) bulk_wait_all();
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  const bool bad = *failed != 0;
  if (bad && threadIdx.x == 0) atomicOr(&g_update_flags, kErrMbarTimeout);
  if (kFactor && diagonal) {
    // Z_j+1 into the diagonal block of the inverse (zeros above its diagonal)
    float* xo = args.X + args.order0;
    if (!bad) {
      factor_block128(offset, xo, args.ld, args.info, args.order0);
    } else {
      for (int e = (int)threadIdx.x; e < kNb * kNb; e += kDiagThreads)
        xo[(e / kNb) * args.ld + e % kNb] = __int_as_float(0x7FC00000);
    }
  } else if (bad && warp >= 2 && warp < 2 + kEpiWarps) {
    // a wait that ran out makes the CTA's tiles NaN
    for (Tiles<kFactor> T(args); T.valid(); T.next()) {
      float* base = kFactor && T.inverse ? args.X : args.C;
      const int row = T.tm * kBM + (warp & 3) * 32 + lane, c0 = T.col0 + ((warp - 2) >> 2) * 128;
      if (row < args.rows)
        for (int c = c0; c < min(c0 + 128, T.col_end); ++c)
          base[(int64_t)row * args.ld + c] = __int_as_float(0x7FC00000);
    }
  }
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc(tmem_d, 2 * kBN);
  }
}

// A split operand: `rows` rows of three parts of K bf16, boxes of 64 x 1 x box_rows.
cudaError_t encode_operand(EncodeTiledFn encode, CUtensorMap* map, const void* p, int64_t rows, int64_t K,
                           int box_rows) {
  const cuuint64_t dims[3] = {(cuuint64_t)K, 3, (cuuint64_t)rows};
  const cuuint64_t strides[2] = {(cuuint64_t)K * 2, (cuuint64_t)K * 6};
  const cuuint32_t box[3] = {(cuuint32_t)kBK, 1, (cuuint32_t)box_rows};
  const cuuint32_t estr[3] = {1, 1, 1};
  return encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(p), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS
             ? cudaSuccess
             : cudaErrorInvalidValue;
}

// C [rows, cols] fp32 (row stride ld), reduce-added in 32 x 32 boxes.
cudaError_t encode_target(EncodeTiledFn encode, CUtensorMap* map, float* C, int64_t rows, int64_t cols, int64_t ld) {
  if ((reinterpret_cast<uintptr_t>(C) & 15) != 0 || (ld * 4) % 16 != 0) return cudaErrorInvalidValue;
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)ld * 4};
  const cuuint32_t box[2] = {kBoxCols, kBoxRows};
  const cuuint32_t estr[2] = {1, 1};
  return encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, C, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS
             ? cudaSuccess
             : cudaErrorInvalidValue;
}

template <bool kFactor>
cudaError_t launch_update(const CUtensorMap& amap, const CUtensorMap& bmap, const CUtensorMap& cmap,
                          const CUtensorMap& xmap, const UpdateArgs& args, cudaStream_t stream) {
  cudaError_t err = ensure_dynamic_smem(reinterpret_cast<const void*>(update_kernel<kFactor>), (int)kUpdateSmemBytes);
  if (err != cudaSuccess) return err;
  // persistent: one CTA per SM (the shared-memory ring allows no more), tiles strided
  DeviceInfo info;
  if ((err = current_device_info(&info)) != cudaSuccess) return err;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)std::min(args.tiles, info.sm_count), 1, 1);
  cfg.blockDim = dim3(kFactor ? kDiagThreads : kLoopThreads, 1, 1);
  cfg.dynamicSmemBytes = kUpdateSmemBytes;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  err = cudaLaunchKernelEx(&cfg, update_kernel<kFactor>, amap, bmap, cmap, xmap, args);
  if (err != cudaSuccess) return err;
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_split_update(const void* a, const void* b, int64_t rows, int64_t cols, int64_t K, float* C,
                                int64_t ld, cudaStream_t stream) {
  EncodeTiledFn encode = nullptr;
  cudaError_t err = encode_tiled_fn(&encode);
  if (err != cudaSuccess) return err;
  CUtensorMap amap, bmap, bhalf, cmap;
  if ((err = encode_operand(encode, &amap, a, rows, K, kBM)) != cudaSuccess) return err;
  if ((err = encode_operand(encode, &bmap, b, cols, K, kBN)) != cudaSuccess) return err;
  if ((err = encode_operand(encode, &bhalf, b, cols, K, kBN / 2)) != cudaSuccess) return err;
  if ((err = encode_target(encode, &cmap, C, rows, cols, ld)) != cudaSuccess) return err;
  const int64_t tiles = ((rows + kBM - 1) / kBM) * ((cols + kBN - 1) / kBN);
  if (tiles > INT32_MAX / 2) return cudaErrorInvalidValue;
  UpdateArgs args = {};
  args.K = (int)K;
  args.rows = (int)rows;
  args.cols = (int)cols;
  // The tiles of a last round that leaves half of the SMs idle are halved: the round is bound by each
  // SM's MMAs and loads.  Above that line some SM would have two halves, a whole tile's time.  4096 x
  // 4096 in blocks of 128: three of its seven updates, 567 -> 554 us; quarters where three quarters are
  // idle gave no more.
  DeviceInfo info;
  if ((err = current_device_info(&info)) != cudaSuccess) return err;
  const int last = (int)(tiles % info.sm_count);
  args.whole = 2 * last <= info.sm_count ? (int)tiles - last : (int)tiles;
  args.tiles = (int)tiles + ((int)tiles - args.whole);
  args.C = C;
  args.ld = ld;
  return launch_update<false>(amap, bmap, cmap, bhalf, args, stream);
}

cudaError_t launch_factor_update(const void* operand, int64_t rows, int64_t xcols, float* C, float* X, int64_t ld,
                                 int32_t order0, int32_t* info, cudaStream_t stream) {
  EncodeTiledFn encode = nullptr;
  cudaError_t err = encode_tiled_fn(&encode);
  if (err != cudaSuccess) return err;
  CUtensorMap amap, bmap, cmap, xmap;
  if ((err = encode_operand(encode, &amap, operand, rows + xcols, kNb, kBM)) != cudaSuccess) return err;
  if ((err = encode_operand(encode, &bmap, operand, rows + xcols, kNb, kBN)) != cudaSuccess) return err;
  if ((err = encode_target(encode, &cmap, C, rows, rows, ld)) != cudaSuccess) return err;
  if ((err = encode_target(encode, &xmap, X, rows, xcols, ld)) != cudaSuccess) return err;
  UpdateArgs args = {};
  args.K = kNb;
  args.rows = args.cols = (int)rows;
  args.xcols = (int)xcols;
  const int xt = (int)((xcols + kBN - 1) / kBN);
  for (int tm = 0; tm < (int)(rows / kBM); ++tm) args.tiles += tm / 2 + 1 + xt;
  args.C = C;
  args.X = X;
  args.ld = ld;
  args.order0 = order0;
  args.info = info;
  return launch_update<true>(amap, bmap, cmap, xmap, args, stream);
}

cudaError_t read_update_device_error(uint32_t* flags) {
  uint32_t v = 0;
  cudaError_t err = cudaMemcpyFromSymbol(&v, g_update_flags, sizeof v);
  if (err != cudaSuccess) return err;
  *flags = v;
  if (v) {
    const uint32_t zero = 0;
    err = cudaMemcpyToSymbol(g_update_flags, &zero, sizeof zero);
  }
  return err;
}

}  // namespace hscale
