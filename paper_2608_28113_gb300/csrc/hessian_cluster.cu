// hessian_cluster.cu -- H += X^T X (GPTQ's full Hessian) for widths whose tiles leave SMs idle:
// each 128 x 256 tile of H is computed by a thread-block cluster that splits the tokens.
//
// gemm_kernel (output_error.cu) takes one CTA per tile, so n = 1024 (20 tiles on and above the
// diagonal) leaves 132 of 152 SMs idle however many tokens there are.  Here the accumulation
// segments of 2048 tokens that a tile's CTA takes one after another go round the CTAs of a
// cluster: rank r computes segments r, r + kCluster, ...  The segments' partial tiles must be added
// in token order (a call over T tokens gives, bit for bit, what successive calls of 2048 tokens
// give), so after each round of kCluster segments every rank adds the round's partials of its own
// share of the columns, in order, from the other ranks' shared memory:
//   * a rank's epilogue warps copy half of its partial (128 columns) from tensor memory into a
//     64 KB staging area, columns one after another, and tell every rank (`ready`, one arrival per
//     rank);
//   * each rank reads its 128 / kCluster columns of every rank's half, in rank order, adds them
//     to its running sums in registers (fp32 round-to-nearest), and tells every rank (`done`).
// Two tensor-memory accumulators alternate, so this runs beside the next segment's loads and MMAs.
// At the end the sums go through the staging area into H, row by row.
//
// Every wait is bounded.  A rank in which one ran out may have handed the others a partial that was not
// complete, and its arrivals for rounds to come may have let them go on too soon; so it marks every rank
// before the barrier at the end, and the ranks write H after it: the whole tile is then NaN, and
// the error flag set.  Each rank's loads and MMAs in flight finish before that barrier, which also
// keeps every rank's shared memory until the others have read it.
//
// One GB300, 65536 tokens, by gemm_kernel and by clusters: n = 512 311 and 62-65 us, 1000 663 and 193,
// 2048 330 and 221.
#include <cooperative_groups.h>

#include <algorithm>

#include "hscale_internal.h"
#include "tcgen05.cuh"
#include "tma.cuh"

namespace cg = cooperative_groups;

namespace hscale {
namespace {

constexpr int kBM = 128, kBN = 256, kBK = 64, kStages = 3;
constexpr int kSegBlocks = 32;     // 2048 tokens, as in gemm_kernel
constexpr int kThreads = 320;      // TMA warp, MMA warp, 8 epilogue warps
constexpr uint32_t kTileABytes = kBM * kBK * 2, kTileBBytes = kBN * kBK * 2;
constexpr uint32_t kStageBytes = kTileABytes + kTileBBytes;
constexpr uint32_t kBoxBytes = 64 * kBK * 2;
constexpr uint32_t kStagingBytes = kBM * 129 * 4;  // 128 columns of a partial; rows of 129 at the end
constexpr uint32_t kSmemBytes = 1024 /* alignment */ + kStages * kStageBytes + kStagingBytes + 256;

__device__ uint32_t g_hessian_cluster_flags = 0;

__device__ __forceinline__ uint32_t mapa(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ float4 ld_cluster_v4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(addr)
               : "memory");
  return v;
}
// One arrival on rank `rank`'s barrier, releasing at cluster scope what this CTA's threads did
// before (ordered by the barrier among them).
__device__ __forceinline__ void arrive_remote(uint64_t* bar, uint32_t rank) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(mapa(smem_addr(bar), rank))
               : "memory");
}
__device__ __forceinline__ bool wait_cluster(uint64_t* bar, uint32_t parity) {
  const uint32_t a = smem_addr(bar);
  for (uint32_t i = 0; i < kMbarPollLimit; ++i) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(a), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}
// A wait ran out: every rank's `failed` is set.
template <int kCluster>
__device__ __forceinline__ void fail_cluster(volatile uint32_t* failed) {
  const uint32_t at = smem_addr(const_cast<uint32_t*>(failed));
  for (int q = 0; q < kCluster; ++q)
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(mapa(at, (uint32_t)q)), "r"(1u) : "memory");
}
__device__ __forceinline__ void epilogue_sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }

// kMN: X read as it is (both operands MN-major; `grouped`: one 3-D box per operand, see
// launch_hessian_full); otherwise rows of X^T (K-major).
template <int kCluster, bool kMN>
__global__ void __launch_bounds__(kThreads, 1)
hessian_cluster_kernel(const __grid_constant__ CUtensorMap amap, const __grid_constant__ CUtensorMap bmap, int kb_total,
                       int tiles_n, float* __restrict__ H, int64_t n, int64_t ld_h, int grouped) {
  extern __shared__ __align__(16) uint8_t dynamic_smem[];
  uint8_t* smem = dynamic_smem + ((1024u - (smem_addr(dynamic_smem) & 1023u)) & 1023u);
  uint8_t* tile_a = smem;
  uint8_t* tile_b = smem + kStages * kTileABytes;
  float* staging = reinterpret_cast<float*>(smem + kStages * kStageBytes);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + kStages * kStageBytes + kStagingBytes);
  uint64_t* empty = full + kStages;
  uint64_t* acc_full = empty + kStages;
  uint64_t* acc_empty = acc_full + 2;
  uint64_t* ready = acc_empty + 2;  // every rank's half is in its staging area
  uint64_t* done = ready + 1;       // every rank has read this rank's staging area
  uint64_t* mma_done = done + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mma_done + 1);
  volatile uint32_t* failed = tmem_slot + 1;

  cg::cluster_group cluster = cg::this_cluster();
  const int warp = (int)warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int rank = (int)cluster.block_rank();
  // the cluster's tile among those not wholly below the diagonal: row tm has tiles_n - tm / 2
  int tm = 0, tn = (int)blockIdx.x / kCluster;
  while (tn >= tiles_n - tm / 2) {
    tn -= tiles_n - tm / 2;
    ++tm;
  }
  tn += tm / 2;
  constexpr int kShare = 128 / kCluster;  // columns of a half that a rank owns
  constexpr int kPitch = 2 * kShare + 1;  // rows of the sums in the staging area
  const int nseg = (kb_total + kSegBlocks - 1) / kSegBlocks;
  const int rounds = (nseg + kCluster - 1) / kCluster;
  // f(its place in H, its sum in the staging area) for this epilogue thread's part of the rank's
  // columns, row by row
  auto for_own = [&](auto f) {
    for (int x = (int)threadIdx.x - 64; x < kBM * 2 * kShare; x += 256) {
      const int r = x / (2 * kShare), c = x - r * (2 * kShare);
      const int64_t hr = (int64_t)tm * kBM + r;
      const int64_t hc = (int64_t)tn * kBN + (c < kShare ? 0 : 128 - kShare) + rank * kShare + c;
      if (hr < n && hc < n) f(H + hr * ld_h + hc, staging + r * kPitch + c);
    }
  };

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&acc_full[a], 1);
      mbar_init(&acc_empty[a], 256);
    }
    mbar_init(ready, kCluster);
    mbar_init(done, kCluster);
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
  cluster.sync();  // every rank's barriers are initialised before the first remote arrival
  tc_fence_after_sync();
  const uint32_t tmem_d = warp_uniform(*tmem_slot);

  if (warp == 0) {
    uint64_t policy;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(policy));
    uint32_t s = 0, parity = 1;
    bool go = true;
    for (int seg = rank; seg < nseg && go; seg += kCluster) {
      const int kb1 = min(kb_total, (seg + 1) * kSegBlocks);
      for (int kb = seg * kSegBlocks; kb < kb1; ++kb) {
        if (!mbar_wait_warp(&empty[s], parity)) {
          go = false;
          break;
        }
        if (elect_one()) {
          mbar_arrive_expect_tx(&full[s], kStageBytes);
          uint8_t* a = tile_a + s * kTileABytes;
          uint8_t* b = tile_b + s * kTileBBytes;
          if (!kMN) {
            tma_load_2d(a, &amap, kb * kBK, tm * kBM, &full[s], policy);
            tma_load_2d(b, &bmap, kb * kBK, tn * kBN, &full[s], policy);
          } else if (grouped) {
            tma_load_3d(a, &amap, 0, kb * kBK, tm * (kBM / 64), &full[s], policy);
            tma_load_3d(b, &bmap, 0, kb * kBK, tn * (kBN / 64), &full[s], policy);
          } else {
#pragma unroll
            for (int j = 0; j < kBM / 64; ++j)
              tma_load_2d(a + j * kBoxBytes, &amap, tm * kBM + 64 * j, kb * kBK, &full[s], policy);
#pragma unroll
            for (int j = 0; j < kBN / 64; ++j)
              tma_load_2d(b + j * kBoxBytes, &bmap, tn * kBN + 64 * j, kb * kBK, &full[s], policy);
          }
        }
        __syncwarp();
        if (++s == kStages) {
          s = 0;
          parity ^= 1u;
        }
      }
    }
    if (!go && lane == 0) fail_cluster<kCluster>(failed);
    __syncwarp();
    ring_drain(full, kStages, s, parity);
  } else if (warp == 1) {
    uint32_t s = 0, parity = 0, i = 0;
    bool ok = true;
    for (int seg = rank; seg < nseg && ok; seg += kCluster, ++i) {
      const uint32_t acc = i & 1u, d = tmem_d + acc * kBN;
      // the accumulator's previous segment must have been read out of TMEM
      if (i >= 2 && !mbar_wait_warp(&acc_empty[acc], ((i >> 1) - 1) & 1u)) {
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
          if (kMN) {
            // MN-major: 16 K rows are two 1024-byte swizzle atoms further
            const uint64_t ad = smem_desc_mn_sw128(a, kBoxBytes), bd = smem_desc_mn_sw128(b, kBoxBytes);
#pragma unroll
            for (int kk = 0; kk < kBK / 16; ++kk)
              umma_bf16(d, ad + 128 * kk, bd + 128 * kk, idesc_bf16_f32_mn(kBM, kBN), (uint32_t)(kb > kb0 || kk > 0));
          } else {
            umma_bf16_block(d, smem_desc_k_sw128(a), smem_desc_k_sw128(b), idesc_bf16_f32(kBM, kBN), 4,
                            (uint32_t)(kb > kb0));
          }
          umma_commit(smem_addr(&empty[s]));
          // fires once every MMA issued above has completed
          if (kb + 1 == kb1) umma_commit(smem_addr(&acc_full[acc]));
        }
        __syncwarp();
        if (++s == kStages) {
          s = 0;
          parity ^= 1u;
        }
      }
    }
    if (!ok && lane == 0) fail_cluster<kCluster>(failed);
    __syncwarp();
    umma_drain(mma_done);
  } else {
    // epilogue: as a source, this thread's row and 64 columns of a half; as an owner, the warp's
    // columns of the rank's share, rows 4 lane .. + 3
    constexpr int kOwn = kShare / 8;            // of them, a warp's
    const int e = warp - 2, tid = (int)threadIdx.x - 64;
    const uint32_t quarter = (uint32_t)(warp & 3);
    const uint32_t lane_base = (quarter * 32u) << 16;
    const int row = (int)quarter * 32 + lane, ccol = 64 * (e >> 2);
    float4 sum[2][kOwn];
#pragma unroll
    for (int hf = 0; hf < 2; ++hf)
#pragma unroll
      for (int k = 0; k < kOwn; ++k) sum[hf][k] = make_float4(0.f, 0.f, 0.f, 0.f);
    uint32_t turn = 0;  // half rounds
    // a wait that ran out ends the waiting, not the rounds: every thread reaches every barrier
    bool ok = true;
    for (int i = 0; i < rounds; ++i) {
      const uint32_t acc = (uint32_t)i & 1u;
      const bool have = i * kCluster + rank < nseg;
      if (have && ok) ok = mbar_wait_acc(&acc_full[acc], (uint32_t)(i >> 1) & 1u);
      tc_fence_after_sync();
#pragma unroll
      for (int hf = 0; hf < 2; ++hf, ++turn) {
        // the staging area's previous half has been read by every rank
        if (turn >= 1 && ok) ok = wait_cluster(done, (turn - 1) & 1u);
        if (have) {
#pragma unroll
          for (int c = 0; c < 64; c += 32) {
            uint32_t p[32];
            tmem_ld_32x32b_x32(tmem_d + acc * kBN + lane_base + 128 * hf + ccol + (uint32_t)c, p);
            tmem_ld_wait();
#pragma unroll
            for (int k = 0; k < 32; ++k) staging[(ccol + c + k) * kBM + row] = __uint_as_float(p[k]);
          }
          if (hf == 1) {
            tc_fence_before_sync();
            mbar_arrive(&acc_empty[acc]);
          }
        }
        epilogue_sync();
        if (tid < kCluster) arrive_remote(ready, (uint32_t)tid);
        if (ok) ok = wait_cluster(ready, turn & 1u);
#pragma unroll
        for (int k = 0; k < kOwn; ++k) {
          const int c = rank * kShare + e + 8 * k;
          float4 v[kCluster];
#pragma unroll
          for (int q = 0; q < kCluster; ++q)
            if (i * kCluster + q < nseg) v[q] = ld_cluster_v4(mapa(smem_addr(staging + c * kBM + 4 * lane), (uint32_t)q));
#pragma unroll
          for (int q = 0; q < kCluster; ++q) {
            if (i * kCluster + q >= nseg) break;
            float4& s = sum[hf][k];
            if (i == 0 && q == 0)
              s = v[0];
            else
              s = make_float4(__fadd_rn(s.x, v[q].x), __fadd_rn(s.y, v[q].y), __fadd_rn(s.z, v[q].z),
                              __fadd_rn(s.w, v[q].w));
          }
        }
        epilogue_sync();
        if (tid < kCluster) arrive_remote(done, (uint32_t)tid);
      }
    }
    // the sums go into H through the staging area, rows of the rank's 2 kShare columns
    if (ok) ok = wait_cluster(done, (turn - 1) & 1u);
    if (!ok) fail_cluster<kCluster>(failed);
    epilogue_sync();
#pragma unroll
    for (int hf = 0; hf < 2; ++hf)
#pragma unroll
      for (int k = 0; k < kOwn; ++k) {
        float* dst = staging + 4 * lane * kPitch + hf * kShare + e + 8 * k;
        dst[0] = sum[hf][k].x;
        dst[kPitch] = sum[hf][k].y;
        dst[2 * kPitch] = sum[hf][k].z;
        dst[3 * kPitch] = sum[hf][k].w;
      }
    epilogue_sync();
    // H is read before the cluster's barrier and written after it (8192 x 768: 25.2 us, 27.0 with both after)
    for_own([&](float* p, float* s) { *s = *p + *s; });
  }
  tc_fence_before_sync();
  cluster.sync();
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc(tmem_d, 2 * kBN);
  }
  if (warp >= 2) {
    const bool bad = *failed != 0;
    if (bad && threadIdx.x == 64) atomicOr(&g_hessian_cluster_flags, kErrMbarTimeout);
    for_own([&](float* p, float* s) { *p = bad ? __int_as_float(0x7FC00000) : *s; });
  }
}

template <int kCluster, bool kMN>
cudaError_t launch(const CUtensorMap& amap, const CUtensorMap& bmap, int kb_total, int tiles, int tiles_n, float* H,
                   int64_t n, int64_t ld_h, int grouped, cudaStream_t stream) {
  auto kernel = hessian_cluster_kernel<kCluster, kMN>;
  cudaError_t err = ensure_dynamic_smem(reinterpret_cast<const void*>(kernel), (int)kSmemBytes);
  if (err != cudaSuccess) return err;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(tiles * kCluster), 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = kSmemBytes;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kCluster;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  err = cudaLaunchKernelEx(&cfg, kernel, amap, bmap, kb_total, tiles_n, H, n, ld_h, grouped);
  return err != cudaSuccess ? err : cudaGetLastError();
}

}  // namespace

// The split costs about what 2048 tokens do (the cluster's launch and the rounds' hand-over: 4096 or
// 6000 tokens at n = 1024 take 39.0 or 47.9 us with or without it), so it starts at four segments;
// at two where H's rows are not 16-byte aligned, which gemm_kernel's epilogue updates float by
// float, a thread a row, and this one's row by row (5000 x 1001: 98 -> 66 us).
int hessian_cluster_size(int64_t tokens, int64_t n, bool h_aligned, int sm_count) {
  const int64_t rows = (n + kBM - 1) / kBM, cols = (n + kBN - 1) / kBN;
  const int64_t segments = (tokens + kSegBlocks * kBK - 1) / (kSegBlocks * kBK);
  if (rows > 64 || (h_aligned && segments < 4)) return 1;
  int64_t tiles = 0;
  for (int64_t tm = 0; tm < rows; ++tm) tiles += cols - tm / 2;
  int size = 1;
  while (size < 8 && 2 * size <= segments && 2 * size * tiles <= sm_count) size *= 2;
  return size;
}

cudaError_t launch_hessian_cluster(int size, const CUtensorMap& amap, const CUtensorMap& bmap, bool mn_major,
                                   bool grouped, int64_t tokens, int64_t n, float* H, int64_t ld_h,
                                   cudaStream_t stream) {
  const int rows = (int)((n + kBM - 1) / kBM), cols = (int)((n + kBN - 1) / kBN);
  int tiles = 0;
  for (int tm = 0; tm < rows; ++tm) tiles += cols - tm / 2;
  const int kb = (int)((tokens + kBK - 1) / kBK), g = grouped ? 1 : 0;
  switch (size) {
    case 2: return mn_major ? launch<2, true>(amap, bmap, kb, tiles, cols, H, n, ld_h, g, stream)
                            : launch<2, false>(amap, bmap, kb, tiles, cols, H, n, ld_h, g, stream);
    case 4: return mn_major ? launch<4, true>(amap, bmap, kb, tiles, cols, H, n, ld_h, g, stream)
                            : launch<4, false>(amap, bmap, kb, tiles, cols, H, n, ld_h, g, stream);
    default: return mn_major ? launch<8, true>(amap, bmap, kb, tiles, cols, H, n, ld_h, g, stream)
                             : launch<8, false>(amap, bmap, kb, tiles, cols, H, n, ld_h, g, stream);
  }
}

cudaError_t read_hessian_cluster_device_error(uint32_t* flags) {
  uint32_t v = 0;
  cudaError_t err = cudaMemcpyFromSymbol(&v, g_hessian_cluster_flags, sizeof v);
  if (err != cudaSuccess) return err;
  *flags = v;
  if (v) {
    const uint32_t zero = 0;
    err = cudaMemcpyToSymbol(g_hessian_cluster_flags, &zero, sizeof zero);
  }
  return err;
}

}  // namespace hscale
