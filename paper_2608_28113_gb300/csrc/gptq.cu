// gptq.cu -- GPTQ with H-Scale as the local quantizer (Algorithm 3) on sm_103a.
//
//   (the damped inverse-Cholesky factor U is formed in factor.cu)
//   gptq_panel_kernel a panel of whole blocks, up to 512 columns: for each block of the running
//                     fp32 weights the RTN code (Eq. 7), the exact H-Scale search over the window
//                     (Algorithm 1, exact E2M1 decisions, the tie rule of the search), the codes
//                     and packed nibbles, the propagated errors E = (W - W_hat) / U_jj, and
//                     W -= E U for the panel's columns right of the block
//   block_kernel      the same for one block wider than that, without the propagation
//   update            W[:, i+P:] -= E U[i:i+P, i+P:] for the columns right of a panel, with
//                     fp32-level accuracy on the tensor cores (update.cu)
#include <algorithm>

#include <cuda_bf16.h>

#include "chained_launch.h"
#include "hscale_device.cuh"
#include "hscale_internal.h"
#include "search.cuh"
#include "split3.cuh"
#include "tcgen05.cuh"
#include "tma.cuh"

namespace hscale {
namespace {

// ---------------------------------------------------------------- block quantizer
// sum_j h_j (a_j - s' q_j)^2 with exact E2M1 decisions, one rounding per residual and a
// fixed pairwise sum (relative error <= 8 * 2^-24)
__device__ float exact_group_score(const float (&a)[16], const float (&hj)[16], uint32_t c, float sgk) {
  float t[16];
#pragma unroll
  for (int j = 0; j < 16; ++j) t[j] = exact_term(a[j], hj[j], c, sgk);
#pragma unroll
  for (int step = 1; step < 16; step <<= 1)
#pragma unroll
    for (int j = 0; j + step < 16; j += 2 * step) t[j] = __fadd_rn(t[j], t[j + step]);
  return t[0];
}

// Four lanes (a quad) per group: each scores every fourth candidate of the window with exact
// decisions, the quad keeps the best under the search's tie rule (a total order, so every
// lane ends with the same code), and each lane writes the nibbles of four of the group's
// elements and their scaled errors E = (w - w_hat) / U_jj, split in three bf16 parts, into the
// update's operand [m, 3 B] (update.cu), four bf16 (8 bytes) per part.
__global__ void __launch_bounds__(128) block_kernel(const float* __restrict__ W, int64_t m, int64_t n, int64_t col0,
                                                    int B, const float* __restrict__ h, const float* __restrict__ U,
                                                    const float* __restrict__ global_scale, int down, int up,
                                                    uint8_t* __restrict__ codes, uint2* __restrict__ packed,
                                                    uint16_t* __restrict__ A) {
  const int gpb = B / 16;
  const int64_t total = m * gpb * 4;  // lanes
  const int q = threadIdx.x & 3;
  const ScaleDomain d = make_scale_domain(*global_scale);
  const float inv6 = rtn_inv6_raw(d.sgk);
  // block-uniform trip count: every lane of a warp reaches the shuffles together
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < total; base += (int64_t)gridDim.x * blockDim.x) {
    const int64_t lane_id = base + threadIdx.x;
    const bool active = lane_id < total;
    const int64_t g = active ? lane_id >> 2 : 0;
    const int64_t r = g / gpb;
    const int i = (int)(g - r * gpb);
    const int64_t col = col0 + 16 * i;
    float w[16], a[16], hj[16];
    float amax = 0.0f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float4 v = reinterpret_cast<const float4*>(W + r * n + col)[k];
      const float4 hv = reinterpret_cast<const float4*>(h + col)[k];
      w[4 * k] = v.x; w[4 * k + 1] = v.y; w[4 * k + 2] = v.z; w[4 * k + 3] = v.w;
      hj[4 * k] = hv.x; hj[4 * k + 1] = hv.y; hj[4 * k + 2] = hv.z; hj[4 * k + 3] = hv.w;
    }
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      a[j] = __fmul_rn(fabsf(w[j]), d.pw);
      amax = fmaxf(amax, a[j]);
    }
    const int c0 = (int)rtn_code(amax, d.sgk, inv6);
    const int lo = max(1, c0 - down), hi = min((int)kE4M3MaxCode, c0 + up);
    float be = 0.0f;
    int bc = -1;
    for (int c = lo + q; c <= hi; c += 4) {
      const float e = exact_group_score(a, hj, (uint32_t)c, d.sgk);
      if (bc < 0 || better(e, c, be, bc, c0)) {
        be = e;
        bc = c;
      }
    }
#pragma unroll
    for (int off = 1; off < 4; off <<= 1) {
      const float oe = __shfl_xor_sync(0xFFFFFFFFu, be, off);
      const int oc = __shfl_xor_sync(0xFFFFFFFFu, bc, off);
      if (oc >= 0 && (bc < 0 || better(oe, oc, be, bc, c0))) {
        be = oe;
        bc = oc;
      }
    }
    const float l = e4m3_mag((uint32_t)bc);
    const float inv = inv_raw_of(__fmul_rn(l, d.sgk));
    // this lane's elements 4q..4q+3 (read again as one vector: no dynamic register index)
    const float4 wq = reinterpret_cast<const float4*>(W + r * n + col)[q];
    const float wv[4] = {wq.x, wq.y, wq.z, wq.w};
    uint32_t part = 0u;  // this lane's four nibbles in their place in the group's 32-bit word
    float e4[4];         // E of this lane's four elements
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int j = 4 * q + t;
      const float av = __fmul_rn(fabsf(wv[t]), d.pw);
      const uint32_t k = e2m1_code(av, inv, l, d.sgk);
      const uint32_t neg = signbit(wv[t]) ? 1u : 0u;
      part |= ((neg << 3) | k) << (4 * (j & 7));
      float what = __fmul_rn(d.sg, __fmul_rn(e2m1_from_raw(k << 22), l));  // s_g (l q), l q exact
      if (neg) what = -what;
      e4[t] = __fdiv_rn(__fsub_rn(wv[t], what), U[(col + j) * n + col + j]);
    }
    if (active) store_split3x4(A + r * 3 * (int64_t)B + 16 * i + 4 * q, B, e4);
    const uint32_t word = part | __shfl_xor_sync(0xFFFFFFFFu, part, 1);  // lanes 0-1: word 0, 2-3: word 1
    const uint32_t other = __shfl_xor_sync(0xFFFFFFFFu, word, 2);
    if (active && q == 0) {
      codes[r * (n / 16) + col / 16] = (uint8_t)bc;
      packed[r * (n / 16) + col / 16] = make_uint2(word, other);
    }
  }
}

// ---------------------------------------------------------------- the panel
// Algorithm 3 on one panel of `outer` columns (blocks of B; outer a multiple of B, at most
// kPanelCols) for kRows rows a CTA, blocks and their propagation inside the panel included.
// Rows are independent of each other, so a CTA needs nothing from the others: its strip of the
// running weights stays in shared memory from the first block to the last, and only the codes,
// the nibbles and the split errors (the A operand of the update of the columns right of the
// panel) leave it.  So the blocks follow one another at the pace of shared memory and barriers,
// not of kernel launches, and the weights outside the panel are read and written once per panel
// and not once per block.  Per block:
//   * quantize: kLanes lanes per 16-element group, with the search kernels' method: the fast
//     scores of the candidates (split over the lanes), the margin test, and the exact rescoring
//     by the whole warp for the groups it cannot clear; so the codes are those of exact
//     decisions under the search's tie rule.  Then each lane takes 16 / kLanes elements: exact
//     nibbles, E = (w - w_hat) / U_jj, and E's three bf16 parts (split3) into shared memory (the
//     MMA's operand, 128-byte swizzled) and into Es;
//   * propagate inside the panel: W[:, j] -= sum_k E[:, k] U[k, j] for the panel's columns j right
//     of the block, with fp32-level accuracy (the six products of update.cu), by tcgen05 MMAs
//     with U's columns as M (128 at a time, loaded by TMA through six 16 KB slots) and the
//     strip's rows as N.  One MMA takes all of E's parts that go with a part of U, U1 [E1 | E2 | E3],
//     U2 [E1 | E2], U3 E1, half as many as one for each product, into three accumulators side by
//     side in tensor memory, which all warps add up (smallest first) and subtract from the strip.
// What bounds it: the quantizer's arithmetic and latency, then the TMA loads of U's parts
// (96 KB per 128 columns and block of 128).  kRows is 32, or 16 when that still leaves no more
// CTAs than SMs: half the work per CTA, and twice the lanes per group.
// One GB300, 4096 x 4096, blocks of 128: 53 K cycles or 28 us a panel by clock stamps (set-up 5,
// quantizing 4 x 6.5, propagating 6.6 + 4.4 + 2.3, adding to the strip 3 x 0.8, write-out 1.4, barriers
// and what lies between the stamps 5), 30 us alone under a profiler; the four blocks took about 130
// us with a quantizer and two updates launched for each; the whole call 1050 -> 628 us, 567 since its launches overlap, 554 with update.cu's last tiles
// halved.
constexpr int kPanelCols = 512;
constexpr int kPanelThreads = 512;
constexpr int kSlots = 6;
constexpr uint32_t kSlotBytes = 128 * 64 * 2;  // 128 columns of U, 64 of K
constexpr int kMaxLocalBlock = kPanelCols / 2; // a larger block leaves nothing to update in the panel

__device__ uint32_t g_gptq_flags = 0;

__device__ __forceinline__ void tmem_ld_rows(uint32_t src, uint32_t (&r)[32]) { tmem_ld_32x32b_x32(src, r); }
__device__ __forceinline__ void tmem_ld_rows(uint32_t src, uint32_t (&r)[16]) { tmem_ld_32x32b_x16(src, r); }

struct PanelArgs {
  const float* W;  // running weights [m, n], written by the kernels before this one
  const float* h;
  const float* U;
  const float* global_scale;
  uint8_t* codes;
  uint2* packed;
  uint16_t* Es;    // [m, 3 outer]
  int64_t m, n, col0;
  int outer, B, down, up;
};

template <int kRows>
struct PanelSmem {
  static constexpr int kPitch = kPanelCols + 4;
  static constexpr uint32_t kE = kSlots * kSlotBytes;                               // split errors
  static constexpr uint32_t kW = kE + 3 * (kMaxLocalBlock / 64) * kRows * 128;      // the strip
  static constexpr uint32_t kH = kW + kRows * kPitch * 4;                           // h, then diag(U)
  static constexpr uint32_t kTab = kH + 2 * kPanelCols * 4;                         // candidate constants
  static constexpr uint32_t kPacked = kTab + 128 * 16;
  static constexpr uint32_t kCodes = kPacked + kRows * kPanelCols / 2;
  static constexpr uint32_t kBar = kCodes + kRows * kPanelCols / 16;
  static constexpr uint32_t kBytes = kBar + 256 + 1024 /* alignment */;
};

template <int kRows>
__global__ void __launch_bounds__(kPanelThreads, 1)
gptq_panel_kernel(const __grid_constant__ CUtensorMap umap, const PanelArgs args) {
  using L = PanelSmem<kRows>;
  constexpr int kLanes = 64 / kRows;   // lanes per group
  constexpr int kEl = 16 / kLanes;     // a lane's elements
  extern __shared__ __align__(16) uint8_t dynamic_smem[];
  uint8_t* smem = dynamic_smem + ((1024u - (smem_addr(dynamic_smem) & 1023u)) & 1023u);
  float* W = reinterpret_cast<float*>(smem + L::kW);
  float* hs = reinterpret_cast<float*>(smem + L::kH);
  float* ud = hs + kPanelCols;
  float4* tab = reinterpret_cast<float4*>(smem + L::kTab);
  uint8_t* packed_s = smem + L::kPacked;
  uint8_t* codes_s = smem + L::kCodes;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + L::kBar);
  uint64_t* empty = full + kSlots;
  uint64_t* acc_full = empty + kSlots;  // four column tiles
  uint64_t* mma_done = acc_full + 4;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mma_done + 1);
  volatile uint32_t* failed = tmem_slot + 1;
  const int tid = threadIdx.x, lane = tid & 31, warp = (int)warp_uniform(threadIdx.x >> 5);
  const int B = args.B, outer = args.outer, gpb = B / 16, chunks = (B + 63) / 64;
  const int64_t row0 = (int64_t)blockIdx.x * kRows;
  // tensor memory: three accumulators of kRows columns for each of up to four column tiles
  constexpr uint32_t kCols = 16 * kRows;

  if (tid == 0) {
    for (int i = 0; i < kSlots; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < 4; ++i) mbar_init(&acc_full[i], 1);
    mbar_init(mma_done, 1);
    *failed = 0u;
    mbar_fence_init();
    prefetch_tensormap(&umap);
  }
  if (warp == 1) {
    tmem_alloc(smem_addr(tmem_slot), kCols);
    tmem_relinquish();
  }
  // the call's inputs are complete (the call's first kernel is launched in stream order); the
  // running weights and U's parts come from the kernels before this one
  pdl_launch_dependents();
  const ScaleDomain d = make_scale_domain(*args.global_scale);
  const float inv6 = rtn_inv6_raw(d.sgk);
  const float2 b6 = anchor_brackets(d.sgk, 6.0f);
  if (tid < 128) tab[tid] = candidate_constants((uint32_t)tid, d.sgk);
  for (int c = tid; c < outer; c += kPanelThreads) {
    hs[c] = args.h[args.col0 + c];
    ud[c] = args.U[(args.col0 + c) * args.n + args.col0 + c];
  }
  pdl_wait_primary();
  {
    const int quads = outer / 4;
    for (int e = tid; e < kRows * quads; e += kPanelThreads) {
      const int r = e / quads, c = (e - r * quads) * 4;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (row0 + r < args.m) v = *reinterpret_cast<const float4*>(args.W + (row0 + r) * args.n + args.col0 + c);
      *reinterpret_cast<float4*>(W + r * L::kPitch + c) = v;
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_d = warp_uniform(*tmem_slot);

  // U's loads of one block, numbered over its column tiles, parts (1, 2, 3) and chunks of K; load
  // l goes to slot l % kSlots, and warp 2 + slot issues it.  load_par: the parity of the slot's
  // next use (loader); bit s of use_par: that of slot s's next use (warp 0, the MMAs).
  const int slot = warp - 2;
  const bool loader = slot >= 0 && slot < kSlots;
  uint32_t load_par = 0, use_par = 0;
  auto load = [&](int b, int l) {
    const int u = l / (3 * chunks), rest = l - u * 3 * chunks, part = rest / chunks;
    const int c = rest - part * chunks;
    if (elect_one()) {
      mbar_arrive_expect_tx(&full[slot], kSlotBytes);
      tma_load_3d(smem + slot * kSlotBytes, &umap, b * B + 64 * c, part, (b + 1) * B + 128 * u, &full[slot]);
    }
    __syncwarp();
    load_par ^= 1u;
  };

  const int nblk = outer / B;
  for (int b = 0; b < nblk; ++b) {
    const int cb = b * B, rest = outer - cb - B;
    const int tiles = (rest + 127) / 128, loads = tiles * 3 * chunks;
    if (loader && slot < loads) load(b, slot);  // every slot is free here

    // ---- quantize the block
    for (int base = 0; base < kRows * gpb; base += kPanelThreads / kLanes) {
      const int gi = base + tid / kLanes, q = tid % kLanes;
      if (gi >= kRows * gpb) break;  // whole warps: kRows * gpb is a multiple of a warp's groups
      const int r = gi % kRows, i = gi / kRows, cl = cb + 16 * i;
      const float* wrow = W + r * L::kPitch + cl;
      Group G;
      float2 hv2[8];
      float amax = 0.0f;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float4 v = *reinterpret_cast<const float4*>(wrow + 4 * k);
        const float4 hv = *reinterpret_cast<const float4*>(hs + cl + 4 * k);
        G.a[2 * k] = make_float2(__fmul_rn(v.x, d.pw), __fmul_rn(v.y, d.pw));
        G.a[2 * k + 1] = make_float2(__fmul_rn(v.z, d.pw), __fmul_rn(v.w, d.pw));
        hv2[2 * k] = make_float2(hv.x, hv.y);
        hv2[2 * k + 1] = make_float2(hv.z, hv.w);
        amax = fmaxf(amax, fmaxf(fmaxf(fabsf(G.a[2 * k].x), fabsf(G.a[2 * k].y)),
                                 fmaxf(fabsf(G.a[2 * k + 1].x), fabsf(G.a[2 * k + 1].y))));
      }
      const int c0 = (int)anchored_code_fast(amax, d.sgk, b6.x, b6.y, inv6, 3.0f);
      const int lo = max(1, c0 - args.down), hi = min((int)kE4M3MaxCode, c0 + args.up);
      float e1 = kInf, e2 = kInf;
      int best = c0;
      for (int c = lo + q; c <= hi; c += 2 * kLanes) {
        const int cc = c + kLanes;
        const float ea = fast_score(G, hv2, tab[c]);
        const float eb = fast_score(G, hv2, tab[min(cc, (int)kE4M3MaxCode)]);
        keep_best(ea, c, e1, e2, best);
        keep_best(cc <= hi ? eb : kInf, cc, e1, e2, best);
      }
#pragma unroll
      for (int off = 1; off < kLanes; off <<= 1) {
        const float o1 = __shfl_xor_sync(0xFFFFFFFFu, e1, off), o2 = __shfl_xor_sync(0xFFFFFFFFu, e2, off);
        const int ob = __shfl_xor_sync(0xFFFFFFFFu, best, off);
        best = o1 < e1 ? ob : best;
        e2 = fminf(fminf(e2, o2), fmaxf(e1, o1));  // a tie with the best makes e2 = e1
        e1 = fminf(e1, o1);
      }
      // a group of zeros scores zero under every code: the tie rule keeps the initial one (also the
      // rows past m, which would otherwise all go to the exact rescoring)
      if (amax == 0.0f) best = c0;
      bool ambiguous = false;
      if (hi > lo && amax != 0.0f) {
        float2 s2 = make_float2(0.f, 0.f);
#pragma unroll
        for (int k = 0; k < 8; ++k) s2 = __fadd2_rn(s2, hv2[k]);
        ambiguous = !fast_winner_clear(e1, e2, energy_bound(__fadd_rn(s2.x, s2.y), amax));
        if (ambiguous) ambiguous = !fast_winner_certain(e1, e2, group_energy(G, hv2));
      }
      unsigned amb = __ballot_sync(0xFFFFFFFFu, ambiguous && q == 0);
      while (amb) {
        const int owner = __ffs(amb) - 1;
        amb &= amb - 1;
        const int go = __shfl_sync(0xFFFFFFFFu, gi, owner);
        const int c0o = __shfl_sync(0xFFFFFFFFu, c0, owner);
        const int j = cb + 16 * (go / kRows) + (lane & 15);
        const float a_k = __fmul_rn(fabsf(W[(go % kRows) * L::kPitch + j]), d.pw);
        const int bc = warp_exact_codes(a_k, hs[j], c0o, max(1, c0o - args.down),
                                        min((int)kE4M3MaxCode, c0o + args.up), d.sgk);
        if (lane / kLanes == owner / kLanes) best = bc;
      }

      // this lane's elements: nibbles and errors
      const float l = e4m3_mag((uint32_t)best);
      const float inv = inv_raw_of(__fmul_rn(l, d.sgk));
      const int j0 = kEl * q;
      uint32_t nibbles = 0u;
      uint16_t parts[3][kEl];
#pragma unroll
      for (int t = 0; t < kEl; ++t) {
        const float wv = wrow[j0 + t];
        const uint32_t k = e2m1_code(__fmul_rn(fabsf(wv), d.pw), inv, l, d.sgk);
        const uint32_t neg = signbit(wv) ? 1u : 0u;
        nibbles |= ((neg << 3) | k) << (4 * t);
        float what = __fmul_rn(d.sg, __fmul_rn(e2m1_from_raw(k << 22), l));  // s_g (l q), l q exact
        if (neg) what = -what;
        uint16_t pp[3];
        split3(__fdiv_rn(__fsub_rn(wv, what), ud[cl + j0 + t]), pp);
        parts[0][t] = pp[0];
        parts[1][t] = pp[1];
        parts[2][t] = pp[2];
      }
      const int kb = 16 * i + j0;  // the first element within the block
#pragma unroll
      for (int part = 0; part < 3; ++part) {
        uint32_t v[kEl / 2];
#pragma unroll
        for (int t = 0; t < kEl / 2; ++t)
          v[t] = (uint32_t)parts[part][2 * t] | ((uint32_t)parts[part][2 * t + 1] << 16);
        uint16_t* es = args.Es + ((row0 + r) * 3 + part) * outer + cl + j0;
        uint8_t* st = smem + L::kE + (((kb / 64) * 3 + part) * kRows + r) * 128 +
                      ((((kb & 63) >> 3) ^ (r & 7)) << 4) + (kb & 7) * 2;
        if (kEl == 8) {
          const uint4 v4 = make_uint4(v[0], v[1], v[kEl / 2 - 2], v[kEl / 2 - 1]);
          if (tiles > 0) *reinterpret_cast<uint4*>(st) = v4;
          if (row0 + r < args.m) *reinterpret_cast<uint4*>(es) = v4;
        } else {
          if (tiles > 0) *reinterpret_cast<uint2*>(st) = make_uint2(v[0], v[1]);
          if (row0 + r < args.m) *reinterpret_cast<uint2*>(es) = make_uint2(v[0], v[1]);
        }
      }
      if (kEl == 8)
        *reinterpret_cast<uint32_t*>(packed_s + r * (outer / 2) + (cl + j0) / 2) = nibbles;
      else
        *reinterpret_cast<uint16_t*>(packed_s + r * (outer / 2) + (cl + j0) / 2) = (uint16_t)nibbles;
      if (q == 0) codes_s[r * (outer / 16) + cl / 16] = (uint8_t)best;
    }
    if (tiles == 0) break;  // the last block of the panel
    fence_proxy_async_smem();
    __syncthreads();

    // ---- propagate inside the panel
    if (warp == 0) {
      tc_fence_after_sync();
      bool ok = true;
      int s = 0;
      for (int t = 0; t < tiles && ok; ++t) {
        const uint32_t dt = tmem_d + (uint32_t)t * (3 * kRows);
#pragma unroll
        for (int up = 0; up < 3; ++up) {  // U's parts 1, 2, 3
          if (!ok) break;
          for (int c = 0; c < chunks; ++c) {
            if (!mbar_wait_warp(&full[s], (use_par >> s) & 1u)) {
              ok = false;
              break;
            }
            use_par ^= 1u << s;
            tc_fence_after_sync();
            if (elect_one()) {
              // E's parts 1 .. 3 - up, rows of one operand
              umma_bf16_block(dt, smem_desc_k_sw128(smem_addr(smem + s * kSlotBytes)),
                              smem_desc_k_sw128(smem_addr(smem + L::kE + c * 3 * kRows * 128)),
                              idesc_bf16_f32(128, (3 - up) * kRows), min(4, (B - 64 * c + 15) / 16),
                              (uint32_t)(up > 0 || c > 0));
              umma_commit(smem_addr(&empty[s]));
              if (up == 2 && c + 1 == chunks) umma_commit(smem_addr(&acc_full[t]));
            }
            __syncwarp();
            s = s + 1 == kSlots ? 0 : s + 1;
          }
        }
      }
      if (!ok) *failed = 1u;
    } else if (loader) {
      for (int l = slot + kSlots; l < loads; l += kSlots) {
        if (!mbar_wait_warp(&empty[slot], load_par ^ 1u)) {
          *failed = 1u;
          break;
        }
        load(b, l);
      }
    }
    const int t = warp >> 2;
    if (t < tiles) {
      const bool done = mbar_wait_acc(&acc_full[t], (uint32_t)b & 1u);
      if (!done) *failed = 1u;
      tc_fence_after_sync();
      uint32_t p[kRows];
      const uint32_t src = tmem_d + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)t * (3 * kRows);
      tmem_ld_rows(src + 2 * kRows, p);  // with E3, then E2, then E1
#pragma unroll
      for (int g = 1; g >= 0; --g) {
        uint32_t q[kRows];
        tmem_ld_rows(src + g * kRows, q);
        tmem_ld_wait();
#pragma unroll
        for (int r = 0; r < kRows; ++r) p[r] = __float_as_uint(__fadd_rn(__uint_as_float(p[r]), __uint_as_float(q[r])));
      }
      const int c = cb + B + 128 * t + 32 * (warp & 3) + lane;
      if (c < outer) {
#pragma unroll
        for (int r = 0; r < kRows; ++r) {
          float* w = W + r * L::kPitch + c;
          *w = done ? __fsub_rn(*w, __uint_as_float(p[r])) : __int_as_float(0x7FC00000);
        }
      }
    }
    tc_fence_before_sync();
    __syncthreads();
    if (*failed) break;
  }

  if (*failed) {
    // a wait ran out: the loads (each slot's last one) and MMAs in flight finish before the CTA ends
    if (loader) mbar_wait(&full[slot], load_par ^ 1u);
    if (warp == 0) umma_drain(mma_done);
  }
  __syncthreads();
  // codes and nibbles of the panel, whole rows at a time
  const int cpr = outer / 16;
  for (int e = tid; e < kRows * cpr; e += kPanelThreads) {
    const int r = e / cpr, c = e - r * cpr;
    if (row0 + r < args.m) {
      const int64_t o = (row0 + r) * (args.n / 16) + args.col0 / 16 + c;
      args.codes[o] = codes_s[e];
      args.packed[o] = *reinterpret_cast<const uint2*>(packed_s + e * 8);
    }
  }
  if (tid == 0 && *failed) atomicOr(&g_gptq_flags, kErrMbarTimeout);
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc(tmem_d, kCols);
  }
}

// The update's other operand [nn, 3 B] (row j: the three bf16 parts of U[col0 .. col0 + B, c1 + j]),
// transposed through 64 x 64 shared-memory tiles: 16-byte reads along U's rows where n allows,
// 8-byte writes (512 x 4096: 6.8 us with 32 x 32 tiles and 2-byte writes, now 6.0).
__global__ void __launch_bounds__(256) split_u_kernel(const float* __restrict__ U, int64_t n, int64_t col0, int B,
                                                      int64_t c1, uint16_t* Bt) {
  __shared__ float t[64][65];
  pdl_launch_dependents();
  pdl_wait_primary();  // the previous panel's update has read the operand
  const int64_t j0 = (int64_t)blockIdx.x * 64;
  const int k0 = blockIdx.y * 64;
  if (c1 + j0 + 63 <= col0 + k0) return;  // wholly on or below the diagonal: never used
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;  // 16 rows of 16 x 4 columns
  const int64_t col = c1 + j0 + 4 * tx;
#pragma unroll
  for (int kk = ty; kk < 64; kk += 16) {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (k0 + kk < B) {
      const float* src = U + (col0 + k0 + kk) * n + col;
      if ((n & 3) == 0 && col + 4 <= n) {  // U is 16-byte aligned, and col a multiple of 4
        v = *reinterpret_cast<const float4*>(src);
      } else {
        if (col < n) v.x = src[0];
        if (col + 1 < n) v.y = src[1];
        if (col + 2 < n) v.z = src[2];
        if (col + 3 < n) v.w = src[3];
      }
    }
    t[kk][4 * tx] = v.x;
    t[kk][4 * tx + 1] = v.y;
    t[kk][4 * tx + 2] = v.z;
    t[kk][4 * tx + 3] = v.w;
  }
  __syncthreads();
  const int k = k0 + 4 * tx;  // four of K; B is a multiple of 16
#pragma unroll
  for (int jj = ty; jj < 64; jj += 16) {
    const int64_t j = j0 + jj;
    if (c1 + j >= n || k >= B) continue;
    const float v[4] = {t[4 * tx][jj], t[4 * tx + 1][jj], t[4 * tx + 2][jj], t[4 * tx + 3][jj]};
    store_split3x4(Bt + j * 3 * B + k, B, v);
  }
}

// Eight weights a thread: one 16-byte read, two 16-byte writes (4096 x 4096: 39 us with one
// weight a thread and a 64-bit remainder each, now 20.6).
__global__ void __launch_bounds__(256) to_fp32_kernel(const uint4* __restrict__ w, int64_t vectors, uint32_t row_vectors,
                                                      const uint8_t* __restrict__ dead, float4* __restrict__ W) {
  pdl_launch_dependents();
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < vectors; e += (int64_t)gridDim.x * blockDim.x) {
    const uint4 v = ld_stream_v4(w + e);
    const uint32_t x[4] = {v.x, v.y, v.z, v.w};
    float f[8];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      f[2 * k] = bf16_lo(x[k]);
      f[2 * k + 1] = bf16_hi(x[k]);
    }
    if (dead != nullptr) {
      const uint32_t c = vectors <= UINT32_MAX ? (uint32_t)e % row_vectors : (uint32_t)(e % row_vectors);
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (dead[8 * (int64_t)c + k]) f[k] = 0.0f;
    }
    W[2 * e] = make_float4(f[0], f[1], f[2], f[3]);
    W[2 * e + 1] = make_float4(f[4], f[5], f[6], f[7]);
  }
}

}  // namespace

// ---------------------------------------------------------------- host side
namespace {

template <int kRows>
cudaError_t launch_panel(const CUtensorMap& umap, const PanelArgs& args, cudaStream_t stream) {
  const cudaError_t err =
      ensure_dynamic_smem(reinterpret_cast<const void*>(gptq_panel_kernel<kRows>), (int)PanelSmem<kRows>::kBytes);
  if (err != cudaSuccess) return err;
  return launch_chained(gptq_panel_kernel<kRows>, dim3((unsigned)((args.m + kRows - 1) / kRows)), kPanelThreads,
                        PanelSmem<kRows>::kBytes, stream, umap, args);
}

}  // namespace

// Columns quantized per update of the columns right of them: panels of whole blocks, up to 512
// columns, or one block where it is wider.
int64_t gptq_update_cols(int64_t n, int64_t block) {
  return std::min(n, block <= kPanelCols ? kPanelCols / block * block : block);
}

// Algorithm 3's block loop, panel by panel: U's rows of the panel are split (split_u_kernel), the
// panel is quantized with its blocks' propagation inside it (gptq_panel_kernel, which writes
// the split errors), and the columns right of it take their update, W -= E U, as one GEMM over
// K = the panel's columns (update.cu).  Wider blocks (over 512 columns) are a panel each, by
// block_kernel.  Everything runs on the caller's stream, each kernel scheduled
// while the one before it runs (programmatic dependent launch).
cudaError_t launch_gptq_hscale(const void* w, int64_t m, int64_t n, const float* U, const float* h,
                               const float* global_scale, const uint8_t* dead, int block, int64_t cols, int down,
                               int up, uint8_t* codes, uint8_t* packed, float* Wf, uint16_t* Es, uint16_t* Us,
                               cudaStream_t stream) {
  DeviceInfo info;
  cudaError_t err = current_device_info(&info);
  if (err != cudaSuccess) return err;
  EncodeTiledFn encode = nullptr;
  if ((err = encode_tiled_fn(&encode)) != cudaSuccess) return err;
  const unsigned cvt_blocks = (unsigned)std::min<int64_t>((m * n / 8 + 255) / 256, (int64_t)info.sm_count * 8);
  to_fp32_kernel<<<cvt_blocks, 256, 0, stream>>>(static_cast<const uint4*>(w), m * n / 8, (uint32_t)(n / 8), dead,
                                                 reinterpret_cast<float4*>(Wf));
  if ((err = cudaGetLastError()) != cudaSuccess) return err;
  for (int64_t c0 = 0; c0 < n; c0 += cols) {
    const int64_t K = std::min(cols, n - c0), c1 = c0 + K;
    const bool wide = block > kPanelCols;
    // U's columns from the panel's second block on (from the next panel on for a wide block)
    const int64_t first = wide ? c1 : c0;
    if (c0 + block < n) {
      if ((err = launch_chained(split_u_kernel, dim3((unsigned)((n - first + 63) / 64), (unsigned)((K + 63) / 64)), 256, 0,
                                stream, U, n, c0, (int)K, first, Us)) != cudaSuccess)
        return err;
    }
    if (wide) {
      const int64_t groups = m * (K / 16);
      const unsigned qb = (unsigned)std::min<int64_t>((groups * 4 + 127) / 128, (int64_t)info.sm_count * 16);
      block_kernel<<<qb, 128, 0, stream>>>(Wf, m, n, c0, (int)K, h, U, global_scale, down, up, codes,
                                           reinterpret_cast<uint2*>(packed), Es);
      if ((err = cudaGetLastError()) != cudaSuccess) return err;
    } else {
      CUtensorMap umap;
      const cuuint64_t dims[3] = {(cuuint64_t)K, 3, (cuuint64_t)(n - c0)};
      const cuuint64_t strides[2] = {(cuuint64_t)K * 2, (cuuint64_t)K * 6};
      const cuuint32_t box[3] = {64, 1, 128};
      const cuuint32_t estr[3] = {1, 1, 1};
      if (encode(&umap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, Us, dims, strides, box, estr,
                 CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                 CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
      const PanelArgs args = {Wf, h, U, global_scale, codes, reinterpret_cast<uint2*>(packed), Es, m, n, c0,
                              (int)K, block, down, up};
      err = m <= 16 * (int64_t)info.sm_count ? launch_panel<16>(umap, args, stream)
                                             : launch_panel<32>(umap, args, stream);
      if (err != cudaSuccess) return err;
    }
    if (c1 < n && (err = launch_split_update(Es, Us + (wide ? 0 : K * 3 * K), m, n - c1, K, Wf + c1, n, stream)) !=
                      cudaSuccess)
      return err;
  }
  return cudaSuccess;
}

cudaError_t read_gptq_device_error(uint32_t* flags) {
  uint32_t v = 0;
  cudaError_t err = cudaMemcpyFromSymbol(&v, g_gptq_flags, sizeof v);
  if (err != cudaSuccess) return err;
  *flags = v;
  if (v) {
    const uint32_t zero = 0;
    err = cudaMemcpyToSymbol(g_gptq_flags, &zero, sizeof zero);
  }
  return err;
}

}  // namespace hscale
