// factor_block.cuh -- one 128 x 128 diagonal block of the blocked Cholesky factor: factored and
// inverted by one CTA in shared memory (used by factor.cu for the first block and by the
// factor's update kernel in update.cu for every later one).
#pragma once
#include <cuda_bf16.h>

#include <cstdint>

#include "tma.cuh"

namespace hscale {

constexpr int kNb = 128;                  // block of the sweep
constexpr int kSub = 16;                  // sub-block of the diagonal factor (one warp)
constexpr int kLd = kNb + 4;              // padded shared-memory row (16-byte multiple)
constexpr int kDiagThreads = 512;
constexpr int kPlane = kSub + 8;          // row (bf16) of a split operand: eight of them meet no bank twice
// the block, its current column's splits, two sub-factors' splits, the sub-factor's input
constexpr int kDiagSmemBytes = kNb * kLd * 4 + 3 * kNb * kPlane * 2 + 2 * 3 * kSub * kPlane * 2 + kSub * kLd * 4;

__device__ __forceinline__ void record_failure(int32_t* info, int32_t order) {
  atomicCAS(reinterpret_cast<int*>(info), 0, order);
}

// Fast reciprocal and reciprocal square root (relative error within about 2^-22): the quick
// forms take operands and results in the normal range, kFull those outside it too.
template <bool kFull>
__device__ __forceinline__ float fast_rcp(float x) {
  float r;
  if (kFull) asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  else asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
template <bool kFull>
__device__ __forceinline__ float fast_rsqrt(float x) {
  float r;
  if (kFull) asm("rsqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  else asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// The three bf16 parts of a pair of values, packed (x in the low half).
__device__ __forceinline__ void split3_pair(float x, float y, uint32_t (&p)[3]) {
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(x, y);
    p[s] = *reinterpret_cast<const uint32_t*>(&v);
    x = __fsub_rn(x, __uint_as_float(p[s] << 16));
    y = __fsub_rn(y, __uint_as_float(p[s] & 0xFFFF0000u));
  }
}

// One warp factors the 16 x 16 block at A (row stride kLd, lower triangle), A = L L^T, and
// writes Z = L^-1 (lower, zeros above) as three bf16 parts (split3_pair), transposed, kSub rows of
// kPlane each, at Zo.  The block's own L is not needed: only Z is written.
//
// Two halves of the warp run the same instructions: lane i < 16 holds row i of the block,
// lane 16 + c holds column c of the unit-lower inverse Y, which starts as the identity.  The
// elimination is A = M diag(d) M^T with unit-lower M, two pivots per step: with the pivot
// columns C0 (column j) and C1' = C1 - C0 b / a (column j + 1 after pivot j), every lane forms
// its x0 = r_j / a and x1 = r'_j+1 / d_j+1 and subtracts C0_k x0 + C1'_k x1 from its entry k:
// for a row this is the Schur update, for a column of Y the forward substitution, and
// both take the same pair (C0_k, C1'_k), by shuffle from lane k.  At the end row i of Y is
// scaled by 1 / sqrt(d_i), which gives Z.
//
// What bounds it is the chain from one pivot pair to the next, so that chain
// holds no square root, and its two reciprocals run side by side: 1 / a, and 1 / det of the
// 2 x 2 pivot block (1 / d_j+1 = a / det).  Each step forms the next pivot block first, the same
// in every lane from entries shuffled before the update (no shuffle of updated values on the
// chain), and the rest of its update fits in the chain's shadow.  The reciprocals are
// the approximate hardware ones.  The quick form only notes the ranges of a and det, which a pivot
// that is not positive leaves too; kFull keeps the first such pivot in a register and records it
// once at the end, so no step branches.
//
// Measured on one GB300: 1.9 K cycles per 16 columns beside other warps' work; the
// 32-wide sweep before this one, a Cholesky with square roots on the chain and 64 values per
// lane, took 7.5 K per 32 columns.
//
// Returns whether every pivot was positive and in the range where the quick form's reciprocals and
// det neither underflow nor overflow (if not, nothing was recorded and Zo is to be formed again
// with kFull).
template <bool kFull>
__device__ __forceinline__ bool factor_sub16(const float* A, uint16_t* Zo, int lane, int32_t* info, int32_t base) {
  const unsigned full = 0xFFFFFFFFu;
  const bool is_row = lane < kSub;
  const int li = lane & (kSub - 1);
  float r[kSub], zs[kSub];  // the row or column; 1 / sqrt(d_k)
#pragma unroll
  for (int k = 0; k < kSub; k += 4) {
    const float4 a = *reinterpret_cast<const float4*>(A + li * kLd + k);
    r[k] = is_row ? a.x : (k == li ? 1.0f : 0.0f);
    r[k + 1] = is_row ? a.y : (k + 1 == li ? 1.0f : 0.0f);
    r[k + 2] = is_row ? a.z : (k + 2 == li ? 1.0f : 0.0f);
    r[k + 3] = is_row ? a.w : (k + 3 == li ? 1.0f : 0.0f);
  }
  int32_t fail = 0;
  float lo = 1.0f, hi = 1.0f, det_lo = 1.0f, det_hi = 1.0f;  // the ranges of a and of det
  float ia, ic, r1, det;
  // the pivots j and j + 1 from the pivot block [a b; b c] (the same in every lane): ia = 1 / d_j,
  // ic = 1 / d_j+1, r1 = this lane's entry j + 1 after pivot j
  auto pivot = [&](int j, float a, float b, float c) {
    if (!kFull) {
      ia = fast_rcp<kFull>(a);
      det = __fmaf_rn(a, c, -__fmul_rn(b, b));
      ic = __fmul_rn(a, fast_rcp<kFull>(det));
      r1 = __fmaf_rn(-__fmul_rn(b, ia), r[j], r[j + 1]);
      lo = fminf(lo, a);
      hi = fmaxf(hi, a);
      det_lo = fminf(det_lo, det);
      det_hi = fmaxf(det_hi, det);
      return;
    }
    const bool bad_a = !(a > 0.0f);
    fail = (fail == 0 && bad_a) ? base + j + 1 : fail;
    a = bad_a ? 1.0f : a;
    ia = fast_rcp<kFull>(a);
    const float m = __fmul_rn(b, ia);
    // det 2^-e, e the exponent of a, so that it has the magnitude of d_j+1 = det / a
    const float as = __uint_as_float((__float_as_uint(a) & 0x007FFFFFu) | 0x3F800000u);  // a 2^-e
    det = __fmul_rn(as, __fmaf_rn(-m, b, c));
    const bool bad_c = !(det > 0.0f);
    fail = (fail == 0 && bad_c) ? base + j + 2 : fail;
    det = bad_c ? as : det;
    ic = __fmul_rn(as, fast_rcp<kFull>(det));
    r1 = __fmaf_rn(-m, r[j], r[j + 1]);
  };
  pivot(0, __shfl_sync(full, r[0], 0), __shfl_sync(full, r[0], 1), __shfl_sync(full, r[1], 1));
#pragma unroll
  for (int j = 0; j < kSub; j += 2) {
    const float rj = r[j], rj1 = r1, ja = ia, jc = ic;
    r[j + 1] = r1;
    const float x0 = __fmul_rn(rj, ja), x1 = __fmul_rn(rj1, jc);
    if (j + 2 < kSub) {
      // the next pivot block before this step's update, and the pivot columns' entries in its
      // two rows: every lane forms the updated block itself, the same way lanes j + 2 and j + 3
      // update their rows
      const int k = j + 2;
      const float a0 = __shfl_sync(full, r[k], k), b0 = __shfl_sync(full, r[k], k + 1);
      const float c0 = __shfl_sync(full, r[k + 1], k + 1);
      const float s0 = __shfl_sync(full, rj, k), t0 = __shfl_sync(full, rj, k + 1);
      const float s1 = __shfl_sync(full, rj1, k), t1 = __shfl_sync(full, rj1, k + 1);
      const float u0 = __fmul_rn(s0, ja), v0 = __fmul_rn(t0, ja), u1 = __fmul_rn(s1, jc), v1 = __fmul_rn(t1, jc);
      r[k] = __fmaf_rn(-s1, x1, __fmaf_rn(-s0, x0, r[k]));
      r[k + 1] = __fmaf_rn(-t1, x1, __fmaf_rn(-t0, x0, r[k + 1]));
      pivot(k, __fmaf_rn(-s1, u1, __fmaf_rn(-s0, u0, a0)), __fmaf_rn(-s1, v1, __fmaf_rn(-s0, v0, b0)),
            __fmaf_rn(-t1, v1, __fmaf_rn(-t0, v0, c0)));
#pragma unroll
      for (int i = j + 4; i < kSub; ++i)
        r[i] = __fmaf_rn(-__shfl_sync(full, rj1, i), x1, __fmaf_rn(-__shfl_sync(full, rj, i), x0, r[i]));
    }
    zs[j] = __fmul_rn(ja, fast_rsqrt<kFull>(ja));
    zs[j + 1] = __fmul_rn(jc, fast_rsqrt<kFull>(jc));
  }
  // a NaN passes the minima and maxima, but reaches every later pivot
  if (!kFull && !(lo >= 0x1p-50f && hi <= 0x1p50f && det_lo >= 0x1p-100f && det_hi <= 0x1p100f && det > 0.0f))
    return false;
  if (fail != 0 && lane == 0) record_failure(info, fail);
  // lane 16 + c holds column c of Y (row i is zero above the diagonal, i < c) and writes its rows
  // 0-7 of Z, lane c the rows 8-15
  float z[kSub / 2];
#pragma unroll
  for (int i = 0; i < kSub / 2; ++i) {
    const float lower = __shfl_sync(full, r[i + 8], li + kSub);
    const float y = is_row ? __fmul_rn(lower, zs[i + 8]) : __fmul_rn(r[i], zs[i]);
    z[i] = i + (is_row ? 8 : 0) >= li ? y : 0.0f;
  }
  uint32_t part[3][4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    uint32_t pr[3];
    split3_pair(z[2 * i], z[2 * i + 1], pr);
#pragma unroll
    for (int s = 0; s < 3; ++s) part[s][i] = pr[s];
  }
#pragma unroll
  for (int s = 0; s < 3; ++s)
    *reinterpret_cast<uint4*>(Zo + (s * kSub + li) * kPlane + (is_row ? 8 : 0)) =
        make_uint4(part[s][0], part[s][1], part[s][2], part[s][3]);
  __syncwarp();
  return true;
}
static __device__ __noinline__ void factor_sub16_full(const float* A, uint16_t* Zo, int lane, int32_t* info,
                                                      int32_t base) {
  factor_sub16<true>(A, Zo, lane, info, base);
}

// ---------------------------------------------------------------- warp-level products
// mma.sync m16n8k16 on bf16 parts, fp32 accumulation.  These products are too small and too
// dependent on each other for the tcgen05 units (one 16 x 16 x 16 product at a time, needed by the
// next one); they run on registers.  A 16 x 16 block is a fragment of two n8 halves:
// f[h][0..1] row g, columns 8 h + 2 t, + 1; f[h][2..3] row g + 8 (g = lane / 4, t = lane % 4).
__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// A block as the A operand of three parts (the accumulator's layout is the operand's).
__device__ __forceinline__ void split_fragment(const float (&f)[2][4], uint32_t (&a)[3][4]) {
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      uint32_t p[3];
      split3_pair(f[h][2 * q], f[h][2 * q + 1], p);
#pragma unroll
      for (int s = 0; s < 3; ++s) a[s][2 * h + q] = p[s];
    }
}
// f = A B^T to fp32 accuracy, A and B 16 x 16 in three parts each: the six products above 2^-24, the
// small ones in a sum of their own, which also halves the chain of dependent MMAs.
// b[s][0..1]: rows 0-7 of B's part s (columns 0-7, 8-15), b[s][2..3]: rows 8-15.
__device__ __forceinline__ void block_product(float (&f)[2][4], const uint32_t (&a)[3][4], const uint32_t (&b)[3][4]) {
  float e[2][4];
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int q = 0; q < 4; ++q) e[h][q] = f[h][q] = 0.0f;
  auto both = [&](float (&d)[2][4], int i, int j) {
#pragma unroll
    for (int h = 0; h < 2; ++h) mma16816(d[h], a[i], b[j][2 * h], b[j][2 * h + 1]);
  };
  both(e, 0, 2);
  both(f, 0, 1);
  both(e, 2, 0);
  both(f, 1, 0);
  both(e, 1, 1);
  both(f, 0, 0);
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int q = 0; q < 4; ++q) f[h][q] = __fadd_rn(f[h][q], e[h][q]);
}
// The block B of that product (kTransposed: stored as its transpose) from shared memory: three
// parts of kPlane-wide rows, `part` elements apart.
template <bool kTransposed>
__device__ __forceinline__ void load_block(uint32_t (&b)[3][4], const uint16_t* B, int part, int lane) {
  // the 8 x 8 block of lanes 8 i .. 8 i + 7: rows 8 (i / 2) of B, columns 8 (i % 2)
  const int n = (lane >> 1) & 8, k = lane & 8;
  const uint32_t at = smem_addr(B + ((kTransposed ? k : n) + (lane & 7)) * kPlane + (kTransposed ? n : k));
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    const uint32_t src = at + (uint32_t)(s * part * 2);
    if (kTransposed)
      asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                   : "=r"(b[s][0]), "=r"(b[s][1]), "=r"(b[s][2]), "=r"(b[s][3])
                   : "r"(src)
                   : "memory");
    else
      asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                   : "=r"(b[s][0]), "=r"(b[s][1]), "=r"(b[s][2]), "=r"(b[s][3])
                   : "r"(src)
                   : "memory");
  }
}

// Factor the 128 x 128 block B in shared memory (at byte `offset` of the kernel's dynamic shared
// memory, row stride kLd; its lower triangle) and write the factor's inverse, Z = L^-1, to xo (row
// stride ld, zeros above the diagonal).
//
// Elimination of the tall matrix [B ; I], taken in 16-wide columns p = 0..7: with
// Z_p = L_pp^-1 (factor_sub16), every row block has P = V_p Z_p^T (for a row block of B that
// is L_rp; for row block c of I, X_pc^T, a block of the inverse) and V_i -= P L_ip^T for the columns
// i > p.  So a row block needs from the others only Z_p and the L_ip: each of the 16 warps
// holds one row block in registers for the whole elimination (eight 16 x 16 blocks), warps 0-7
// those of B, 8-15 those of I; the products are warp-level MMAs on three bf16 parts, and only
// Z_p and the column's L_ip go through shared memory, as parts.
//
// What bounds it is the chain of the sub-factors, about 1.9 K of a column's 2.7 K cycles.  The warp of
// row block p + 1 carries it: with Z_p it forms P and from that its diagonal block, both in
// registers (P's fragment is either operand of P P^T), and factors it, while the other warps
// update their columns.  Row block r of B is done with column r - 1, so the lead passes from warp
// to warp, each of which has split its first block before Z_p comes.  The warp index has to be
// uniform: with one taken per thread the n = 4096 factor took 934 us in place of 868.
//
// One GB300: 10.5 us a block inside the update kernel, against 16.4 with the products on CUDA cores
// through shared memory, whose reads bound them (n = 4096 factor 1030 -> 852 us in a graph); about
// 0.3 us less since the others no longer wait for the lead's L_p+1,p before their own P (837 -> 825
// eager).
constexpr int kGrid16 = kNb / kSub;
static __device__ __noinline__ void factor_block128(uint32_t offset, float* __restrict__ xo, int64_t ld, int32_t* info,
                                                    int32_t j0) {
  extern __shared__ __align__(16) uint8_t dynamic_smem[];
  const float* S = reinterpret_cast<const float*>(dynamic_smem + offset);
  uint16_t* Lp = reinterpret_cast<uint16_t*>(dynamic_smem + offset + kNb * kLd * 4);
  uint16_t* Zp = Lp + 3 * kNb * kPlane;  // two of them
  float* D = reinterpret_cast<float*>(Zp + 2 * 3 * kSub * kPlane);
  const int lane = (int)threadIdx.x & 31, warp = (int)warp_uniform(threadIdx.x >> 5);
  const int g = lane >> 2, t = lane & 3, r = warp & 7;
  const bool of_b = warp < kGrid16;
  float v[kGrid16][2][4];  // the row block's columns p, p + 1, ...
  if (warp != 0) {
#pragma unroll
    for (int i = 0; i < kGrid16; ++i)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int c = 8 * h + 2 * t;
        float2 x = make_float2(0.0f, 0.0f), y = x;
        if (of_b && i <= r) {
          x = *reinterpret_cast<const float2*>(S + (kSub * r + g) * kLd + kSub * i + c);
          y = *reinterpret_cast<const float2*>(S + (kSub * r + g + 8) * kLd + kSub * i + c);
        }
        v[i][h][0] = x.x; v[i][h][1] = x.y; v[i][h][2] = y.x; v[i][h][3] = y.y;
      }
  }

#pragma unroll 1
  for (int p = 0; p < kGrid16; ++p) {
    if (warp == p) {  // this row block of B has only its sub-factor left
      const float* A = p == 0 ? S : D;
      uint16_t* Zn = Zp + (p & 1) * 3 * kSub * kPlane;
      __syncwarp();  // D is in place
      const int32_t base = j0 + kSub * p;
      if (!factor_sub16<false>(A, Zn, lane, info, base)) factor_sub16_full(A, Zn, lane, info, base);
      // the row block's registers are the sub-factor's until here
#pragma unroll
      for (int i = 0; i < kGrid16; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int q = 0; q < 4; ++q) v[i][h][q] = 0.0f;
    }
    uint32_t a[3][4];
    if (!of_b && r == p) {  // its first column
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int q = 0; q < 4; ++q) v[0][h][q] = g + 8 * (q >> 1) == 8 * h + 2 * t + (q & 1) ? 1.0f : 0.0f;
    }
    const bool active = of_b ? r > p : r <= p;
    const bool lead = of_b && r == p + 1;
    if (active) split_fragment(v[0], a);
    __syncthreads();  // Z_p is in place, the reads of the last column's L are done
    float P[2][4] = {};
    if (active) {
      uint32_t z[3][4];
      load_block<true>(z, Zp + (p & 1) * 3 * kSub * kPlane, kSub * kPlane, lane);
      block_product(P, a, z);
      split_fragment(P, a);
      if (of_b) {
#pragma unroll
        for (int s = 0; s < 3; ++s)
#pragma unroll
          for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int q = 0; q < 2; ++q)
              *reinterpret_cast<uint32_t*>(Lp + (s * kNb + kSub * r + g + 8 * q) * kPlane + 8 * h + 2 * t) =
                  a[s][2 * h + q];
      }
    }
    if (!of_b) {
      // X[16 p + column][16 r + row]; zeros above the block diagonal (p < r)
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int q = 0; q < 4; ++q)
          xo[(int64_t)(kSub * p + 8 * h + 2 * t + (q & 1)) * ld + kSub * r + g + 8 * (q >> 1)] = P[h][q];
    }
    if (p + 1 == kGrid16) break;
    if (lead) {
      asm volatile("bar.arrive 1, 512;" ::: "memory");  // L_p+1,p is in place
      uint32_t b[3][4];
      float d[2][4];
#pragma unroll
      for (int s = 0; s < 3; ++s) {
        b[s][0] = a[s][0];
        b[s][1] = a[s][2];
        b[s][2] = a[s][1];
        b[s][3] = a[s][3];
      }
      block_product(d, a, b);
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int q = 0; q < 2; ++q)
          *reinterpret_cast<float2*>(D + (g + 8 * q) * kLd + 8 * h + 2 * t) = make_float2(
              __fsub_rn(v[1][h][2 * q], d[h][2 * q]), __fsub_rn(v[1][h][2 * q + 1], d[h][2 * q + 1]));
    } else {
      asm volatile("bar.sync 1, 512;" ::: "memory");  // the column's L is in place
      if (active) {
        const int last = of_b ? r - p : kGrid16 - 1 - p;
#pragma unroll
        for (int k = 1; k < kGrid16; ++k)
          if (k <= last) {
            uint32_t b[3][4];
            float f[2][4];
            load_block<false>(b, Lp + kSub * (p + k) * kPlane, kNb * kPlane, lane);
            block_product(f, a, b);
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
              for (int q = 0; q < 4; ++q) v[k - 1][h][q] = __fsub_rn(v[k][h][q], f[h][q]);
          }
      }
    }
  }
}

}  // namespace hscale
