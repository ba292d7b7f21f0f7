// factor_block.cuh -- one 128 x 128 diagonal block of the blocked Cholesky factor: factored and
// inverted by one CTA in shared memory (used by factor.cu for the first block and by the
// factor's update kernel in update.cu for every later one).
#pragma once
#include <cstdint>

namespace hscale {

constexpr int kNb = 128;                  // block of the sweep
constexpr int kSub = 16;                  // sub-block of the diagonal factor (one warp)
constexpr int kLd = kNb + 4;              // padded shared-memory row (16-byte multiple)
constexpr int kDiagThreads = 512;
constexpr int kDiagSmemBytes = (2 * kNb * kLd + 4) * 4;

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

// One warp factors the 16 x 16 block at A (row stride kLd, lower triangle), A = L L^T, and
// writes Z = L^-1 (lower, zeros above) at Zo (row stride kLd).  The block's own L is not
// needed: only Z is written.
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
// the approximate hardware ones.  A pivot that is not positive is kept in a register (the first
// one) and recorded once at the end, so no step branches.
//
// Measured on one GB300: 1.7 K cycles per 16 columns beside the other warps' products; the
// 32-wide sweep before this one, a Cholesky with square roots on the chain and 64 values per
// lane, took 7.5 K per 32 columns.
//
// Returns whether every pivot was in the range of the quick reciprocals (if not, nothing was
// recorded and Zo is to be formed again with kFull).
template <bool kFull>
__device__ __forceinline__ bool factor_sub16(const float* A, float* Zo, int lane, int32_t* info, int32_t base) {
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
  float lo = 1.0f, hi = 1.0f;  // the range of the pivots
  float ia, ic, r1;
  // the pivots j and j + 1 from the pivot block [a b; b c] (the same in every lane): ia = 1 / d_j,
  // ic = 1 / d_j+1, r1 = this lane's entry j + 1 after pivot j
  auto pivot = [&](int j, float a, float b, float c) {
    const bool bad_a = !(a > 0.0f);
    fail = (fail == 0 && bad_a) ? base + j + 1 : fail;
    a = bad_a ? 1.0f : a;
    ia = fast_rcp<kFull>(a);
    const float m = __fmul_rn(b, ia);
    // det 2^-e, e the exponent of a, so that it has the magnitude of d_j+1 = det / a
    const float as = __uint_as_float((__float_as_uint(a) & 0x007FFFFFu) | 0x3F800000u);  // a 2^-e
    const float bs = __fmul_rn(b, __uint_as_float(0x7F000000u - (__float_as_uint(a) & 0x7F800000u)));
    float det = __fmaf_rn(as, c, -__fmul_rn(bs, b));
    if (kFull) det = __fmul_rn(as, __fmaf_rn(-m, b, c));
    const bool bad_c = !(det > 0.0f);
    fail = (fail == 0 && bad_c) ? base + j + 2 : fail;
    det = bad_c ? as : det;
    ic = __fmul_rn(as, fast_rcp<kFull>(det));
    r1 = __fmaf_rn(-m, r[j], r[j + 1]);
    lo = fminf(lo, fminf(a, det));
    hi = fmaxf(hi, fmaxf(a, det));
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
  if (!kFull && !(lo >= 0x1p-100f && hi <= 0x1p100f)) return false;
  if (fail != 0 && lane == 0) record_failure(info, fail);
  // lane 16 + c holds column c of Y: row i is zero above the diagonal (i < c)
  if (!is_row) {
#pragma unroll
    for (int i = 0; i < kSub; ++i) Zo[i * kLd + li] = i >= li ? __fmul_rn(r[i], zs[i]) : 0.0f;
  }
  __syncwarp();
  return true;
}
static __device__ __noinline__ void factor_sub16_full(const float* A, float* Zo, int lane, int32_t* info, int32_t base) {
  factor_sub16<true>(A, Zo, lane, info, base);
}

__device__ __forceinline__ void block_factor(const float* A, float* Zo, int lane, int32_t* info, int32_t base) {
  if (!factor_sub16<false>(A, Zo, lane, info, base)) factor_sub16_full(A, Zo, lane, info, base);
}

// One warp's product of 16 x 16 blocks in shared memory (row stride kLd = 4 mod 32 words).
// A lane holds rows h, h + 8 and four columns: 4 cl + q (kNT false) or cl + 4 q (kNT true).
// Per four m, A's rows are 16-byte words, and B is read either row by row (kNT false: B[m][c]
// at B + m kLd + c) or in place from the transposed operand's rows (kNT true: B[m][c] at
// B + c kLd + m), 16-byte words too.  Shared-memory reads bound these products (a 16-byte read
// takes four cycles of the SM, two when neighbouring lanes i and i ^ 1, or i and i ^ 2, share
// the address; measured), so h leaves out lane bit 0, cl lane bit 1, and the rows and columns
// are dealt so that no read or write meets a bank twice.
//   acc[r][q] += sum_m A[h + 8 r][m] B[m][column q]   (-= with kNeg), over m in order
__device__ __forceinline__ int block_row(int lane) { return ((lane >> 3) & 3) + 2 * (lane & 2); }
__device__ __forceinline__ int block_col(int lane) { return ((lane >> 1) & 2) + (lane & 1); }

template <bool kNT, bool kNeg>
__device__ __forceinline__ void block_mma(float (&acc)[2][4], const float* A, const float* B, int lane) {
  const int h = block_row(lane), cl = block_col(lane);
#pragma unroll
  for (int m = 0; m < kSub; m += 4) {
    float b[4][4];  // b[m][q]
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float4 v = kNT ? *reinterpret_cast<const float4*>(B + (cl + 4 * q) * kLd + m)
                           : *reinterpret_cast<const float4*>(B + (m + q) * kLd + 4 * cl);
      const float e[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int k = 0; k < 4; ++k) (kNT ? b[k][q] : b[q][k]) = kNeg ? -e[k] : e[k];
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const float4 v = *reinterpret_cast<const float4*>(A + (h + 8 * r) * kLd + m);
      const float a[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[r][q] = __fmaf_rn(a[k], b[k][q], acc[r][q]);
    }
  }
}
__device__ __forceinline__ void block_zero(float (&acc)[2][4]) {
#pragma unroll
  for (int q = 0; q < 4; ++q) acc[0][q] = acc[1][q] = 0.0f;
}
template <bool kNT>
__device__ __forceinline__ void block_load(float (&acc)[2][4], const float* T, int lane) {
  const int h = block_row(lane), cl = block_col(lane);
#pragma unroll
  for (int r = 0; r < 2; ++r)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[r][q] = T[(h + 8 * r) * kLd + (kNT ? cl + 4 * q : 4 * cl + q)];
}
template <bool kNT>
__device__ __forceinline__ void block_store(const float (&acc)[2][4], float* T, int lane) {
  const int h = block_row(lane), cl = block_col(lane);
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    if (kNT) {
#pragma unroll
      for (int q = 0; q < 4; ++q) T[(h + 8 * r) * kLd + cl + 4 * q] = acc[r][q];
    } else {
      *reinterpret_cast<float4*>(T + (h + 8 * r) * kLd + 4 * cl) =
          make_float4(acc[r][0], acc[r][1], acc[r][2], acc[r][3]);
    }
  }
}

// P = P Z^T in place
__device__ __forceinline__ void block_panel(float* P, const float* Z, int lane) {
  float acc[2][4];
  block_zero(acc);
  block_mma<true, false>(acc, P, Z, lane);
  __syncwarp();
  block_store<true>(acc, P, lane);
}
// T = Z T in place
__device__ __forceinline__ void block_row_solve(float* T, const float* Z, int lane) {
  float acc[2][4];
  block_zero(acc);
  block_mma<false, false>(acc, Z, T, lane);
  __syncwarp();
  block_store<false>(acc, T, lane);
}
// T = -sum over count blocks of L (16 columns further each) times X (16 rows further each)
__device__ __forceinline__ void block_row_sum(float* T, const float* L, const float* X, int count, int lane) {
  float acc[2][4];
  block_zero(acc);
  for (int k = 0; k < count; ++k) block_mma<false, true>(acc, L + k * kSub, X + k * kSub * kLd, lane);
  block_store<false>(acc, T, lane);
}
// C -= A B^T
__device__ __forceinline__ void block_sub_nt(float* C, const float* A, const float* B, int lane) {
  float acc[2][4];
  block_load<true>(acc, C, lane);
  block_mma<true, true>(acc, A, B, lane);
  block_store<true>(acc, C, lane);
}
// The same for a 16 x 32 tile, C -= A B^T: a lane holds rows 2 h, 2 h + 1, 2 h + 8,
// 2 h + 9 and columns cl + 8 q (q < 4), which reads 32 bytes of shared memory per 16 products instead of 48.
__device__ __forceinline__ void wide_sub_nt(float* C, const float* A, const float* B, int lane) {
  const int h2 = (lane & 2) + ((lane >> 2) & 4), cl = (lane & 1) + ((lane >> 1) & 2) + ((lane >> 1) & 4);
  constexpr int kRow[4] = {0, 1, 8, 9};
  float acc[4][4];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[r][q] = C[(h2 + kRow[r]) * kLd + cl + 8 * q];
#pragma unroll
  for (int m = 0; m < kSub; m += 4) {
    float4 b[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) b[q] = *reinterpret_cast<const float4*>(B + (cl + 8 * q) * kLd + m);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const float4 a = *reinterpret_cast<const float4*>(A + (h2 + kRow[r]) * kLd + m);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        acc[r][q] = __fmaf_rn(-a.x, b[q].x, acc[r][q]);
        acc[r][q] = __fmaf_rn(-a.y, b[q].y, acc[r][q]);
        acc[r][q] = __fmaf_rn(-a.z, b[q].z, acc[r][q]);
        acc[r][q] = __fmaf_rn(-a.w, b[q].w, acc[r][q]);
      }
    }
  }
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int q = 0; q < 4; ++q) C[(h2 + kRow[r]) * kLd + cl + 8 * q] = acc[r][q];
}

// Factor the 128 x 128 block in S (row stride kLd, lower triangle; B_jj = L_jj L_jj^T) and
// invert the factor: Z_jj = L_jj^-1 in X (zero on entry above the diagonal; lower).  The block
// is an 8 x 8 grid of 16 x 16 blocks, taken in columns p = 0..7:
//   (a) warp 0 factors and inverts the block on the diagonal (factor_sub16): Z_p into X_pp;
//   (b) one warp each: the blocks below it, L_ip = B_ip Z_p^T (i > p, in place), and the
//       inverse's row, X_pc = Z_p T_pc (c < p, in place);
//   (c) right-looking in S, B_ik -= L_ip L_kp^T (p < k <= i), and left-looking in X, the next
//       row's T_p+1,c = -sum_{k=c..p} L_p+1,k X_kc (c <= p).
// Warp 0 runs ahead: of (b) and (c) it takes only the products on the way to the next diagonal
// block, L_p+1,p and B_p+1,p+1, and goes on to its (a) while the other warps run the rest,
// taking the products of (c) one at a time from a counter (the longest sums first).  A column
// costs the slower of the two.  Left-looking in X keeps (c) even: 19 to 28 products in every
// column, where right-looking would put 34 in the first and 7 in the last.
// Bound by the reads of shared memory in (c) (16 bytes a lane take two to four cycles of the SM)
// and, behind them, by the sub-factors.  One GB300: about 30 K cycles per 128-block, against 52 K
// for 32-wide tiles without look-ahead (the whole factor at n = 4096: 1755 -> 1540 us from this).
//
// S, X and the counter of (c) sit at byte `offset` of the kernel's dynamic shared memory
// (kDiagSmemBytes): the function finds them there itself, so that its accesses are shared-memory
// instructions (through a pointer whose origin the compiler does not see they are generic ones:
// 21.7 us a block instead of 16).
constexpr int kGrid16 = kNb / kSub;
static __device__ __noinline__ void factor_block128(uint32_t offset, int32_t* info, int32_t j0) {
  extern __shared__ __align__(16) uint8_t dynamic_smem[];
  float* S = reinterpret_cast<float*>(dynamic_smem + offset);
  float* X = S + kNb * kLd;
  int* next = reinterpret_cast<int*>(X + kNb * kLd);
  const int tid = (int)threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // column -1 is only warp 0's first sub-factor
#pragma unroll 1
  for (int p = -1; p < kGrid16; ++p) {
    const int c0 = p * kSub, d0 = c0 + kSub;
    const float* Zp = X + c0 * kLd + c0;
    if (warp == 0) {
      if (p + 1 == kGrid16) break;
      float* D = S + d0 * kLd + d0;
      if (p >= 0) {
        block_panel(S + d0 * kLd + c0, Zp, lane);
        __syncwarp();
        asm volatile("bar.arrive 1, 512;" ::: "memory");  // L_p+1,p is in place
        block_sub_nt(D, S + d0 * kLd + c0, S + d0 * kLd + c0, lane);
        __syncwarp();
      }
      block_factor(D, X + d0 * kLd + d0, lane, info, j0 + d0);
    } else if (p >= 0) {
      // (b): c < p on warps 1..p, i > p + 1 on warps p + 1..6
      if (warp <= p) {
        block_row_solve(X + c0 * kLd + (warp - 1) * kSub, Zp, lane);
      } else if (warp + 1 < kGrid16) {
        block_panel(S + (warp + 1) * kSub * kLd + c0, Zp, lane);
      } else if (tid == kDiagThreads - 1) {
        *next = 0;
      }
      if (p + 1 == kGrid16) break;
      asm volatile("bar.sync 1, 512;" ::: "memory");
      // (c): T_p+1,c for c = 0..p, then rows i > p + 1 of S, two blocks (i, k), (i, k + 1)
      // at a time
      for (;;) {
        int e = 0;
        if (lane == 0) e = atomicAdd(next, 1);
        e = __shfl_sync(0xFFFFFFFFu, e, 0);
        if (e <= p) {
          block_row_sum(X + d0 * kLd + e * kSub, S + d0 * kLd + e * kSub, X + e * kSub * kLd + e * kSub, p + 1 - e,
                        lane);
          continue;
        }
        int i = p + 2, k = e - (p + 1);  // row i has (i - p + 1) / 2 tiles
        while (i < kGrid16 && k >= (i - p + 1) / 2) {
          k -= (i - p + 1) / 2;
          ++i;
        }
        if (i >= kGrid16) break;
        k = p + 1 + 2 * k;
        float* C = S + i * kSub * kLd + k * kSub;
        const float* L = S + i * kSub * kLd + c0;
        if (k < i)
          wide_sub_nt(C, L, S + k * kSub * kLd + c0, lane);
        else
          block_sub_nt(C, L, L, lane);
      }
    }
    __syncthreads();
  }
  __syncthreads();
}

}  // namespace hscale
