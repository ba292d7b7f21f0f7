// factor.cu -- the damped inverse-Cholesky factor of GPTQ (Algorithm 3) on sm_103a.
//
// U is upper triangular with U^T U = A^-1 for the damped Hessian A = H + damp * mean(diag H) I
// (dead channels, H_jj = 0, get H_jj = 1 first).  With J the order-reversing permutation and
// B = J A J = L L^T (L lower, Cholesky), A = (J L J)(J L^T J), so U = (J L J)^-1 = J L^-1 J:
// upper triangular with a positive diagonal, hence the Cholesky factor of A^-1.  No inverse of
// A is formed.
//
// B is padded to n_pad = 128 * ceil(n / 128) with an identity block, whose factor and inverse
// are the identity.  B (then L, lower) and X (R, then X = L^-1, lower) sit side by side in one
// [n_pad, 2 n_pad] buffer, so that the two updates of a step are one GEMM over contiguous
// columns.  The sweep takes 128-wide block columns j = 0, 1, ...  (right-looking):
//   diag     the CTA of factor_diag_kernel factors the (updated) diagonal block,
//            B_jj = L_jj L_jj^T, in shared memory and inverts it, Z_jj = L_jj^-1, into the
//            inverse's diagonal block (16-wide blocks: one warp factors and inverts each 16 x 16
//            block on the diagonal and runs ahead, the CTA's other warps update the rest);
//   strips   panel L_ij = B_ij Z_jj^T (i > j) and the inverse's row X_j,c = Z_jj R_j,c (c < j),
//            in 64-wide strips on CUDA cores (factor_strip_kernel);
//   updates  B_ik -= L_ij L_kj^T over the trailing square, and R_ic -= L_ij X_jc for i > j,
//            c <= j: for the rows below the diagonal block, the columns from the trailing
//            square's first to the inverse's block j are contiguous in the buffer, n_pad of
//            them, and both updates are one product -L_:j [L_:j ; X_j,:]^T.  It runs on the
//            tensor cores: the tcgen05 GEMM with three-way bf16 splits of both operands (the
//            six products above 2^-24 relative, one GEMM over K = 6 * 128), which carries
//            fp32-level accuracy.
// X = L^-1 is built alongside: row blocks below the diagonal accumulate
// R_ic = -sum_k L_ik X_kc as the sweep passes, and X_ic = Z_ii R_ic once row block i is reached.
// A last kernel writes U_ij = X_{n-1-i, n-1-j}.
//
// A pivot that is not positive (the damped matrix is then not positive definite) is recorded
// in info[0] as its 1-based order in B and replaced by 1, so the sweep ends with finite values;
// U is then unspecified.
#include <cuda_bf16.h>

#include <algorithm>

#include "hscale_internal.h"
#include "tma.cuh"

namespace hscale {
namespace {

constexpr int kNb = 128;                  // block of the sweep
constexpr int kSub = 16;                  // sub-block of the diagonal factor (one warp)
constexpr int kLd = kNb + 4;              // padded shared-memory row (16-byte multiple)
constexpr int kDiagThreads = 512;
constexpr int kDiagSmemBytes = (2 * kNb * kLd + 4) * 4;
constexpr int kStripRows = 32;            // rows (or columns) of one strip
constexpr int kStripThreads = 256;
constexpr int kStripSmemBytes = (kNb * (kNb + 4) + kNb * (kStripRows + 4)) * 4;
constexpr int kSplitK = 6 * kNb;          // K of the split update GEMMs

// ---------------------------------------------------------------- set-up
// One block: dead channels (H_jj = 0) and the damped diagonal dd_j = d_j + damp * mean(d),
// d_j = H_jj, or 1 for a dead channel (fp32; the mean in fp64).
__global__ void __launch_bounds__(1024) damp_diagonal_kernel(const float* __restrict__ H, int64_t n, int64_t ld_h,
                                                             float damp, uint8_t* __restrict__ dead,
                                                             float* __restrict__ dd) {
  __shared__ double part[1024];
  double s = 0.0;
#pragma unroll 4
  for (int64_t j = threadIdx.x; j < n; j += blockDim.x) {
    float d = H[j * ld_h + j];
    const bool is_dead = (d == 0.0f);
    if (is_dead) d = 1.0f;
    if (dead) dead[j] = (uint8_t)is_dead;
    dd[j] = d;
    s += (double)d;
  }
  part[threadIdx.x] = s;
  __syncthreads();
  for (int step = 512; step > 0; step >>= 1) {
    if ((int)threadIdx.x < step) part[threadIdx.x] += part[threadIdx.x + step];
    __syncthreads();
  }
  const float add = (float)((double)damp * part[0] / (double)n);
  for (int64_t j = threadIdx.x; j < n; j += blockDim.x) dd[j] = dd[j] + add;
}

// W2 [n_pad, 2 n_pad]: the left half B_ij = A_{n-1-i, n-1-j} for i, j < n, A the damped H
// (read from H's upper triangle, row stride ld_h, and the damped diagonal dd), the identity
// beyond n; the right half (X) zero where the sweep accumulates into it, strictly below the
// 128-block diagonal (nothing reads X above it).  One 32 x 32 tile of each half per block.
// Every read and write runs along a row: a tile of B below the diagonal reads H's rows
// (reversed), a tile above it reads the mirrored tile of H and transposes it in shared
// memory, and a tile on the diagonal reads the entries on and below it and takes the rest
// from its own transpose.
__global__ void __launch_bounds__(256) reverse_pad_kernel(const float* __restrict__ H, int64_t n, int64_t ld_h,
                                                          const float* __restrict__ dd, int64_t n_pad,
                                                          float* __restrict__ W2) {
  __shared__ float t[32][33];
  const int bi = (int)blockIdx.y, bj = (int)blockIdx.x;
  const int64_t i0 = 32 * (int64_t)bi, j0 = 32 * (int64_t)bj, ld = 2 * n_pad;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  if (bi < bj) {
    // B_ij = A_{n-1-j, n-1-i}: t[jj][ii]
    for (int jj = ty; jj < 32; jj += 8) {
      const int64_t j = j0 + jj, i = i0 + tx;
      t[jj][tx] = (i < n && j < n) ? H[(n - 1 - j) * ld_h + (n - 1 - i)] : 0.0f;
    }
    __syncthreads();
    for (int ii = ty; ii < 32; ii += 8) W2[(i0 + ii) * ld + j0 + tx] = t[tx][ii];  // i < j: 0 beyond n
  } else {
    // B_ij = A_{n-1-i, n-1-j} for i >= j: t[ii][jj]
    for (int ii = ty; ii < 32; ii += 8) {
      const int64_t i = i0 + ii, j = j0 + tx;
      t[ii][tx] = (i < n && j < n && i >= j) ? H[(n - 1 - i) * ld_h + (n - 1 - j)] : 0.0f;
    }
    __syncthreads();
    for (int ii = ty; ii < 32; ii += 8) {
      const int64_t i = i0 + ii, j = j0 + tx;
      float v;
      if (i < n && j < n)
        v = i == j ? dd[n - 1 - i] : (i > j ? t[ii][tx] : t[tx][ii]);
      else
        v = i == j ? 1.0f : 0.0f;
      W2[i * ld + j] = v;
    }
  }
  if (bi / (kNb / 32) > bj / (kNb / 32))
    for (int ii = ty; ii < 32; ii += 8) W2[(i0 + ii) * ld + n_pad + j0 + tx] = 0.0f;
}

// U_ij = X_{n-1-i, n-1-j} for j >= i, 0 below the diagonal (U row stride n; X row stride ld);
// rows i = blockIdx.y, + gridDim.y, ...
__global__ void __launch_bounds__(256) reverse_out_kernel(const float* __restrict__ Xw, int64_t ld, int64_t n,
                                                          float* __restrict__ U) {
  const int64_t j = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (j >= n) return;
#pragma unroll 4
  for (int64_t i = blockIdx.y; i < n; i += gridDim.y) U[i * n + j] = j >= i ? Xw[(n - 1 - i) * ld + (n - 1 - j)] : 0.0f;
}

// ---------------------------------------------------------------- diagonal block
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
__device__ __noinline__ void factor_sub16_full(const float* A, float* Zo, int lane, int32_t* info, int32_t base) {
  factor_sub16<true>(A, Zo, lane, info, base);
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
// and, behind them, by the sub-factors.  One GB300: 29 K cycles per 128-block, against 52 K for
// 32-wide tiles without look-ahead; n = 4096: the call 1755 -> 1540 us.
constexpr int kGrid16 = kNb / kSub;
__device__ __forceinline__ void factor_block128(float* S, float* X, int* next, int tid, int32_t* info, int32_t j0) {
  const int lane = tid & 31, warp = tid >> 5;
  auto sub = [&](float* A, float* Z, int32_t base) {
    if (!factor_sub16<false>(A, Z, lane, info, base)) factor_sub16_full(A, Z, lane, info, base);
  };
  if (warp == 0) sub(S, X, j0);
  __syncthreads();
  for (int p = 0; p < kGrid16; ++p) {
    const int c0 = p * kSub, d0 = c0 + kSub;
    const float* Zp = X + c0 * kLd + c0;
    auto panel = [&](int i) {
      float* P = S + i * kSub * kLd + c0;
      float acc[2][4];
      block_zero(acc);
      block_mma<true, false>(acc, P, Zp, lane);
      __syncwarp();
      block_store<true>(acc, P, lane);
    };
    if (warp == 0) {
      if (p + 1 == kGrid16) break;
      panel(p + 1);
      __syncwarp();
      asm volatile("bar.arrive 1, 512;" ::: "memory");  // L_p+1,p is in place
      float acc[2][4];
      float* D = S + d0 * kLd + d0;
      block_load<true>(acc, D, lane);
      block_mma<true, true>(acc, S + d0 * kLd + c0, S + d0 * kLd + c0, lane);
      block_store<true>(acc, D, lane);
      __syncwarp();
      sub(D, X + d0 * kLd + d0, j0 + d0);
    } else {
      // (b): c < p on warps 1..p, i > p + 1 on warps p + 1..6 (7 in the last column)
      if (warp <= p) {
        float* T = X + c0 * kLd + (warp - 1) * kSub;
        float acc[2][4];
        block_zero(acc);
        block_mma<false, false>(acc, Zp, T, lane);
        __syncwarp();
        block_store<false>(acc, T, lane);
      } else if (warp + 1 < kGrid16) {
        panel(warp + 1);
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
          float acc[2][4];
          block_zero(acc);
          for (int k = e; k <= p; ++k)
            block_mma<false, true>(acc, S + d0 * kLd + k * kSub, X + k * kSub * kLd + e * kSub, lane);
          block_store<false>(acc, X + d0 * kLd + e * kSub, lane);
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
        if (k < i) {
          wide_sub_nt(C, L, S + k * kSub * kLd + c0, lane);
        } else {
          float acc[2][4];
          block_load<true>(acc, C, lane);
          block_mma<true, true>(acc, L, L, lane);
          block_store<true>(acc, C, lane);
        }
      }
    }
    __syncthreads();
  }
  __syncthreads();
}

// The diagonal block at (j0, j0) of Bw: Z_jj into Xw's diagonal block (zeros above the
// diagonal).  One CTA.  Only the lower triangle of the block is used.
__global__ void __launch_bounds__(kDiagThreads, 1)
factor_diag_kernel(const float* __restrict__ Bw, int64_t ld, int64_t j0, float* __restrict__ Xw,
                   int32_t* __restrict__ info) {
  extern __shared__ __align__(16) float sm[];
  float* S = sm;                 // [128][kLd] the block, then L (lower)
  float* X = S + kNb * kLd;      // [128][kLd] the inverse (lower)
  int* next = reinterpret_cast<int*>(X + kNb * kLd);  // the counter of factor_block128
  const int tid = threadIdx.x;

  // programmatic dependent launch: the strips may be scheduled now; the previous step's update
  // must have finished before the block is read
  pdl_launch_dependents();
  pdl_wait_primary();
  const float* blk = Bw + j0 * ld + j0;
  // independent 16-byte loads per thread in flight
#pragma unroll
  for (int t = 0; t < kNb * kNb / 4 / kDiagThreads; ++t) {
    const int e = tid + t * kDiagThreads;
    const int r = e >> 5, c = (e & 31) * 4;
    *reinterpret_cast<float4*>(S + r * kLd + c) = *reinterpret_cast<const float4*>(blk + r * ld + c);
    *reinterpret_cast<float4*>(X + r * kLd + c) = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  __syncthreads();
  factor_block128(S, X, next, tid, info, (int32_t)j0);
  // write-out: Z into Xw's diagonal block (16-byte words).  L_jj itself is not needed again:
  // the panel uses Z_jj, and the rest of the sweep reads only the blocks below the diagonal.
  float* xo = Xw + j0 * ld + j0;
#pragma unroll 4
  for (int t = 0; t < kNb * kNb / 4 / kDiagThreads; ++t) {
    const int e = tid + t * kDiagThreads;
    const int r = e >> 5, c = (e & 31) * 4;
    *reinterpret_cast<float4*>(xo + r * ld + c) = *reinterpret_cast<const float4*>(X + r * kLd + c);
  }
}

// ---------------------------------------------------------------- strips (CUDA cores)
// Blocks [0, panel_strips): the panel below the diagonal block, 32 rows each:
//   P[i][c] = sum_{m <= c} B[i][j0 + m] Z[c][m]        (L_ij = B_ij Z_jj^T, rows i of B)
// written to P (row stride 128, rows relative to r_first).
// Blocks [panel_strips, ...): the inverse's row j, 32 columns each, in place in Xw:
//   X[j0 + r][c] = sum_{m <= r} Z[r][m] R[j0 + m][c]   (X_jc = Z_jj R_jc, c < j0)
// Z = Z_jj is Xw's diagonal block.  256 threads; each computes 4 x 4 outputs over K = 128 from
// shared memory, reading four consecutive m per 16-byte load: the panel's columns
// c = tx + 32 k take Z's rows 132 words apart (each load spans every bank in four
// wavefronts), the shared operand of a warp is a broadcast, and the row's columns are one
// 16-byte word.  The sums run over m in order.  The staging loads are unrolled so that each
// thread has several in flight.
__global__ void __launch_bounds__(kStripThreads)
factor_strip_kernel(const float* __restrict__ Bw, float* __restrict__ Xw, int64_t ld, int64_t j0,
                    float* __restrict__ P, int panel_strips, int64_t r_first) {
  // launched in stream order (scheduled early, beside the diagonal block's CTA, the strips ran
  // slower); lets the split kernel be scheduled
  pdl_launch_dependents();
  extern __shared__ __align__(16) float sm[];
  constexpr int kZl = kNb + 4;       // row-major Z (16-byte rows; rows 4 banks apart)
  constexpr int kRl = kStripRows + 4;
  const int tid = threadIdx.x;
  const bool panel = (int)blockIdx.x < panel_strips;
  const int sb = panel ? (int)blockIdx.x : (int)blockIdx.x - panel_strips;
  float* Zs = sm;                    // 128 x kZl
  float* Ss = sm + kNb * kZl;        // panel: B rows (i, m), 32 x kZl; row: R (m, c), 128 x kRl
  const float* zsrc = Xw + j0 * ld + j0;
  float acc[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = 0.0f;
#pragma unroll 16
  for (int e = tid; e < kNb * kNb / 4; e += kStripThreads) {
    const int r = e >> 5, c = (e & 31) * 4;
    *reinterpret_cast<float4*>(Zs + r * kZl + c) = *reinterpret_cast<const float4*>(zsrc + r * ld + c);
  }
  // Both products run over m in order, four m per step: 16-byte loads of four consecutive m
  // (the same address across a warp where the operand is shared: a broadcast).
  if (panel) {
    const int64_t row0 = r_first + (int64_t)sb * kStripRows;
#pragma unroll 4
    for (int e = tid; e < kStripRows * kNb / 4; e += kStripThreads) {
      const int i = e >> 5, m = (e & 31) * 4;
      *reinterpret_cast<float4*>(Ss + i * kZl + m) = *reinterpret_cast<const float4*>(Bw + (row0 + i) * ld + j0 + m);
    }
    __syncthreads();
    // outputs 32 rows x 128 columns: rows 4 ty .. +3, columns tx + 32 k (k < 4); Z's rows
    // tx + 32 k are read four m at a time (lanes 4 banks apart: four wavefronts per load)
    const int ty = tid >> 5, tx = tid & 31;
#pragma unroll 2
    for (int m = 0; m < kNb; m += 4) {
      float4 bv[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) bv[k] = *reinterpret_cast<const float4*>(Zs + (tx + 32 * k) * kZl + m);
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const float4 av = *reinterpret_cast<const float4*>(Ss + (4 * ty + a) * kZl + m);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          acc[a][k] = __fmaf_rn(av.x, bv[k].x, acc[a][k]);
          acc[a][k] = __fmaf_rn(av.y, bv[k].y, acc[a][k]);
          acc[a][k] = __fmaf_rn(av.z, bv[k].z, acc[a][k]);
          acc[a][k] = __fmaf_rn(av.w, bv[k].w, acc[a][k]);
        }
      }
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int k = 0; k < 4; ++k) P[((int64_t)sb * kStripRows + 4 * ty + a) * kNb + tx + 32 * k] = acc[a][k];
  } else {
    const int64_t col0 = (int64_t)sb * kStripRows;
#pragma unroll 4
    for (int e = tid; e < kNb * kStripRows / 4; e += kStripThreads) {
      const int m = e >> 3, c = (e & 7) * 4;
      *reinterpret_cast<float4*>(Ss + m * kRl + c) = *reinterpret_cast<const float4*>(Xw + (j0 + m) * ld + col0 + c);
    }
    __syncthreads();
    // outputs 128 rows x 32 columns: rows 4 ty .. +3, columns 4 tx .. +3
    const int ty = tid >> 3, tx = tid & 7;
#pragma unroll 2
    for (int m = 0; m < kNb; m += 4) {
      float4 av[4], bv[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) av[a] = *reinterpret_cast<const float4*>(Zs + (4 * ty + a) * kZl + m);
#pragma unroll
      for (int q = 0; q < 4; ++q) bv[q] = *reinterpret_cast<const float4*>(Ss + (m + q) * kRl + 4 * tx);
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const float am[4] = {av[a].x, av[a].y, av[a].z, av[a].w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          acc[a][0] = __fmaf_rn(am[q], bv[q].x, acc[a][0]);
          acc[a][1] = __fmaf_rn(am[q], bv[q].y, acc[a][1]);
          acc[a][2] = __fmaf_rn(am[q], bv[q].z, acc[a][2]);
          acc[a][3] = __fmaf_rn(am[q], bv[q].w, acc[a][3]);
        }
      }
    }
    // R was staged into shared memory before the first barrier, so the outputs may overwrite it
#pragma unroll
    for (int a = 0; a < 4; ++a)
      *reinterpret_cast<float4*>(Xw + (j0 + 4 * ty + a) * ld + col0 + 4 * tx) =
          make_float4(acc[a][0], acc[a][1], acc[a][2], acc[a][3]);
  }
}

// ---------------------------------------------------------------- three-way bf16 splits
// x = x1 + x2 + x3 with bf16 parts, each difference exact in fp32: the parts carry x to
// about 2^-24 relative.
__device__ __forceinline__ void split3(float x, uint16_t (&p)[3]) {
  const __nv_bfloat16 a = __float2bfloat16_rn(x);
  const float r1 = __fsub_rn(x, __bfloat162float(a));
  const __nv_bfloat16 b = __float2bfloat16_rn(r1);
  const float r2 = __fsub_rn(r1, __bfloat162float(b));
  const __nv_bfloat16 c = __float2bfloat16_rn(r2);
  p[0] = __bfloat16_as_ushort(a);
  p[1] = __bfloat16_as_ushort(b);
  p[2] = __bfloat16_as_ushort(c);
}

// Both split operands of a step's update in one launch.  Blocks [0, panel_blocks): the panel
// P [rows, 128] (fp32) into its place in Bw (rows r_first.., columns j0..) and as the two
// operands of the updates: An = [-P1 | -P1 | -P2 | -P1 | -P2 | -P3] and
// Bp = [P1 | P2 | P1 | P3 | P2 | P1] (rows of 6 * 128 bf16), so that An Bp^T = -P P^T to fp32
// accuracy (the six products E1U1, E1U2, E2U1, E1U3, E2U2, E3U1).  The blocks after them: the
// inverse's row block j (Xw rows j0..j0+127, columns 0..cols-1) transposed, as the B operand
// of the R update: Bx[c] = [X1 | X2 | X1 | X3 | X2 | X1] of column c of the row block, one
// 32 x 32 tile per block (4 tiles per 32 columns) through shared memory (coalesced reads
// along c, writes along the row index).  The two parts are independent.
__global__ void __launch_bounds__(256) factor_split_kernel(const float* __restrict__ P, int64_t rows,
                                                           float* __restrict__ Bw, const float* __restrict__ Xw,
                                                           int64_t ld, int64_t r_first, int64_t j0, int64_t cols,
                                                           int panel_blocks, uint16_t* __restrict__ An,
                                                           uint16_t* __restrict__ Bp, uint16_t* __restrict__ Bx) {
  pdl_launch_dependents();
  pdl_wait_primary();  // the strips' panel and row (programmatic dependent launch)
  if ((int)blockIdx.x < panel_blocks) {
    const int64_t total = rows * kNb;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (int64_t)panel_blocks * blockDim.x) {
      const int64_t i = e >> 7;
      const int k = (int)(e & (kNb - 1));
      const float x = P[e];
      Bw[(r_first + i) * ld + j0 + k] = x;
      uint16_t p[3], q[3];
      split3(x, p);
      split3(-x, q);
      uint16_t* a = An + i * kSplitK + k;
      uint16_t* b = Bp + i * kSplitK + k;
      a[0] = q[0]; a[kNb] = q[0]; a[2 * kNb] = q[1]; a[3 * kNb] = q[0]; a[4 * kNb] = q[1]; a[5 * kNb] = q[2];
      b[0] = p[0]; b[kNb] = p[1]; b[2 * kNb] = p[0]; b[3 * kNb] = p[2]; b[4 * kNb] = p[1]; b[5 * kNb] = p[0];
    }
    return;
  }
  __shared__ float t[32][33];
  const int rb = (int)blockIdx.x - panel_blocks;
  const int64_t c0 = (int64_t)(rb >> 2) * 32;
  const int m0 = (rb & 3) * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  for (int mm = ty; mm < 32; mm += 8) t[mm][tx] = c0 + tx < cols ? Xw[(j0 + m0 + mm) * ld + c0 + tx] : 0.0f;
  __syncthreads();
  for (int cc = ty; cc < 32; cc += 8) {
    const int64_t c = c0 + cc;
    if (c >= cols) continue;
    uint16_t p[3];
    split3(t[tx][cc], p);
    uint16_t* b = Bx + c * kSplitK + m0 + tx;
    b[0] = p[0]; b[kNb] = p[1]; b[2 * kNb] = p[0]; b[3 * kNb] = p[2]; b[4 * kNb] = p[1]; b[5 * kNb] = p[0];
  }
}

inline int64_t round256(int64_t bytes) { return (bytes + 255) / 256 * 256; }

// The diagonal block, split and update kernels are launched with programmatic dependent launch:
// the kernel before each lets it be scheduled as soon as it starts, and it waits for that
// kernel's writes before its first read, so those launches do not each wait out a launch's
// latency (n = 4096: 1.92 -> 1.88 ms).  The strips are launched in stream order: scheduled
// early, beside the diagonal block, they made the sweep 4 % slower.
template <typename... KArgs, typename... Args>
cudaError_t launch_chained(void (*kernel)(KArgs...), unsigned grid, unsigned block, int smem, cudaStream_t stream,
                           Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid, 1, 1);
  cfg.blockDim = dim3(block, 1, 1);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaError_t err = cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
  if (err != cudaSuccess) return err;
  return cudaGetLastError();
}

}  // namespace

int64_t gptq_factor_padded(int64_t n) { return (n + kNb - 1) / kNb * kNb; }

// W2 = [B | X] (n_pad x 2 n_pad fp32), the panel (n_pad x 128 fp32) and the split operands (A: n_pad x 768 bf16; B: [L_:j ; X_j,:], n_pad x 768 bf16), each region
// 256-byte aligned.
size_t gptq_factor_workspace(int64_t n) {
  const int64_t np = gptq_factor_padded(n);
  return (size_t)(round256(2 * np * np * 4) + round256(np * kNb * 4) + 2 * round256(np * kSplitK * 2));
}

cudaError_t launch_gptq_factor(const float* H, int64_t n, int64_t ld_h, float damp, float* Uo, uint8_t* dead,
                               int32_t* info, void* workspace, cudaStream_t stream) {
  DeviceInfo dinfo;
  cudaError_t err = current_device_info(&dinfo);
  if (err != cudaSuccess) return err;
  const int64_t np = gptq_factor_padded(n);
  const int64_t ld = 2 * np;
  uint8_t* base = static_cast<uint8_t*>(workspace);
  float* Bw = reinterpret_cast<float*>(base);  // left half of W2; X = Bw + np
  float* Xw = Bw + np;
  float* P = reinterpret_cast<float*>(base + round256(2 * np * np * 4));
  uint8_t* ops = base + round256(2 * np * np * 4) + round256(np * kNb * 4);
  uint16_t* An = reinterpret_cast<uint16_t*>(ops);
  uint16_t* Bo = reinterpret_cast<uint16_t*>(ops + round256(np * kSplitK * 2));

  if ((err = cudaMemsetAsync(info, 0, 3 * sizeof(int32_t), stream)) != cudaSuccess) return err;
  // the damped diagonal, in the panel's buffer until the sweep writes the first panel
  float* dd = P;
  damp_diagonal_kernel<<<1, 1024, 0, stream>>>(H, n, ld_h, damp, dead, dd);
  if ((err = cudaGetLastError()) != cudaSuccess) return err;
  reverse_pad_kernel<<<dim3((unsigned)(np / 32), (unsigned)(np / 32)), 256, 0, stream>>>(H, n, ld_h, dd, np, Bw);
  if ((err = cudaGetLastError()) != cudaSuccess) return err;
  if ((err = ensure_dynamic_smem(reinterpret_cast<const void*>(factor_diag_kernel), kDiagSmemBytes)) != cudaSuccess)
    return err;
  if ((err = ensure_dynamic_smem(reinterpret_cast<const void*>(factor_strip_kernel), kStripSmemBytes)) != cudaSuccess)
    return err;

  const int64_t nblk = np / kNb;
  for (int64_t jb = 0; jb < nblk; ++jb) {
    const int64_t j0 = jb * kNb;
    const int64_t r_first = j0 + kNb;          // first row below the diagonal block
    const int64_t rows = np - r_first;         // rows of the panel
    if ((err = launch_chained(factor_diag_kernel, 1, kDiagThreads, kDiagSmemBytes, stream, (const float*)Bw, ld, j0,
                              Xw, info)) != cudaSuccess)
      return err;
    const int panel_strips = (int)(rows / kStripRows);
    const int row_strips = (int)(j0 / kStripRows);
    if (panel_strips + row_strips > 0) {
      factor_strip_kernel<<<(unsigned)(panel_strips + row_strips), kStripThreads, kStripSmemBytes, stream>>>(
          Bw, Xw, ld, j0, P, panel_strips, r_first);
      if ((err = cudaGetLastError()) != cudaSuccess) return err;
    }
    if (rows == 0) break;
    const int sblocks = (int)std::max<int64_t>(1, std::min<int64_t>((rows * kNb + 255) / 256,
                                                                    (int64_t)dinfo.sm_count * 8));
    const int64_t xcols = j0 + kNb;            // columns of the inverse's row block j, diagonal included
    const int64_t rblocks = (xcols + 31) / 32 * (kNb / 32);
    if ((err = launch_chained(factor_split_kernel, (unsigned)(sblocks + rblocks), 256, 0, stream, (const float*)P, rows,
                              Bw, (const float*)Xw, ld, r_first, j0, xcols, sblocks, An, Bo, Bo + rows * kSplitK)) !=
        cudaSuccess)
      return err;
    // rows below the diagonal block, columns r_first .. np + xcols of W2 (rows + xcols = np):
    // the trailing square and the inverse's rows, -= L_:j [L_:j ; X_j,:]^T
    if ((err = launch_gemm_accumulate(An, Bo, rows, rows + xcols, kSplitK, Bw + r_first * ld + r_first, ld, stream,
                                      true)) != cudaSuccess)
      return err;
  }
  // 256 columns per block, rows strided over 512 blocks (several independent rows per thread)
  reverse_out_kernel<<<dim3((unsigned)((n + 255) / 256), (unsigned)std::min<int64_t>(n, 512)), 256, 0, stream>>>(
      Xw, ld, n, Uo);
  return cudaGetLastError();
}

}  // namespace hscale
