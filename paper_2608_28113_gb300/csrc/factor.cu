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
// [n_pad, 2 n_pad] buffer.  The sweep takes 128-wide block columns j = 0, 1, ...
// (right-looking), two kernels each:
//   panel    L_ij = B_ij Z_jj^T (i > j; Z_jj = L_jj^-1) and the inverse's row X_jc = Z_jj R_jc
//            (c < j), on CUDA cores, written as three-way bf16 splits (factor_panel_kernel);
//   update   B_ik -= L_ij L_kj^T over the trailing square's lower triangle, and
//            R_ic -= L_ij X_jc for i > j, c <= j, on the tensor cores with fp32-level accuracy;
//            one CTA of it takes the next diagonal block, B_j+1,j+1 = L L^T, factors it in
//            shared memory and writes its inverse Z_j+1 into the inverse's diagonal block
//            (update.cu, factor_block.cuh).
// So the serial part of step j + 1 runs beside the update of step j, and the chain per step is
// one panel, one tile of the update and one diagonal block.  The first diagonal block has a kernel of its
// own (factor_diag_kernel).
// One GB300, n = 4096: 0.80 ms in a graph (1.755 ms with the diagonal block, panel, splits and update one
// after another), of which about 31 steps of 23 us: diagonal block 11, its tile 4, panel 4,
// launches and hand-over the rest.
// X = L^-1 is built alongside: row blocks below the diagonal accumulate
// R_ic = -sum_k L_ik X_kc as the sweep passes, and X_ic = Z_ii R_ic once row block i is reached.
// A last kernel writes U_ij = X_{n-1-i, n-1-j}.
//
// A pivot that is not positive (the damped matrix is then not positive definite) is recorded
// in info[0] as its 1-based order in B and replaced by 1, so the sweep ends with finite values;
// U is then unspecified.
#include <cuda_bf16.h>

#include <algorithm>

#include "chained_launch.h"
#include "factor_block.cuh"
#include "hscale_internal.h"
#include "split3.cuh"
#include "tma.cuh"

namespace hscale {
namespace {

constexpr int kPanelRows = 32;            // rows (or columns) of one panel block
constexpr int kPanelThreads = 256;
constexpr int kPanelSmemBytes = (kNb * kLd + kNb * (kPanelRows + 4)) * 4;

// ---------------------------------------------------------------- set-up
// One block: info cleared, dead channels (H_jj = 0) and the damped diagonal dd_j = d_j + damp * mean(d),
// d_j = H_jj, or 1 for a dead channel (fp32; the mean in fp64).
__global__ void __launch_bounds__(1024) damp_diagonal_kernel(const float* __restrict__ H, int64_t n, int64_t ld_h,
                                                             float damp, uint8_t* __restrict__ dead,
                                                             float* __restrict__ dd, int32_t* __restrict__ info) {
  if (threadIdx.x < 3) info[threadIdx.x] = 0;
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

// W2 [n_pad, 2 n_pad]: the left half B_ij = A_{n-1-i, n-1-j} for i, j < n on and below the 128-block
// diagonal, A the damped H (read from H's upper triangle, row stride ld_h, and the damped diagonal
// dd), the identity beyond n; the right half (X) zero where the sweep accumulates into it,
// strictly below the 128-block diagonal.  Nothing reads either half above it (so half of both is
// never written: n = 4096 43 -> 25.6 us).  One 32 x 32 tile of each half per block.
// Every read and write runs along a row: a tile below the diagonal reads H's rows (reversed), one above it (within a diagonal 128-block) reads the
// mirrored tile of H and transposes it in shared memory, and a tile on the diagonal reads the
// entries on and below it and takes the rest from its own transpose.
__global__ void __launch_bounds__(256) reverse_pad_kernel(const float* __restrict__ H, int64_t n, int64_t ld_h,
                                                          const float* __restrict__ dd, int64_t n_pad,
                                                          float* __restrict__ W2) {
  __shared__ float t[32][33];
  const int bi = (int)blockIdx.y, bj = (int)blockIdx.x;
  if (bj / (kNb / 32) > bi / (kNb / 32)) return;
  const int64_t i0 = 32 * (int64_t)bi, j0 = 32 * (int64_t)bj, ld = 2 * n_pad;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  float v[4];
  if (bi < bj) {
    // B_ij = A_{n-1-j, n-1-i}: t[jj][ii]
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int64_t j = j0 + ty + 8 * k, i = i0 + tx;
      v[k] = (i < n && j < n) ? H[(n - 1 - j) * ld_h + (n - 1 - i)] : 0.0f;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) t[ty + 8 * k][tx] = v[k];
    __syncthreads();
    for (int ii = ty; ii < 32; ii += 8) W2[(i0 + ii) * ld + j0 + tx] = t[tx][ii];  // i < j: 0 beyond n
  } else {
    // B_ij = A_{n-1-i, n-1-j} for i >= j: t[ii][jj]
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int64_t i = i0 + ty + 8 * k, j = j0 + tx;
      v[k] = (i < n && j < n && i >= j) ? H[(n - 1 - i) * ld_h + (n - 1 - j)] : 0.0f;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) t[ty + 8 * k][tx] = v[k];
    __syncthreads();
    for (int ii = ty; ii < 32; ii += 8) {
      const int64_t i = i0 + ii, j = j0 + tx;
      float x;
      if (i < n && j < n)
        x = i == j ? dd[n - 1 - i] : (i > j ? t[ii][tx] : t[tx][ii]);
      else
        x = i == j ? 1.0f : 0.0f;
      W2[i * ld + j] = x;
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
// The diagonal block at (j0, j0) of Bw: Z_jj into Xw's diagonal block (zeros above the
// diagonal).  One CTA.  Only the lower triangle of the block is used.
__global__ void __launch_bounds__(kDiagThreads, 1)
factor_diag_kernel(const float* Bw, int64_t ld, int64_t j0, float* Xw, int32_t* info) {
  extern __shared__ __align__(16) uint8_t dynamic_smem[];
  float* S = reinterpret_cast<float*>(dynamic_smem);  // [128][kLd] the block
  const int tid = threadIdx.x;

  // programmatic dependent launch on both sides
  pdl_launch_dependents();
  pdl_wait_primary();
  const float* blk = Bw + j0 * ld + j0;
  // independent 16-byte loads per thread in flight
#pragma unroll
  for (int t = 0; t < kNb * kNb / 4 / kDiagThreads; ++t) {
    const int e = tid + t * kDiagThreads;
    const int r = e >> 5, c = (e & 31) * 4;
    *reinterpret_cast<float4*>(S + r * kLd + c) = *reinterpret_cast<const float4*>(blk + r * ld + c);
  }
  __syncthreads();
  factor_block128(0, Xw + j0 * ld + j0, ld, info, (int32_t)j0);
}

// ---------------------------------------------------------------- panel (CUDA cores)
// What step j's update needs, 32 rows or columns a block, written as the update's split operand
// Bo (rows of three 128-wide bf16 parts, split3):
//   blocks [0, panel)            rows of the panel below the diagonal block,
//                                L_ij = B_ij Z_jj^T: row i - r_first of Bo;
//   blocks [panel, panel + row)  columns of the inverse's row j, X_jc = Z_jj R_jc (c < j0), in
//                                place in Xw, and transposed as row rows + c of Bo;
//   four blocks                  the columns of Z_jj itself, rows rows + j0 .. of Bo.
// L_ij itself is not stored: the rest of the sweep needs only its splits.
// Z = Z_jj is Xw's diagonal block, lower triangular: the sums stop at each 32 columns' (16
// rows') last non-zero term.  256 threads, 4 x 4 outputs each over K = 128 from shared memory,
// four m per 16-byte read: a warp computes 16 rows x 32 columns, its lanes 4 x 8 such tiles, so
// that every read has neighbours (lanes i and i ^ 1, or i ^ 2) that share the address and
// takes two cycles of the SM, and both operands' rows are dealt so that no bank is met twice
// (Z's rows are permuted in shared memory: row 32 Q + 4 a + q at 32 Q + 8 q + a).  Warps w and
// w + 4, on one scheduler, take a short and a long part of the triangle.  The sums run over m
// in order.
// One GB300, n = 4096: this one kernel takes the place of two (products, then splits), whose
// launches took 8.2 and 6.1 us a step.
__global__ void __launch_bounds__(kPanelThreads)
factor_panel_kernel(const float* Bw, float* Xw, int64_t ld, int64_t j0, int64_t r_first, int64_t rows, int panel_blocks,
                    int row_blocks, uint16_t* Bo) {
  extern __shared__ __align__(16) uint8_t dynamic_smem[];
  float* sm = reinterpret_cast<float*>(dynamic_smem);
  constexpr int kRl = kPanelRows + 4;
  float* Zs = sm;             // 128 x kLd, rows permuted
  float* Ss = sm + kNb * kLd; // panel: B rows, 32 x kLd; row: R (m, c), 128 x kRl
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // lane tile (h, cl) of 4 x 8: h leaves out lane bit 0 and cl lane bit 1
  const int h = ((lane >> 1) & 1) + ((lane >> 3) & 2), cl = (lane & 1) + ((lane >> 1) & 6);
  const int kind = (int)blockIdx.x < panel_blocks ? 0 : ((int)blockIdx.x < panel_blocks + row_blocks ? 1 : 2);
  const int sb = (int)blockIdx.x - (kind == 0 ? 0 : (kind == 1 ? panel_blocks : panel_blocks + row_blocks));

  // programmatic dependent launch on both sides
  pdl_launch_dependents();
  pdl_wait_primary();

  const float* zsrc = Xw + j0 * ld + j0;
#pragma unroll
  for (int t = 0; t < kNb * kNb / 4 / kPanelThreads; ++t) {
    const int e = tid + t * kPanelThreads;
    const int r = e >> 5, c = (e & 31) * 4;
    const int pos = (r & ~31) + 8 * (r & 3) + ((r & 31) >> 2);
    *reinterpret_cast<float4*>(Zs + pos * kLd + c) = *reinterpret_cast<const float4*>(zsrc + r * ld + c);
  }
  float acc[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = 0.0f;

  if (kind == 0) {
    const int64_t row0 = r_first + (int64_t)sb * kPanelRows;
#pragma unroll
    for (int t = 0; t < kPanelRows * kNb / 4 / kPanelThreads; ++t) {
      const int e = tid + t * kPanelThreads;
      const int i = e >> 5, m = (e & 31) * 4;
      *reinterpret_cast<float4*>(Ss + i * kLd + m) = *reinterpret_cast<const float4*>(Bw + (row0 + i) * ld + j0 + m);
    }
    __syncthreads();
    // rows 16 (warp / 4) + h + 4 r, columns 32 Q + 4 cl + q, m < 32 (Q + 1)
    const int Q = warp < 4 ? warp : 7 - warp, r0 = 16 * (warp >> 2) + h;
    const float* As = Ss + r0 * kLd;
    const float* Bs = Zs + (32 * Q + cl) * kLd;
#pragma unroll 2
    for (int m = 0; m < 32 * (Q + 1); m += 4) {
      float4 bv[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) bv[q] = *reinterpret_cast<const float4*>(Bs + 8 * q * kLd + m);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const float4 av = *reinterpret_cast<const float4*>(As + 4 * r * kLd + m);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          acc[r][q] = __fmaf_rn(av.x, bv[q].x, acc[r][q]);
          acc[r][q] = __fmaf_rn(av.y, bv[q].y, acc[r][q]);
          acc[r][q] = __fmaf_rn(av.z, bv[q].z, acc[r][q]);
          acc[r][q] = __fmaf_rn(av.w, bv[q].w, acc[r][q]);
        }
      }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r)
      store_split3x4(Bo + ((int64_t)sb * kPanelRows + r0 + 4 * r) * (3 * kNb) + 32 * Q + 4 * cl, kNb, acc[r]);
    return;
  }

  // rows 16 W + 4 h + r, columns 4 cl + q of this block's 32, m < 16 (W + 1)
  const int W = warp < 4 ? warp : 11 - warp, r0 = 16 * W + 4 * h;
  const float* As = Zs + ((r0 & ~31) + ((r0 & 31) >> 2)) * kLd;  // row r0 + r: 8 r rows further
  const int64_t col0 = (int64_t)sb * kPanelRows + (kind == 2 ? j0 : 0);
  if (kind == 1) {
#pragma unroll
    for (int t = 0; t < kPanelRows * kNb / 4 / kPanelThreads; ++t) {
      const int e = tid + t * kPanelThreads;
      const int m = e >> 3, c = (e & 7) * 4;
      *reinterpret_cast<float4*>(Ss + m * kRl + c) = *reinterpret_cast<const float4*>(Xw + (j0 + m) * ld + col0 + c);
    }
    __syncthreads();
#pragma unroll 2
    for (int m = 0; m < 16 * (W + 1); m += 4) {
      float4 bv[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) bv[q] = *reinterpret_cast<const float4*>(Ss + (m + q) * kRl + 4 * cl);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const float4 v = *reinterpret_cast<const float4*>(As + 8 * r * kLd + m);
        const float av[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          acc[r][0] = __fmaf_rn(av[q], bv[q].x, acc[r][0]);
          acc[r][1] = __fmaf_rn(av[q], bv[q].y, acc[r][1]);
          acc[r][2] = __fmaf_rn(av[q], bv[q].z, acc[r][2]);
          acc[r][3] = __fmaf_rn(av[q], bv[q].w, acc[r][3]);
        }
      }
    }
    // R was staged into shared memory before the barrier, so the outputs may overwrite it
#pragma unroll
    for (int r = 0; r < 4; ++r)
      *reinterpret_cast<float4*>(Xw + (j0 + r0 + r) * ld + col0 + 4 * cl) =
          make_float4(acc[r][0], acc[r][1], acc[r][2], acc[r][3]);
  } else {
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[r][q] = As[8 * r * kLd + (col0 - j0) + 4 * cl + q];
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float v[4] = {acc[0][q], acc[1][q], acc[2][q], acc[3][q]};
    store_split3x4(Bo + (rows + col0 + 4 * cl + q) * (3 * kNb) + r0, kNb, v);
  }
}

inline int64_t round256(int64_t bytes) { return (bytes + 255) / 256 * 256; }

}  // namespace

int64_t gptq_factor_padded(int64_t n) { return (n + kNb - 1) / kNb * kNb; }

// W2 = [B | X] (n_pad x 2 n_pad fp32), the damped diagonal (in a region of n_pad x 128 floats) and
// the update's split operand [L_:j ; X_j,:^T] (n_pad rows of 3 x 128 bf16, in a region of four
// times that); the regions keep the sizes that callers' workspaces were made for.
size_t gptq_factor_workspace(int64_t n) {
  const int64_t np = gptq_factor_padded(n);
  return (size_t)(round256(2 * np * np * 4) + round256(np * kNb * 4) + 2 * round256(np * 6 * kNb * 2));
}

cudaError_t launch_gptq_factor(const float* H, int64_t n, int64_t ld_h, float damp, float* Uo, uint8_t* dead,
                               int32_t* info, void* workspace, cudaStream_t stream) {
  cudaError_t err;
  const int64_t np = gptq_factor_padded(n);
  const int64_t ld = 2 * np;
  uint8_t* base = static_cast<uint8_t*>(workspace);
  float* Bw = reinterpret_cast<float*>(base);  // left half of W2; X = Bw + np
  float* Xw = Bw + np;
  float* dd = reinterpret_cast<float*>(base + round256(2 * np * np * 4));
  uint16_t* Bo = reinterpret_cast<uint16_t*>(base + round256(2 * np * np * 4) + round256(np * kNb * 4));

  damp_diagonal_kernel<<<1, 1024, 0, stream>>>(H, n, ld_h, damp, dead, dd, info);
  if ((err = cudaGetLastError()) != cudaSuccess) return err;
  reverse_pad_kernel<<<dim3((unsigned)(np / 32), (unsigned)(np / 32)), 256, 0, stream>>>(H, n, ld_h, dd, np, Bw);
  if ((err = cudaGetLastError()) != cudaSuccess) return err;
  if ((err = ensure_dynamic_smem(reinterpret_cast<const void*>(factor_diag_kernel), kDiagSmemBytes)) != cudaSuccess)
    return err;
  if ((err = ensure_dynamic_smem(reinterpret_cast<const void*>(factor_panel_kernel), kPanelSmemBytes)) != cudaSuccess)
    return err;

  // the first diagonal block; every later one is factored by the update before it
  if ((err = launch_chained(factor_diag_kernel, dim3(1), kDiagThreads, kDiagSmemBytes, stream, (const float*)Bw, ld,
                            (int64_t)0, Xw, info)) != cudaSuccess)
    return err;
  const int64_t nblk = np / kNb;
  for (int64_t jb = 0; jb < nblk; ++jb) {
    const int64_t j0 = jb * kNb;
    const int64_t r_first = j0 + kNb;          // first row below the diagonal block
    const int64_t rows = np - r_first;         // rows of the panel
    // the last block column has no panel: only the inverse's row
    const int panel_blocks = (int)(rows / kPanelRows), row_blocks = (int)(j0 / kPanelRows);
    const int blocks = panel_blocks + row_blocks + (rows > 0 ? kNb / kPanelRows : 0);
    if (blocks > 0 && (err = launch_chained(factor_panel_kernel, dim3((unsigned)blocks), kPanelThreads, kPanelSmemBytes,
                                            stream, (const float*)Bw, Xw, ld, j0, r_first, rows, panel_blocks,
                                            row_blocks, Bo)) != cudaSuccess)
      return err;
    if (rows == 0) break;
    // the rows below the diagonal block, -= L_:j [L_:j ; X_j,:]^T, and the next diagonal block
    if ((err = launch_factor_update(Bo, rows, j0 + kNb, Bw + r_first * ld + r_first, Xw + r_first * ld, ld,
                                    (int32_t)r_first, info, stream)) != cudaSuccess)
      return err;
  }
  // 256 columns per block, rows strided over 512 blocks (several independent rows per thread)
  reverse_out_kernel<<<dim3((unsigned)((n + 255) / 256), (unsigned)std::min<int64_t>(n, 512)), 256, 0, stream>>>(
      Xw, ld, n, Uo);
  return cudaGetLastError();
}

}  // namespace hscale
