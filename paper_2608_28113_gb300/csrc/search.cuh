// search.cuh -- the per-group pieces of the H-Scale search (Algorithm 1), shared by the search
// kernels (scales.cu, whose file comment has the error bounds) and the quantizer of GPTQ's block
// loop (gptq.cu).
#pragma once
#include <cstdint>

#include "hscale_device.cuh"

namespace hscale {

constexpr float kInf = __builtin_huge_valf();

// a_j keeps the sign of w_j.  Every score is even in a_j (round-to-nearest-even and
// saturation are symmetric, and only squares of residuals enter), so the search pays
// nothing for the sign, and the pack converts the signed quotients directly.
struct Group {
  float2 a[8];     // w * 2^-K, elements (2i, 2i+1)
};

// The group's 16 bf16 values, given as two 16-byte words (element 2i in the low half of
// word i), unpacked and scaled.
__device__ __forceinline__ void unpack_group(const uint4& p, const uint4& q, float pw, Group& G) {
  const uint32_t wb[8] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w};
#pragma unroll
  for (int i = 0; i < 8; ++i)
    G.a[i] = __fmul2_rn(make_float2(bf16_lo(wb[i]), bf16_hi(wb[i])), make_float2(pw, pw));
}

// The group whose 16 bf16 values start at wg (16-byte aligned).
__device__ __forceinline__ void load_group_at(const uint4* wg, float pw, Group& G) {
  unpack_group(ld_stream_v4(wg), ld_stream_v4(wg + 1), pw, G);
}

// Per-block table of the candidate constants of every E4M3 code c (1..126), filled once
// per CTA and stored pre-splatted for the packed arithmetic: x = y = s'^2 and
// z = w = 1 / s' (correctly rounded), with s' = l(c) * sgk in [2^-21, 2^-2], so both are
// normal numbers.  One 16-byte shared load per candidate replaces a decode, a multiply
// and a reciprocal on the candidate's critical path.
__device__ __forceinline__ float4 candidate_constants(uint32_t c, float sgk) {
  const float sp = __fmul_rn(e4m3_mag(c), sgk);
  const float s2 = __fmul_rn(sp, sp), inv = c ? __frcp_rn(sp) : 0.0f;
  return make_float4(s2, s2, inv, inv);
}

// q - y for a pair of quotients y (real units): q = RNE_sat(y) by the hardware E2M1
// conversion, back to f16 (exact), and one mixed f16 - f32 subtract per element.
__device__ __forceinline__ float2 e2m1_residual2(float2 y) {
  float d0, d1;
  asm("{\n\t.reg .b8 c;\n\t.reg .b32 q;\n\t.reg .f16 lo, hi;\n\t"
      "cvt.rn.satfinite.e2m1x2.f32 c, %3, %2;\n\t"
      "cvt.rn.f16x2.e2m1x2 q, c;\n\t"
      "mov.b32 {lo, hi}, q;\n\t"
      "sub.rn.f32.f16 %0, lo, %2;\n\t"
      "sub.rn.f32.f16 %1, hi, %3;\n\t}"
      : "=f"(d0), "=f"(d1)
      : "f"(y.x), "f"(y.y));
  return make_float2(d0, d1);
}

// Fast score of one candidate from its table entry t (see the file comment): per pair of
// elements one packed multiply for the quotients, the hardware rounding and residuals,
// a packed square and a packed FMA into the h-weighted sum (one chain per half of the
// pair: the candidates scored side by side give the independent work); then the halves'
// sum and one multiply by s'^2.
__device__ __forceinline__ float fast_score(const Group& G, const float2 (&hv2)[8], float4 t) {
  const float2 inv2 = make_float2(t.z, t.w);
  float2 acc = make_float2(0.f, 0.f);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float2 d = e2m1_residual2(__fmul2_rn(G.a[i], inv2));
    acc = __ffma2_rn(hv2[i], __fmul2_rn(d, d), acc);
  }
  return __fmul_rn(t.x, __fadd_rn(acc.x, acc.y));
}

// Running best (e1, best) and runner-up e2 (e1 <= e2); branch-free: a select and three
// min/max.  A tie with the best makes e2 = e1 (the margin test then fails); NaN scores
// are ignored.
__device__ __forceinline__ void keep_best(float e, int c, float& e1, float& e2, int& best) {
  best = e < e1 ? c : best;
  e2 = fminf(e2, fmaxf(e1, e));
  e1 = fminf(e1, e);
}

// Scores the codes [a, b) two at a time (independent chains interleave).
__device__ __forceinline__ void score_range(const Group& G, const float2 (&hv2)[8],
                                            const float4* tab, int a, int b, float& e1, float& e2,
                                            int& best) {
  int c = a;
  for (; c + 1 < b; c += 2) {
    const float4 t0 = tab[c], t1 = tab[c + 1];
    const float ea = fast_score(G, hv2, t0);
    const float eb = fast_score(G, hv2, t1);
    keep_best(ea, c, e1, e2, best);
    keep_best(eb, c + 1, e1, e2, best);
  }
  if (c < b) keep_best(fast_score(G, hv2, tab[c]), c, e1, e2, best);
}

// Upper bound of A = sum_j h_j a_j^2, the scale of the fast-score error bound:
// (sum_j h_j) * max_j a_j^2.  Two multiplies instead of a pass over the group; a larger A
// only widens the margin (the rounding of the bound, a relative 2^-20 at most, is far
// inside the margin's 2x slack).
__device__ __forceinline__ float energy_bound(float hsum, float amax_k) {
  return __fmul_rn(hsum, __fmul_rn(amax_k, amax_k));
}

// A = sum_j h_j a_j^2 itself (scaled domain), for the search's margin test.  (sum h) amax^2
// can exceed it many times over (one large weight, or h concentrated on small ones), and
// the margin's dominant term grows with sqrt(A), so the tighter value sends several times
// fewer groups to the exact rescoring.  The fp32 sum of non-negative terms is within a
// relative 12 * 2^-24 of A; the factor 1 + 2^-19 makes the result an upper bound.
__device__ __forceinline__ float group_energy(const Group& G, const float2 (&hv2)[8]) {
  float2 acc = __fmul2_rn(hv2[0], __fmul2_rn(G.a[0], G.a[0]));
#pragma unroll
  for (int i = 1; i < 8; ++i) acc = __ffma2_rn(hv2[i], __fmul2_rn(G.a[i], G.a[i]), acc);
  return __fmul_rn(__fadd_rn(acc.x, acc.y), 1.0f + 0x1p-19f);
}

// A sufficient condition for fast_winner_certain that costs six operations: a relative
// gap above 2^-9 with A <= 2^18 E2 (A_bound any upper bound of A, here (sum h) amax^2)
// gives a margin of at most (2^-18 + 2^-19 2^9 + 2^-35 2^18) E2 < 2^-9 E2, and
// E2 >= 2^-36 A.  (The fp32 rounding of the gap and of A_bound is a few units of 2^-24,
// far inside the factor of two between 2^-9 and the margin.)  The scores' error bound
// holds for results in the normal range, so a runner-up below 2^-100 is left to
// fast_winner_certain (which sends denormal ones to the exact rescoring); a zero,
// infinite or NaN runner-up fails it too.
__device__ __forceinline__ bool fast_winner_clear(float e1, float e2, float A_bound) {
  return e2 >= 0x1p-100f && __fsub_rn(e2, e1) > __fmul_rn(0x1p-9f, e2) && A_bound <= __fmul_rn(0x1p18f, e2);
}

// tie rule of the search: smaller error, then smaller |shift|, then smaller shift
__device__ __forceinline__ bool better(float e, int c, float be, int bc, int c0) {
  if (e != be) return e < be;
  const int s = c - c0, bs = bc - c0;
  const int as = s < 0 ? -s : s, abs_ = bs < 0 ? -bs : bs;
  return as < abs_ || (as == abs_ && s < bs);
}

// Exact-decision score of one element under code c (scaled domain, one rounding in the
// residual: q * l is exact and the FMA rounds once).
__device__ __forceinline__ float exact_term(float a_k, float hj, uint32_t c, float sgk) {
  const float l = e4m3_mag(c);
  const float inv = inv_raw_of(__fmul_rn(l, sgk));
  const uint32_t k = e2m1_code(a_k, inv, l, sgk);
  const float ql = __fmul_rn(e2m1_from_raw(k << 22), l);
  const float r = __fmaf_rn(-ql, sgk, a_k);
  return __fmul_rn(hj, __fmul_rn(r, r));
}

// The whole warp rescores one group with exact rounding decisions and returns its winning code
// (in every lane); a_k and hj are element lane & 15 of the group (magnitude, scaled domain) and
// its weight.  Lanes 0-15 take the candidates lo, lo + 2, ..., lanes 16-31 lo + 1, lo + 3, ...
__device__ __forceinline__ int warp_exact_codes(float a_k, float hj, int c0, int lo, int hi, float sgk) {
  const int half = (threadIdx.x & 31) >> 4;
  const unsigned mask = 0xFFFFu << (16 * half);
  float be = kInf;
  int bc = -1;
  // two candidates a step: their chains of shuffles run side by side
  for (int c = lo + half; c <= hi; c += 4) {
    const int c2 = c + 2 <= hi ? c + 2 : c;
    float e = exact_term(a_k, hj, (uint32_t)c, sgk), f = exact_term(a_k, hj, (uint32_t)c2, sgk);
#pragma unroll
    for (int off = 1; off < 16; off <<= 1) {
      const float eo = __shfl_xor_sync(mask, e, off), fo = __shfl_xor_sync(mask, f, off);
      e = __fadd_rn(e, eo);
      f = __fadd_rn(f, fo);
    }
    if (bc < 0 || better(e, c, be, bc, c0)) { be = e; bc = c; }
    if (c2 != c && better(f, c2, be, bc, c0)) { be = f; bc = c2; }
  }
  __syncwarp();
  const float oe = __shfl_xor_sync(0xFFFFFFFFu, be, 16);
  const int oc = __shfl_xor_sync(0xFFFFFFFFu, bc, 16);
  if (oc >= 0 && (bc < 0 || better(oe, oc, be, bc, c0))) { be = oe; bc = oc; }
  return bc;
}

// Is the fast winner (fast score e1) certainly ahead of the runner-up (e2), given the
// energy A = sum_j h_j a_j^2 of the group (or an upper bound of it)?  The test of the file comment, in units of e2
// (no underflow or overflow for 2^-36 A <= e2 <= A-ish):
//   g = (e2 - e1) / e2 - 2^-18 - 2^-35 A / e2 > 2^-19 sqrt(A / e2), tested on squares.
// A zero, denormal or non-finite e2 makes the reciprocal infinite or NaN and g fails.
__device__ __forceinline__ bool fast_winner_certain(float e1, float e2, float A) {
  const float r = rcp_approx(e2);
  const float ratio = __fmul_rn(A, r);
  const float g = __fsub_rn(__fsub_rn(__fmul_rn(__fsub_rn(e2, e1), r), 0x1p-18f), __fmul_rn(0x1p-35f, ratio));
  const bool certain = g > 0.0f && __fmul_rn(g, g) > __fmul_rn(0x1p-38f, ratio);
  return certain && ratio <= 0x1p36f && A > 0.0f;
}

// The anchored code of Eq. 7 (anchor c = 2 * half_c; RTN is c = 6), decided by the hardware
// E4M3 conversion (round-to-nearest-even, saturating at 448) of two bracketing quotients
// r_lo = amax_k * inv_lo and r_hi = amax_k * inv_hi, with inv_lo and inv_hi the reciprocal
// 1 / (c sgk) (relative error <= 2^-23) scaled by 1 -+ 2^-20: r_lo lies below the exact
// quotient amax_g / (c s_g) and r_hi above it, so where the two conversions (one
// instruction for the pair) agree, that code is the exact rounding; otherwise an E4M3
// midpoint lies between them and the exact midpoint tests of anchored_code() decide.
// Quotients below the fp32 normal range convert to code 0 under both.  Code 0 is clamped
// to 1.
__device__ __forceinline__ uint32_t anchored_code_fast(float amax_k, float sgk, float inv_lo, float inv_hi,
                                                       float inv_raw, float half_c) {
  const float rl = __fmul_rn(amax_k, inv_lo), rh = __fmul_rn(amax_k, inv_hi);
  uint32_t p;
  asm("{\n\t.reg .b16 t;\n\tcvt.rn.satfinite.e4m3x2.f32 t, %1, %2;\n\tcvt.u32.u16 %0, t;\n\t}"
      : "=r"(p)
      : "f"(rh), "f"(rl));
  uint32_t c = p & 0xFFu;
  if (c != (p >> 8)) c = anchored_code(amax_k, sgk, inv_raw, half_c);
  return c < 1u ? 1u : c;
}

// Bracketing factors of a reciprocal (see quantize_pack): 1 -+ 2^-20.
constexpr float kBracketLo = 1.0f - 0x1p-20f;
constexpr float kBracketHi = 1.0f + 0x1p-20f;

// Reciprocal 1 / (c sgk) scaled by the bracketing factors (lo, hi) of anchored_code_fast.
__device__ __forceinline__ float2 anchor_brackets(float sgk, float c) {
  const float r = __frcp_rn(__fmul_rn(c, sgk));
  return make_float2(__fmul_rn(r, kBracketLo), __fmul_rn(r, kBracketHi));
}

}  // namespace hscale
