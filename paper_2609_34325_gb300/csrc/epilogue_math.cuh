// Row arithmetic of the linears' epilogues on 32-column chunks held in registers.
#pragma once

#include <stdint.h>

#include "dora_ptx.cuh"
#include "token_ops.cuh"

namespace dora {

// GELU(x) = x * Phi(x) = max(x, 0) - |x| Q(|x|), Q(a) = 1 - Phi(a): no select on
// the sign.  Q = 2^p with p a polynomial of degree 8 for log2 Q, which is smooth,
// and p(0) = -1 exactly, so that the relative error does not grow towards zero.
// Fitted on 5700 points of [0, 7.2] by linear programming to the least largest
// ratio to bounds a little below the errors of erf by formula 7.1.26 of Abramowitz &
// Stegun (with its reciprocal and exponential).  In fp32 against 64 bits, in brackets
// that formula: |error| <= 2.7e-7 (3.3e-7); relative 3.7e-7 (6.5e-7) for |x| < 0.1,
// 4.7e-7 (7.9e-7) for |x| < 1, 3.7e-6 (4.0e-6) down to x = -2.5, 3.0e-3 (3.6e-3) to
// -6; not above it in the largest or the rms error of any range down to -7.  Below
// -7, where |GELU| < 1e-11, p falls too fast: the error stays below 6e-16, but is
// 0.1 of GELU (0.01) at -8 and 0.5 (0.015) at -9.
// Evaluated on two values at once with the paired fp32 instructions
// (fma.rn.f32x2), in -|x|: the epilogue's ALU work is what limits this GEMM, about
// 2 us for each degree.  fc1 at 50432 x 3072 x 768, us: 162.1, with the formula
// 168.5; degree 7 with p(0) fitted too 160 (relative 8.3e-6 near zero), degree 10
// on [0, 11], nowhere further off than the formula, 166.3.
__device__ __forceinline__ void gelu_erf2(float& x0, float& x1) {
  constexpr float kP[9] = {-1.0f,            1.15111219f,      -0.45913319f,
                           0.0527509033f,    0.00745460154f,   0.000444294797f,
                           -5.89050899e-05f, -1.312108e-05f,   -7.22790292e-07f};
  const uint64_t NX = f2_pack(-fabsf(x0), -fabsf(x1));
  uint64_t p = f2_pack(kP[8], kP[8]);
#pragma unroll
  for (int k = 7; k >= 0; --k) p = f2_fma(p, NX, f2_pack(kP[k], kP[k]));
  float p0, p1;
  f2_unpack(p, p0, p1);
  f2_unpack(f2_fma(NX, f2_pack(ex2_approx(p0), ex2_approx(p1)),
                   f2_pack(fmaxf(x0, 0.0f), fmaxf(x1, 0.0f))),
            x0, x1);
}

// The folded LayerNorm of 32 columns: v = rstd (v - mean c) + d.
__device__ __forceinline__ void fold_layernorm(float (&v)[32], float neg_mean, float rstd,
                                               const float* cs, const float* cb) {
  const float4* cp = reinterpret_cast<const float4*>(cs);
  const float4* dp = reinterpret_cast<const float4*>(cb);
  const uint64_t NM = f2_pack(neg_mean, neg_mean), RS = f2_pack(rstd, rstd);
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const float4 c = cp[q], d = dp[q];
    f2_unpack(f2_fma(RS, f2_fma(NM, f2_pack(c.x, c.y), f2_pack(v[4 * q], v[4 * q + 1])),
                     f2_pack(d.x, d.y)),
              v[4 * q], v[4 * q + 1]);
    f2_unpack(f2_fma(RS, f2_fma(NM, f2_pack(c.z, c.w), f2_pack(v[4 * q + 2], v[4 * q + 3])),
                     f2_pack(d.z, d.w)),
              v[4 * q + 2], v[4 * q + 3]);
  }
}

// Adds 8 bf16 values (one 16-byte piece) to v[0..7] in fp32 pairs.
__device__ __forceinline__ void add_bf16x8(float* v, const uint4& piece) {
  const uint32_t* w = reinterpret_cast<const uint32_t*>(&piece);
#pragma unroll
  for (int e = 0; e < 4; ++e)
    f2_unpack(f2_add(f2_pack(v[2 * e], v[2 * e + 1]), f2_pack(bf16_lo(w[e]), bf16_hi(w[e]))),
              v[2 * e], v[2 * e + 1]);
}

__device__ __forceinline__ void pack_row(const float (&v)[32], uint32_t (&o)[16]) {
#pragma unroll
  for (int e = 0; e < 16; ++e) o[e] = pack_bf16x2(v[2 * e], v[2 * e + 1]);
}

// Slice moments (mean, sum of squared deviations from it) of one 64-column
// slice of a rounded output row, from its two packed 32-column chunks.
__device__ __forceinline__ float2 slice_moments(const uint32_t (&lo)[16], const uint32_t (&hi)[16]) {
  float s4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int e = 0; e < 16; ++e) {
    s4[e & 1] += bf16_lo(lo[e]) + bf16_hi(lo[e]);
    s4[2 + (e & 1)] += bf16_lo(hi[e]) + bf16_hi(hi[e]);
  }
  const float mean = ((s4[0] + s4[1]) + (s4[2] + s4[3])) * (1.0f / kSliceCols);
  float q4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int e = 0; e < 16; ++e) {
    const float a = bf16_lo(lo[e]) - mean, b = bf16_hi(lo[e]) - mean;
    const float c = bf16_lo(hi[e]) - mean, d = bf16_hi(hi[e]) - mean;
    q4[e & 1] += a * a + b * b;
    q4[2 + (e & 1)] += c * c + d * d;
  }
  return make_float2(mean, (q4[0] + q4[1]) + (q4[2] + q4[3]));
}

// Row moments (mean, var) of one row from its S slice moments (mean_s, M2_s)
// over 64 columns each, stored slice-major with `stride` rows between slices:
// mean = (1/S) sum mean_s, M2 = sum (M2_s + 64 (mean_s - mean)^2) (the
// pairwise update of Chan, Golub & LeVeque with equal counts), var = M2 / (64 S).
// Every rounding is explicit, so each caller gets the same bits.
__device__ __forceinline__ float2 merge_slice_moments(const float2* __restrict__ p, size_t stride,
                                                      int slices) {
  constexpr int kHeld = 16;     // slice means held in registers (dim <= 1024)
  const float inv_s = __frcp_rn(static_cast<float>(slices));
  float mean, m2 = 0.f;
  if (slices <= kHeld) {
    float mu[kHeld];
#pragma unroll
    for (int j = 0; j < kHeld; ++j)
      if (j < slices) mu[j] = __ldg(&p[j * stride].x);
    float sum = 0.f;
#pragma unroll
    for (int j = 0; j < kHeld; ++j)
      if (j < slices) sum = __fadd_rn(sum, mu[j]);
    mean = __fmul_rn(sum, inv_s);
#pragma unroll
    for (int j = 0; j < kHeld; ++j)
      if (j < slices) {             // the M2 halves are read again (L1)
        const float d = __fsub_rn(mu[j], mean);
        m2 = __fadd_rn(m2, __fmaf_rn(__fmul_rn(static_cast<float>(kSliceCols), d), d,
                                     __ldg(&p[j * stride].y)));
      }
  } else {
    float sum = 0.f;
    for (int j = 0; j < slices; ++j) sum = __fadd_rn(sum, __ldg(&p[j * stride].x));
    mean = __fmul_rn(sum, inv_s);
    for (int j = 0; j < slices; ++j) {
      const float2 t = __ldg(p + j * stride);
      const float d = __fsub_rn(t.x, mean);
      m2 = __fadd_rn(m2, __fmaf_rn(__fmul_rn(static_cast<float>(kSliceCols), d), d, t.y));
    }
  }
  return make_float2(mean, __fmul_rn(__fmul_rn(m2, inv_s), 1.0f / kSliceCols));
}

// Row moments (mean, biased variance) of a 128-column row from its two slices'
// moments, rounded as the general merge rounds.
__device__ __forceinline__ float2 merge_two_slices(float2 lo, float2 hi) {
  const float mean = __fmul_rn(__fadd_rn(lo.x, hi.x), 0.5f);
  const float dl = __fsub_rn(lo.x, mean), dh = __fsub_rn(hi.x, mean);
  constexpr float kN = static_cast<float>(kSliceCols);
  float m2 = __fmaf_rn(__fmul_rn(kN, dl), dl, lo.y);
  m2 = __fadd_rn(m2, __fmaf_rn(__fmul_rn(kN, dh), dh, hi.y));
  return make_float2(mean, __fmul_rn(m2, 1.0f / (2.0f * kN)));
}

}  // namespace dora
