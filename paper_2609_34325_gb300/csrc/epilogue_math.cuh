// Row arithmetic of the linears' epilogues on 32-column chunks held in registers.
#pragma once

#include <stdint.h>

#include "dora_ptx.cuh"
#include "token_ops.cuh"

namespace dora {

__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// GELU(x) = x * Phi(x), Phi(x) = (1 + erf(x / sqrt 2)) / 2, with erf from
// formula 7.1.26 of Abramowitz & Stegun, Handbook of Mathematical Functions
// (|erf error| <= 1.5e-7): for z >= 0,
//     erf(z) = 1 - t (a1 + t (a2 + t (a3 + t (a4 + t a5)))) exp(-z^2),
//     t = 1 / (1 + p z).
// With z = |x| / sqrt 2 and q = (1 - erf(z)) / 2, Phi = 1 - q for x >= 0 and
// q for x < 0, so in both cases GELU(x) = max(x, 0) - |x| q: no select on
// the sign.  The constants below fold in the 1/sqrt 2, the 1/2 and the sign
// of q.  Evaluated on two values at once with the paired fp32 instructions
// (fma/mul.rn.f32x2): the epilogue's ALU work is what limits this GEMM.
__device__ __forceinline__ void gelu_erf2(float& x0, float& x1) {
  const uint64_t P2 = f2_pack(0.3275911f * 0.70710678118654752f, 0.3275911f * 0.70710678118654752f);
  const uint64_t ONE2 = f2_pack(1.0f, 1.0f);
  const uint64_t A1 = f2_pack(-0.5f * 0.254829592f, -0.5f * 0.254829592f);
  const uint64_t A2 = f2_pack(-0.5f * -0.284496736f, -0.5f * -0.284496736f);
  const uint64_t A3 = f2_pack(-0.5f * 1.421413741f, -0.5f * 1.421413741f);
  const uint64_t A4 = f2_pack(-0.5f * -1.453152027f, -0.5f * -1.453152027f);
  const uint64_t A5 = f2_pack(-0.5f * 1.061405429f, -0.5f * 1.061405429f);
  const uint64_t C2 = f2_pack(-0.72134752044448170f, -0.72134752044448170f);   // -log2(e) / 2
  const uint64_t AX = f2_pack(fabsf(x0), fabsf(x1));
  float d0, d1;
  f2_unpack(f2_fma(P2, AX, ONE2), d0, d1);
  const uint64_t T = f2_pack(rcp_approx(d0), rcp_approx(d1));
  const uint64_t poly =
      f2_mul(T, f2_fma(T, f2_fma(T, f2_fma(T, f2_fma(T, A5, A4), A3), A2), A1));
  float e0, e1;
  f2_unpack(f2_mul(f2_mul(AX, AX), C2), e0, e1);
  const uint64_t neg_q = f2_mul(poly, f2_pack(ex2_approx(e0), ex2_approx(e1)));
  f2_unpack(f2_fma(AX, neg_q, f2_pack(fmaxf(x0, 0.0f), fmaxf(x1, 0.0f))), x0, x1);
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
