// The deterministic actor of DORA at deployment (Sec. 3.2 "The actor";
// Appendix A.1-A.3), at one block, for every image of a packed batch:
//   gate      p = sigmoid(MLP_G([K_CLS, e^G_l, h_l])), a (d + 19) -> 64 -> 1
//             SiLU MLP;
//   encoder   X = W_in K + b_in + e^C_l (+ W_h h_l on the CLS row), then one
//             pre-LayerNorm Transformer block of width 128 (four heads of 32,
//             GELU feed-forward 128 -> 256 -> 128): X and QKV in one kernel
//             (actor_front.cu), the varlen attention, and all that follows it in
//             another (actor_tail.cu);
//   budget    the highest logit of MLP_B(LayerNorm(Z_CLS)) among the budgets
//             k <= N_l - 4 (ties to the smaller), and
//   selector  s_j = MLP_S(Z_j + W_k k / N_l), a 128 -> 64 -> 1 SiLU MLP,
//             written W_1 Z_j + b_1 + (k / N_l) W_1 W_k: the first term comes
//             with Z, W_1 W_k is made once per set of weights, and the rest runs
//             per token.
// Four launches: gate, budget and the selector's rest are the last one (one CTA
// per image).  With a launch each for the input projection, gate with history, row
// moments, QKV, budget and selector the call took 133.6 us at 256 x 197 tokens, now
// 106.4; 8 ragged images of d = 384 took 53.5, now 37.9.
// The attention kernel has an instance for heads of 32 (softmax scale
// 1/sqrt(32)).  On heads zero-padded to 64 the QKV linear wrote twice the bytes
// and both MMAs did twice the work: 256 x 197 tokens, QKV 29.7 -> 16.5 us,
// attention 33 -> 30.8, output projection 14.7 -> 14.0.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "dora.h"
#include "dora_ptx.cuh"
#include "token_ops.cuh"

namespace dora {
namespace actor {

constexpr int W = 128;          // encoder width
constexpr int HEADS = 4;
constexpr int HD = 32;          // encoder head width
constexpr int FF = 256;         // feed-forward width
constexpr int GH = 64;          // gate hidden units
constexpr int GE = 16;          // gate block embedding
constexpr int SH = 64;          // selector hidden units
constexpr int kMaxDim = 2048;
constexpr int kMaxN0 = 1028;    // budget-head outputs (n0 - 4) / 2 <= 512
constexpr int kMaxBudgets = (kMaxN0 - 4) / 2;

__device__ __forceinline__ float ld(const uint16_t* __restrict__ p, size_t i) {
  return __uint_as_float(static_cast<uint32_t>(p[i]) << 16);
}
__device__ __forceinline__ uint16_t to_bf16(float v) {
  const __nv_bfloat16 h = __float2bfloat16_rn(v);
  return *reinterpret_cast<const uint16_t*>(&h);
}
__device__ __forceinline__ float4 bf16x4(uint2 v) {
  return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xFFFF0000u),
                     __uint_as_float(v.y << 16), __uint_as_float(v.y & 0xFFFF0000u));
}
__device__ __forceinline__ float silu(float x) { return x / (1.f + expf(-x)); }
__device__ __forceinline__ float gelu(float x) {
  return 0.5f * x * (1.f + erff(x * 0.70710678118654752f));
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ---------------------------------------------------------------------------
// preparation (once per set of weights)
// ---------------------------------------------------------------------------
// The selector's W_1 W_k (fp32 [64]).
__global__ void sel_wk_kernel(const uint16_t* __restrict__ w1, const uint16_t* __restrict__ w_k,
                              float* __restrict__ out) {
  const int h = threadIdx.x;
  float a = 0.f;
  for (int c = 0; c < W; ++c) a = fmaf(ld(w1, static_cast<size_t>(h) * W + c), ld(w_k, c), a);
  out[h] = a;
}

// The input projection's bias at every block: bf16(b_in + e^C_l).
__global__ void bias_in_kernel(const uint16_t* __restrict__ b_in, const uint16_t* __restrict__ emb,
                               uint16_t* __restrict__ out) {
  const int l = blockIdx.x;
  for (int c = threadIdx.x; c < W; c += blockDim.x)
    out[static_cast<size_t>(l) * W + c] = to_bf16(ld(b_in, c) + ld(emb, static_cast<size_t>(l) * W + c));
}

// ---------------------------------------------------------------------------
// W^T of the gate's first layer, [inputs, outputs]
// ---------------------------------------------------------------------------
__global__ void transpose_kernel(const uint16_t* __restrict__ w, int rows, int cols,
                                 uint16_t* __restrict__ wt) {
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < rows * cols;
       idx += gridDim.x * blockDim.x) {
    const int c = idx / rows, r = idx % rows;    // wt [cols, rows]
    wt[idx] = w[static_cast<size_t>(r) * cols + c];
  }
}

// h_l = [N_l / N0, rho_l, E_<l / (L - 1)]
struct History {
  float h0, h1, h2;
};
__device__ __forceinline__ History history(int n, int n0, const float* __restrict__ rho,
                                           const int32_t* __restrict__ interventions, int depth,
                                           int i) {
  return {static_cast<float>(n) / static_cast<float>(n0), rho[i],
          static_cast<float>(interventions[i]) / static_cast<float>(max(depth - 1, 1))};
}
// Visual tokens of the image with bounds [lo, hi); -1 if it is empty or
// outside the buffer.
__device__ __forceinline__ int visual_tokens(int lo, int hi, int t_cap) {
  return (lo < 0 || hi > t_cap) ? -1 : hi - lo - 1;
}

// ---------------------------------------------------------------------------
// gate, budget head and selector tail (Appendix A.1-A.3; Eq. 2): one CTA of 16
// warps per image.  Warps 8-15 run the gate, its first layer reading the
// transposed weights 16 bytes (eight hidden units) at a time; warps 0-7 run the
// budget head, each normalising Z_CLS for itself (four columns a lane) and
// taking an output at a time of each layer.  Then the selector's tail with two
// threads per visual token, s = w_2 . silu(S1_j + (k / N_l) W_1 W_k) + b_2, where
// S1_j = W_1 Z_j + b_1 came with Z and k is the image's budget.
// Latency bounds it: the chain of dependent loads, so each phase's weights are
// in flight before its input is known.  13.8 us at 256 x 197 tokens, d = 768,
// where the three kernels it replaces took 14, 13 and 10 (the gate staged 100 KB
// of weights for two-byte reads, so the second wave of images waited for the
// first); one group of 8 warps doing all in turn took 23.
// ---------------------------------------------------------------------------
constexpr int kDecideThreads = 512;
constexpr int kHeadThreads = kDecideThreads / 2;     // of the budget head, and of the gate
constexpr int kHeadWarps = kHeadThreads / 32;
constexpr int kFlight = 8;                           // a warp's weight rows in flight

__device__ __forceinline__ void bar_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

__device__ __forceinline__ void fma_bf16x8(float (&acc)[8], const uint4& w, float x) {
  const uint32_t p[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    acc[2 * e] = fmaf(__uint_as_float(p[e] << 16), x, acc[2 * e]);
    acc[2 * e + 1] = fmaf(__uint_as_float(p[e] & 0xFFFF0000u), x, acc[2 * e + 1]);
  }
}

// Rows m0, m0 + kHeadWarps, ... of w [rows, 128], this lane's four columns.
__device__ __forceinline__ void load_rows(uint2 (&r)[kFlight], const uint16_t* __restrict__ w,
                                          int m0, int rows) {
#pragma unroll
  for (int e = 0; e < kFlight; ++e) {
    const int m = m0 + e * kHeadWarps;
    r[e] = m < rows ? __ldg(reinterpret_cast<const uint2*>(w + static_cast<size_t>(m) * W) +
                            (threadIdx.x & 31))
                    : make_uint2(0u, 0u);
  }
}
// Their dot products with x (this lane's columns): lane e < kFlight gets row e's.
__device__ __forceinline__ float dot_rows(const uint2 (&r)[kFlight], const float4& x) {
  const int lane = threadIdx.x & 31;
  float mine = 0.f;
#pragma unroll
  for (int e = 0; e < kFlight; ++e) {
    float s = __uint_as_float(r[e].x << 16) * x.x;
    s = fmaf(__uint_as_float(r[e].x & 0xFFFF0000u), x.y, s);
    s = fmaf(__uint_as_float(r[e].y << 16), x.z, s);
    s = fmaf(__uint_as_float(r[e].y & 0xFFFF0000u), x.w, s);
    s = warp_sum(s);
    if (lane == e) mine = s;
  }
  return mine;
}

struct DecideArgs {
  const uint16_t* qkv;              // the block's, [t_cap, 3 dim]
  const int32_t* cu;
  int t_cap, dim, block, depth, n0;
  float eps;
  const float* rho;
  const int32_t* interventions;
  const uint16_t *gate_w1t, *gate_b1, *gate_w2, *gate_b2, *gate_emb;
  const uint16_t* z;                // Z [t_cap, 128]
  const uint16_t *ln_w, *ln_b, *bw1, *bb1, *bw2, *bb2;
  const uint16_t* s1;               // S1 [t_cap, 64]
  const float* sel_wk;
  const uint16_t *sw2, *sb2;
  float* p_gate;                    // nullable
  int32_t *gate, *budget, *k_out, *keep;
  float* rho_next;                  // nullable
  int32_t* e_next;                  // nullable
  float* scores;
};

__global__ void __launch_bounds__(kDecideThreads, 2) decide_kernel(const DecideArgs a) {
  __shared__ float zin[kMaxDim + GE + 3];
  __shared__ float part[kHeadWarps][GH];
  __shared__ __align__(16) float hb[W];
  __shared__ float logit[kMaxBudgets], swk[SH], sw2s[SH];
  __shared__ float glogit;
  __shared__ int s_best;
  pdl_trigger();
  pdl_wait();
  const int i = blockIdx.x, t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int lo = a.cu[i], n = visual_tokens(lo, a.cu[i + 1], a.t_cap);
  if (n < 0) {                                       // empty (or outside the buffer): closed
    if (t == 0) {
      if (a.p_gate != nullptr) a.p_gate[i] = 0.f;
      a.gate[i] = a.budget[i] = a.k_out[i] = a.keep[i] = 0;
      if (a.rho_next != nullptr) a.rho_next[i] = 0.f;
      if (a.e_next != nullptr) a.e_next[i] = a.interventions[i];
    }
    return;
  }
  const int m_out = (a.n0 - 4) / 2;
  if (t < kHeadThreads) {
    // ---- budget head: LayerNorm(Z_CLS) -> 128 GELU -> M logits ----
    const uint2 zr = reinterpret_cast<const uint2*>(a.z + static_cast<size_t>(lo) * W)[lane];
    const uint2 gr = reinterpret_cast<const uint2*>(a.ln_w)[lane];
    const uint2 br = reinterpret_cast<const uint2*>(a.ln_b)[lane];
    uint2 r[kFlight];
    load_rows(r, a.bw1, warp, W);
    const float4 zv = bf16x4(zr), gv = bf16x4(gr), bv = bf16x4(br);
    const float mean = warp_sum((zv.x + zv.y) + (zv.z + zv.w)) * (1.f / W);
    float4 x = make_float4(zv.x - mean, zv.y - mean, zv.z - mean, zv.w - mean);
    const float rstd =
        rsqrtf(warp_sum((x.x * x.x + x.y * x.y) + (x.z * x.z + x.w * x.w)) * (1.f / W) + a.eps);
    x = make_float4(x.x * rstd * gv.x + bv.x, x.y * rstd * gv.y + bv.y, x.z * rstd * gv.z + bv.z,
                    x.w * rstd * gv.w + bv.w);
#pragma unroll
    for (int m0 = 0; m0 < W; m0 += kFlight * kHeadWarps) {
      const float s = dot_rows(r, x);
      if (m0 + kFlight * kHeadWarps < W) load_rows(r, a.bw1, m0 + kFlight * kHeadWarps + warp, W);
      else load_rows(r, a.bw2, warp, m_out);
      const int m = m0 + lane * kHeadWarps + warp;
      if (lane < kFlight) hb[m] = gelu(s + ld(a.bb1, m));
    }
    bar_sync(1, kHeadThreads);
    const float4 h = reinterpret_cast<const float4*>(hb)[lane];
    for (int m0 = 0; m0 < m_out; m0 += kFlight * kHeadWarps) {
      const float s = dot_rows(r, h);
      load_rows(r, a.bw2, m0 + kFlight * kHeadWarps + warp, m_out);
      const int m = m0 + lane * kHeadWarps + warp;
      if (lane < kFlight && m < m_out) logit[m] = s + ld(a.bb2, m);
    }
    bar_sync(1, kHeadThreads);
    if (warp == 0) {
      // the first of the highest among the feasible (2 (m + 1) <= n - 4); a NaN
      // counts only in the first place, where nothing is higher than it
      const int feasible = min(n >= 6 ? (n - 4) / 2 : 0, m_out);
      int best = feasible;
      float bv_ = -INFINITY;
      for (int m = lane; m < feasible; m += 32)
        if (logit[m] > bv_ || (best == feasible && logit[m] == bv_)) {
          best = m;
          bv_ = logit[m];
        }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, bv_, o);
        const int om = __shfl_xor_sync(0xffffffffu, best, o);
        if (ov > bv_ || (ov == bv_ && om < best)) {
          best = om;
          bv_ = ov;
        }
      }
      if (feasible == 0) best = -1;
      else if (best == feasible || logit[0] != logit[0]) best = 0;
      if (lane == 0) s_best = best;
    }
  } else {
    // ---- gate: SiLU MLP of [K_CLS, e^G_l, h_l] ----
    const int tg = t - kHeadThreads, kin = a.dim + GE + 3;
    const size_t krow = static_cast<size_t>(lo) * 3 * a.dim + a.dim;   // the CLS key
    for (int c = tg; c < a.dim; c += kHeadThreads) zin[c] = ld(a.qkv, krow + c);
    if (tg < GE) zin[a.dim + tg] = ld(a.gate_emb, static_cast<size_t>(a.block) * GE + tg);
    if (tg == kHeadThreads - 1) {
      const History hs = history(n, a.n0, a.rho, a.interventions, a.depth, i);
      zin[a.dim + GE] = hs.h0;
      zin[a.dim + GE + 1] = hs.h1;
      zin[a.dim + GE + 2] = hs.h2;
    }
    if (tg < SH) {
      swk[tg] = a.sel_wk[tg];
      sw2s[tg] = ld(a.sw2, tg);
    }
    bar_sync(2, kHeadThreads);
    // hidden units 8 (tg % 8) .. + 7 over inputs tg / 8, tg / 8 + 32, ...
    const uint4* w = reinterpret_cast<const uint4*>(a.gate_w1t) + tg % 8;
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int c = tg / 8; c < kin; c += 8 * 32) {
      uint4 r[8];
#pragma unroll
      for (int e = 0; e < 8; ++e)
        r[e] = c + 32 * e < kin ? __ldg(w + static_cast<size_t>(c + 32 * e) * (GH / 8))
                                : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
      for (int e = 0; e < 8; ++e)
        if (c + 32 * e < kin) fma_bf16x8(acc, r[e], zin[c + 32 * e]);
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], 8);
      acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], 16);
      if (lane < 8) part[warp - kHeadWarps][8 * lane + e] = acc[e];
    }
    bar_sync(2, kHeadThreads);
    if (warp == kHeadWarps) {
      float s = 0.f;
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int h = lane + 32 * e;
        float p[kHeadWarps];
#pragma unroll
        for (int q = 0; q < kHeadWarps; ++q) p[q] = part[q][h];
        s += ld(a.gate_w2, h) *
             silu((((p[0] + p[1]) + (p[2] + p[3])) + ((p[4] + p[5]) + (p[6] + p[7]))) +
                  ld(a.gate_b1, h));
      }
      s = warp_sum(s);
      if (lane == 0) {
        const float lg = s + ld(a.gate_b2, 0);
        glogit = lg;
        if (a.p_gate != nullptr) a.p_gate[i] = 1.f / (1.f + expf(-lg));
      }
    }
  }
  // ---- selector tail: threads 2 j and 2 j + 1 take 32 hidden units each of token j ----
  const int half = t & 1;
  uint4 v[SH / 16];
  auto load_s1 = [&](int j) {
    if (j <= n) {
      const uint4* p = reinterpret_cast<const uint4*>(a.s1 + static_cast<size_t>(lo + j) * SH) +
                       half * (SH / 16);
#pragma unroll
      for (int q = 0; q < SH / 16; ++q) v[q] = p[q];
    }
  };
  load_s1(1 + t / 2);
  const float b2 = ld(a.sb2, 0);
  __syncthreads();
  const int bud = s_best < 0 ? 0 : 2 * (s_best + 1);
  if (t == 0) {
    const int g = (glogit >= 0.f && bud > 0) ? 1 : 0;
    const int kk = g ? bud : 0;
    a.budget[i] = bud;
    a.gate[i] = g;
    a.k_out[i] = kk;
    a.keep[i] = n + 1 - kk;
    if (a.rho_next != nullptr) a.rho_next[i] = n > 0 ? static_cast<float>(kk) / n : 0.f;
    if (a.e_next != nullptr) a.e_next[i] = a.interventions[i] + g;
    a.scores[lo] = 0.f;
  }
  const float kr = static_cast<float>(bud) / n;      // n = 0: no token uses it
  const float* wk = swk + half * (SH / 2);
  const float* w2 = sw2s + half * (SH / 2);
#pragma unroll 1
  for (int j0 = 0; j0 < n; j0 += kDecideThreads / 2) {
    const int j = 1 + j0 + t / 2;
    float acc = 0.f;
    if (j <= n) {
#pragma unroll
      for (int q = 0; q < SH / 16; ++q) {
        const uint32_t wv[4] = {v[q].x, v[q].y, v[q].z, v[q].w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int h = 8 * q + 2 * e;
          acc = fmaf(w2[h], silu(__uint_as_float(wv[e] << 16) + kr * wk[h]), acc);
          acc = fmaf(w2[h + 1], silu(__uint_as_float(wv[e] & 0xFFFF0000u) + kr * wk[h + 1]), acc);
        }
      }
    }
    acc += __shfl_xor_sync(0xffffffffu, acc, 1);
    if (j <= n && half == 0) a.scores[lo + j] = acc + b2;
    load_s1(j + kDecideThreads / 2);
  }
}

// ---------------------------------------------------------------------------
// host side: layouts
// ---------------------------------------------------------------------------
size_t up256(size_t v) { return (v + 255) & ~static_cast<size_t>(255); }

struct Prep {
  size_t bias_in, wqkv, cqkv, dqkv, wfc1, cfc1, dfc1, sel_wk, gate_w1t, total;
};

Prep prep_layout(const dora_actor_weights* w) {
  Prep P{};
  size_t off = 0;
  P.bias_in = off; off += up256(static_cast<size_t>(w->depth) * W * 2);
  P.wqkv = off;    off += up256(3 * W * W * 2);
  P.cqkv = off;    off += up256(3 * W * 4);
  P.dqkv = off;    off += up256(3 * W * 4);
  P.wfc1 = off;    off += up256(FF * W * 2);
  P.cfc1 = off;    off += up256(FF * 4);
  P.dfc1 = off;    off += up256(FF * 4);
  P.sel_wk = off;  off += up256(SH * 4);
  P.gate_w1t = off; off += up256(static_cast<size_t>(w->dim + GE + 3) * GH * 2);
  P.total = off;
  return P;
}

struct Ws {
  size_t status, x, qkv, o, z, s1, prep, total;
};

Ws ws_layout(int32_t t_cap, int32_t batch, const dora_actor_weights* w) {
  Ws L{};
  const size_t t = static_cast<size_t>(t_cap), b = static_cast<size_t>(batch);
  size_t off = 0;
  L.status = off; off += 256;
  L.x = off;      off += up256(t * W * 2);
  L.qkv = off;    off += up256(t * 3 * W * 2);
  L.o = off;      off += up256(t * W * 2);
  L.z = off;      off += up256(t * W * 2);
  L.s1 = off;     off += up256(t * SH * 2);
  // More than the present launches use: the size is part of the interface, as it was
  // when heads were padded to 64 and Z1, moments, the feed-forward's hidden rows and
  // the gate's logits were kept (a smaller one would refuse nobody, but change it).
  off += up256(b * 4) + up256(t * (3 * W * 2 + W * 2 + W * 2 + 3 * 8 + FF * 2));
  L.prep = off;   off += w->prepared != nullptr ? 0 : prep_layout(w).total;
  L.total = off;
  return L;
}

bool weights_ok(const dora_actor_weights* w) {
  if (w == nullptr) return false;
  if (w->dim <= 0 || w->dim % 64 != 0 || w->dim > kMaxDim) return false;
  if (w->depth <= 0 || w->n0 < 6 || w->n0 > kMaxN0) return false;
  if (!(w->eps >= 0.f) || !isfinite(w->eps)) return false;
  const void* req[] = {w->gate_w1, w->gate_b1, w->gate_w2, w->gate_b2, w->gate_emb,
                       w->enc_w_in, w->enc_b_in, w->enc_emb, w->enc_w_h, w->enc_ln1_w,
                       w->enc_ln1_b, w->enc_w_qkv, w->enc_b_qkv, w->enc_w_o, w->enc_b_o,
                       w->enc_ln2_w, w->enc_ln2_b, w->enc_w_fc1, w->enc_b_fc1, w->enc_w_fc2,
                       w->enc_b_fc2, w->bud_ln_w, w->bud_ln_b, w->bud_w1, w->bud_b1,
                       w->bud_w2, w->bud_b2, w->sel_w_k, w->sel_w1, w->sel_b1, w->sel_w2,
                       w->sel_b2};
  for (const void* p : req)
    if (p == nullptr || (reinterpret_cast<uintptr_t>(p) & 15u) != 0) return false;
  return (reinterpret_cast<uintptr_t>(w->prepared) & 255u) == 0;
}

cudaError_t prepare(const dora_actor_weights* w, uint8_t* prep, cudaStream_t stream) {
  const Prep P = prep_layout(w);
  cudaError_t e = launch_fold_ln(w->enc_w_qkv, 3 * W, W, w->enc_ln1_w, w->enc_ln1_b,
                                 w->enc_b_qkv, reinterpret_cast<uint16_t*>(prep + P.wqkv),
                                 reinterpret_cast<float*>(prep + P.cqkv),
                                 reinterpret_cast<float*>(prep + P.dqkv), stream);
  if (e != cudaSuccess) return e;
  bias_in_kernel<<<w->depth, W, 0, stream>>>(w->enc_b_in, w->enc_emb,
                                             reinterpret_cast<uint16_t*>(prep + P.bias_in));
  sel_wk_kernel<<<1, SH, 0, stream>>>(w->sel_w1, w->sel_w_k, reinterpret_cast<float*>(prep + P.sel_wk));
  transpose_kernel<<<64, 256, 0, stream>>>(w->gate_w1, GH, w->dim + GE + 3,
                                           reinterpret_cast<uint16_t*>(prep + P.gate_w1t));
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_fold_ln(w->enc_w_fc1, FF, W, w->enc_ln2_w, w->enc_ln2_b, w->enc_b_fc1,
                        reinterpret_cast<uint16_t*>(prep + P.wfc1),
                        reinterpret_cast<float*>(prep + P.cfc1),
                        reinterpret_cast<float*>(prep + P.dfc1), stream);
}

}  // namespace actor
}  // namespace dora

using namespace dora;

extern "C" {

size_t dora_actor_prepared_size(const dora_actor_weights* w) {
  if (w == nullptr || w->depth <= 0) return 0;
  return actor::prep_layout(w).total;
}

size_t dora_actor_workspace_size(int32_t t_cap, int32_t batch, const dora_actor_weights* w) {
  if (w == nullptr || t_cap < 0 || batch < 0 || w->depth <= 0) return 0;
  return actor::ws_layout(t_cap, batch, w).total;
}

int dora_actor_prepare(const dora_actor_weights* w, void* prepared, size_t prepared_bytes,
                       dora_stream_t stream) {
  if (!actor::weights_ok(w) || prepared == nullptr ||
      (reinterpret_cast<uintptr_t>(prepared) & 255u) != 0 ||
      prepared_bytes < actor::prep_layout(w).total)
    return DORA_ERR_INVALID_ARG;
  const int dev = checked_device();
  if (dev == -1) return DORA_ERR_CUDA;
  if (dev < 0) return DORA_ERR_UNSUPPORTED;
  return actor::prepare(w, static_cast<uint8_t*>(prepared),
                        reinterpret_cast<cudaStream_t>(stream)) == cudaSuccess
             ? DORA_OK
             : DORA_ERR_CUDA;
}

int dora_actor(const dora_bf16* qkv, const int32_t* cu, int32_t batch, int32_t max_seqlen,
               int32_t t_cap, int32_t block, const dora_actor_weights* w, const float* rho,
               const int32_t* interventions, float* p_gate, int32_t* gate, int32_t* budget,
               int32_t* k, int32_t* keep_counts, float* scores, float* rho_next,
               int32_t* interventions_next, dora_bf16* z_out, void* workspace,
               size_t workspace_bytes, dora_stream_t stream_) {
  using namespace actor;
  if (!weights_ok(w)) return DORA_ERR_INVALID_ARG;
  if (batch < 0 || batch > 65535 || t_cap < 0 || max_seqlen < 0 || max_seqlen > 65535)
    return DORA_ERR_INVALID_ARG;
  if (block < 0 || block >= w->depth) return DORA_ERR_INVALID_ARG;
  if (cu == nullptr || workspace == nullptr ||
      (reinterpret_cast<uintptr_t>(workspace) & 255u) != 0)
    return DORA_ERR_INVALID_ARG;
  if (batch > 0 && (qkv == nullptr || rho == nullptr || interventions == nullptr ||
                    gate == nullptr || budget == nullptr || k == nullptr ||
                    keep_counts == nullptr || scores == nullptr))
    return DORA_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(qkv) & 15u) != 0 ||
      (reinterpret_cast<uintptr_t>(z_out) & 15u) != 0)
    return DORA_ERR_INVALID_ARG;
  const Ws L = ws_layout(t_cap, batch, w);
  if (workspace_bytes < L.total) return DORA_ERR_INVALID_ARG;
  const int dev = checked_device();
  if (dev == -1) return DORA_ERR_CUDA;
  if (dev < 0) return DORA_ERR_UNSUPPORTED;
  if (t_cap == 0 || batch == 0) return DORA_OK;

  cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  int32_t* status = reinterpret_cast<int32_t*>(ws + L.status);
  uint16_t* x = reinterpret_cast<uint16_t*>(ws + L.x);
  uint16_t* qkv_e = reinterpret_cast<uint16_t*>(ws + L.qkv);
  uint16_t* o_e = reinterpret_cast<uint16_t*>(ws + L.o);
  uint16_t* z = z_out != nullptr ? z_out : reinterpret_cast<uint16_t*>(ws + L.z);
  uint8_t* prep = ws + L.prep;
  if (w->prepared != nullptr) prep = static_cast<uint8_t*>(const_cast<void*>(w->prepared));
  else if (prepare(w, prep, stream) != cudaSuccess) return DORA_ERR_CUDA;
  const Prep P = prep_layout(w);
  const int32_t* rows = cu + batch;
  const int d = w->dim;

  // X = W_in K + (b_in + e^C_l), K read in place from the block's qkv rows, with the
  // history term on every CLS row, and the attention's LayerNorm and QKV linear
  FrontArgs fa;
  fa.cu = cu;
  fa.batch = batch;
  fa.n0 = w->n0;
  fa.depth = w->depth;
  fa.rho = rho;
  fa.interventions = interventions;
  fa.w_h = w->enc_w_h;
  fa.bias = reinterpret_cast<const uint16_t*>(prep + P.bias_in) + static_cast<size_t>(block) * W;
  fa.c = reinterpret_cast<const float*>(prep + P.cqkv);
  fa.d = reinterpret_cast<const float*>(prep + P.dqkv);
  fa.eps = w->eps;
  fa.x = x;
  fa.qkv = qkv_e;
  if (launch_actor_front(qkv + d, 3 * d, d, w->enc_w_in,
                         reinterpret_cast<const uint16_t*>(prep + P.wqkv), fa, t_cap, status,
                         stream) != cudaSuccess ||
      launch_varlen_attn(qkv_e, cu, batch, max_seqlen, t_cap, HEADS, 0.17677669529663688f, o_e,
                         status, stream, HD) != cudaSuccess)
    return DORA_ERR_CUDA;
  // output projection, feed-forward and the selector's first layer on every
  // token, then gate, budget head and selector tail
  uint16_t* s1 = reinterpret_cast<uint16_t*>(ws + L.s1);
  TailArgs ta;
  ta.x = x;
  ta.bo = w->enc_b_o;
  ta.c1 = reinterpret_cast<const float*>(prep + P.cfc1);
  ta.d1 = reinterpret_cast<const float*>(prep + P.dfc1);
  ta.eps = w->eps;
  ta.b2 = w->enc_b_fc2;
  ta.bs = w->sel_b1;
  ta.z = z;
  ta.s1 = s1;
  if (launch_actor_tail(o_e, w->enc_w_o, reinterpret_cast<const uint16_t*>(prep + P.wfc1),
                        w->enc_w_fc2, w->sel_w1, ta, t_cap, rows, status, stream) != cudaSuccess)
    return DORA_ERR_CUDA;
  DecideArgs da;
  da.qkv = qkv;
  da.cu = cu;
  da.t_cap = t_cap;
  da.dim = d;
  da.block = block;
  da.depth = w->depth;
  da.n0 = w->n0;
  da.eps = w->eps;
  da.rho = rho;
  da.interventions = interventions;
  da.gate_w1t = reinterpret_cast<const uint16_t*>(prep + P.gate_w1t);
  da.gate_b1 = w->gate_b1;
  da.gate_w2 = w->gate_w2;
  da.gate_b2 = w->gate_b2;
  da.gate_emb = w->gate_emb;
  da.z = z;
  da.ln_w = w->bud_ln_w;
  da.ln_b = w->bud_ln_b;
  da.bw1 = w->bud_w1;
  da.bb1 = w->bud_b1;
  da.bw2 = w->bud_w2;
  da.bb2 = w->bud_b2;
  da.s1 = s1;
  da.sel_wk = reinterpret_cast<const float*>(prep + P.sel_wk);
  da.sw2 = w->sel_w2;
  da.sb2 = w->sel_b2;
  da.p_gate = p_gate;
  da.gate = gate;
  da.budget = budget;
  da.k_out = k;
  da.keep = keep_counts;
  da.rho_next = rho_next;
  da.e_next = interventions_next;
  da.scores = scores;
  if (launch_pdl(decide_kernel, dim3(batch), dim3(kDecideThreads), 0, stream, da) != cudaSuccess)
    return DORA_ERR_CUDA;
  return DORA_OK;
}

}  // extern "C"
