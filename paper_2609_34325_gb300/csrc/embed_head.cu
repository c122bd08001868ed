// The two ends of the ViT forward, which the paper's GFLOPs and throughput
// include (App. E.4 "GFLOPs accounting"; backbones of Sec. 4.1):
//   patch embedding   a patch x patch convolution with stride patch, as
//                     patchify (a pure relayout) + one tcgen05 GEMM whose rows
//                     are the packed tokens, CLS rows included, and whose
//                     epilogue adds bias, CLS and position embeddings (a pass of
//                     its own over the tokens: 18.5 us for 128 x 257 x 768, the
//                     GEMM with it 32.6 us against 28.6);
//   classifier head   the final LayerNorm on each image's CLS row and the
//                     linear layer to the class logits (tcgen05 GEMM);
//   LC1 head          DINOv2's readout (App. E.3): the final LayerNorm on every
//                     surviving token, normalised CLS ++ the mean of the
//                     normalised visual rows of each image, then the linear
//                     layer on the 2 d features;
//   LayerScale fold   DINOv2's per-channel branch scales folded once into the
//                     rows of the attention output and fc2 linears.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <float.h>
#include <stdint.h>

#include "dora.h"
#include "dora_ptx.cuh"
#include "token_ops.cuh"

namespace dora {
namespace embed {

__device__ __forceinline__ float lo_f(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float hi_f(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }
__device__ __forceinline__ uint32_t pack2(float a, float b) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// The patch matrix has a row per token of the packed layout, image after image:
// row b (g + 1) is image b's CLS row, zero (the GEMM's epilogue puts the CLS
// token there), and row b (g + 1) + 1 + gy gw + gx its patch (gy, gx), column
// c p^2 + dy p + dx.  So the GEMM's output rows are the tokens themselves.

// p a multiple of 8: 8 pixels (16 bytes) a thread, twice as many where p is a
// multiple of 16.  The weights [d, C, p, p] flattened are the GEMM's B.
template <int V>
__global__ void patchify_kernel(const uint4* __restrict__ img, int batch, int ch, int h, int w,
                                int p, uint4* __restrict__ out) {
  pdl_trigger();
  pdl_wait();
  const int gw = w / p, g = gw * (h / p), wv = w / (8 * V), kcols8 = ch * p * p / 8;
  const uint32_t row_segs = static_cast<uint32_t>(h) * wv;      // V-vectors of a channel
  const uint32_t segs = static_cast<uint32_t>(batch) * ch * row_segs;
  const uint32_t zeros = static_cast<uint32_t>(batch) * (kcols8 / V);
  for (uint32_t s = blockIdx.x * blockDim.x + threadIdx.x; s < segs + zeros;
       s += gridDim.x * blockDim.x) {
    if (s >= segs) {                                            // CLS rows
      const uint32_t z = s - segs, b = z / (kcols8 / V), c = z - b * (kcols8 / V);
#pragma unroll
      for (int v = 0; v < V; ++v)
        out[static_cast<size_t>(b) * (g + 1) * kcols8 + c * V + v] = make_uint4(0u, 0u, 0u, 0u);
      continue;
    }
    const uint32_t bc = s / row_segs, in = s - bc * row_segs;
    const int y = in / wv, x = (in - y * wv) * 8 * V;
    const int b = bc / ch, c = bc - b * ch, gy = y / p, gx = x / p;
    const size_t row = static_cast<size_t>(b) * (g + 1) + 1 + gy * gw + gx;
    const int col8 = (c * p * p + (y - gy * p) * p + x - gx * p) / 8;
#pragma unroll
    for (int v = 0; v < V; ++v) out[row * kcols8 + col8 + v] = __ldg(img + static_cast<size_t>(s) * V + v);
  }
}

// Any patch side: one thread writes 8 consecutive columns of one row of the
// K-padded patch matrix [B (g + 1), kpad] (2-byte gathers; columns >= C p^2 and
// CLS rows are zero).
__global__ void patchify_any_kernel(const uint16_t* __restrict__ img, int batch, int ch, int h,
                                    int w, int p, int kpad, uint4* __restrict__ out) {
  pdl_trigger();
  pdl_wait();
  const int gw = w / p, gh = h / p, g = gw * gh, pp = p * p, k = ch * pp, kp8 = kpad / 8;
  const long long total = static_cast<long long>(batch) * (g + 1) * kp8;
  for (long long s = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; s < total;
       s += static_cast<long long>(gridDim.x) * blockDim.x) {
    const int c8 = static_cast<int>(s % kp8);
    const long long r = s / kp8, b = r / (g + 1);
    const int tok = static_cast<int>(r - b * (g + 1)) - 1;      // -1: CLS
    const int gy = tok / gw, gx = tok - gy * gw;
    uint32_t v[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      uint32_t pair = 0;
#pragma unroll
      for (int hlf = 0; hlf < 2; ++hlf) {
        const int col = c8 * 8 + 2 * e + hlf;
        if (tok >= 0 && col < k) {
          const int c = col / pp, rem = col - c * pp, dy = rem / p, dx = rem - dy * p;
          const long long pix =
              ((b * ch + c) * h + gy * p + dy) * static_cast<long long>(w) + gx * p + dx;
          pair |= static_cast<uint32_t>(img[pix]) << (16 * hlf);
        }
      }
      v[e] = pair;
    }
    out[s] = make_uint4(v[0], v[1], v[2], v[3]);
  }
}

// Even patch side (DINOv2's 14): one thread writes one 4-byte pixel pair of
// the K-padded patch matrix, consecutive threads consecutive pairs of a
// token row, so every store is coalesced; the pair (an even pair never
// straddles two patches) is read from the image, pad pairs and CLS rows are
// zero.  All counts fit in 31 bits (checked by the caller).
__global__ void patchify_even_kernel(const uint32_t* __restrict__ img, int batch, int ch, int h,
                                     int w, int p, int kpad, uint32_t* __restrict__ out) {
  pdl_trigger();
  pdl_wait();
  const int gw = w / p, gh = h / p, p2 = p / 2, row2 = p * p2, k2 = ch * row2, w2 = w / 2;
  const int kp2 = kpad / 2, g = gw * gh;
  // unsigned: the last stride may step past 2^31
  const uint32_t total = static_cast<uint32_t>(batch) * (g + 1) * kp2;
  for (uint32_t s = blockIdx.x * blockDim.x + threadIdx.x; s < total;
       s += gridDim.x * blockDim.x) {
    const int r = s / kp2, q = s - static_cast<uint32_t>(r) * kp2, b = r / (g + 1);
    const int tok = r - b * (g + 1) - 1;
    uint32_t v = 0u;
    if (tok >= 0 && q < k2) {
      const int c = q / row2, rem = q - c * row2, dy = rem / p2, e = rem - dy * p2;
      const int gy = tok / gw, gx = tok - gy * gw;
      v = __ldg(img + (static_cast<size_t>((b * ch + c) * h + gy * p + dy) * w2 + gx * p2 + e));
    }
    out[s] = v;
  }
}

// Piece s (8 columns) of w [d, k] padded with zero columns to [d, kpad].
__device__ __forceinline__ uint4 padded_piece(const uint16_t* __restrict__ w, int k, int kpad,
                                              long long s) {
  const int kp8 = kpad / 8, c8 = static_cast<int>(s % kp8);
  const uint16_t* row = w + (s / kp8) * k;
  uint32_t v[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const int j = c8 * 8 + 2 * e;
    v[e] = (j < k ? static_cast<uint32_t>(row[j]) : 0u) |
           (j + 1 < k ? static_cast<uint32_t>(row[j + 1]) << 16 : 0u);
  }
  return make_uint4(v[0], v[1], v[2], v[3]);
}

// The same relayout with the patch side and channel count fixed at compile
// time (DINOv2-B/14 on RGB), staged through shared memory: one block per
// band of patches (image b, patch row gy).  The band's CH x P image rows are
// read with coalesced 16-byte loads, then its gw token rows are written with
// coalesced 16-byte stores, each 8-column piece gathered from shared memory as
// four pixel pairs (P even: a pair never straddles two rows of a patch).  Needs
// w % 8 == 0.  The blocks past the bands pad the weights [d, CH P^2] for the
// GEMM, instead of a launch of their own.  128 images of 16 x 16 patches: 25.6 +
// 5.7 us as two kernels with 2-byte gathers -> 17.4 us, 4.9 TB/s.
template <int P, int CH>
__global__ void __launch_bounds__(256)
    patchify_band_kernel(const uint4* __restrict__ img, int batch, int gh, int gw, int h, int w,
                         uint4* __restrict__ out, const uint16_t* __restrict__ wt, int d,
                         uint4* __restrict__ wp) {
  static_assert(P % 2 == 0, "pixel pairs");
  extern __shared__ uint32_t band[];                   // [CH][P][w / 2]
  constexpr int kK = CH * P * P, kKp8 = (kK + 63) / 64 * 8;
  pdl_trigger();
  pdl_wait();
  const int bands = batch * gh;
  if (static_cast<int>(blockIdx.x) >= bands) {
    const long long s = (blockIdx.x - bands) * 256LL + threadIdx.x;
    if (s < static_cast<long long>(d) * kKp8) wp[s] = padded_piece(wt, kK, 8 * kKp8, s);
    return;
  }
  const int gy = blockIdx.x % gh, b = blockIdx.x / gh;
  const int w8 = w / 8, w2 = w / 2;
  uint4* band4 = reinterpret_cast<uint4*>(band);
  for (int i = threadIdx.x; i < CH * P * w8; i += blockDim.x) {
    const int x8 = i % w8, r = i / w8, dy = r % P, c = r / P;
    band4[i] = __ldg(img + (static_cast<size_t>((b * CH + c) * h + gy * P + dy) * w8 + x8));
  }
  uint4* dst = out + (static_cast<size_t>(b) * (gh * gw + 1) + 1 + gy * gw) * kKp8;
  if (gy == 0)
    for (int i = threadIdx.x; i < kKp8; i += blockDim.x) dst[i - kKp8] = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
  for (int i = threadIdx.x; i < gw * kKp8; i += blockDim.x) {
    const int gx = i / kKp8, c8 = i - gx * kKp8;
    uint32_t v[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int col = c8 * 8 + 2 * e;
      const int r = col / P, dx = col - r * P;         // r = c P + dy
      v[e] = col < kK ? band[r * w2 + (gx * P + dx) / 2] : 0u;
    }
    dst[i] = make_uint4(v[0], v[1], v[2], v[3]);
  }
}

// w [d, k] -> [d, kpad] with zero columns k..kpad-1 (the GEMM's B for K-padded patches).
__global__ void pad_cols_kernel(const uint16_t* __restrict__ w, int d, int k, int kpad,
                                uint4* __restrict__ out) {
  pdl_trigger();
  pdl_wait();
  const long long s = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
  if (s < static_cast<long long>(d) * (kpad / 8)) out[s] = padded_piece(w, k, kpad, s);
}

// LayerNorm of each image's CLS row (row cu[i]) into u [batch, dim]: one warp
// per image, fp32, biased variance.
__global__ void cls_ln_kernel(const uint16_t* __restrict__ x, const int32_t* __restrict__ cu,
                              int batch, int t_cap, int dim, const uint16_t* __restrict__ gam,
                              const uint16_t* __restrict__ bet, float eps,
                              uint16_t* __restrict__ u, int32_t* status) {
  pdl_trigger();
  pdl_wait();
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (warp >= batch) return;
  const int r = cu[warp];
  uint16_t* ur = u + static_cast<size_t>(warp) * dim;
  if (r < 0 || r >= t_cap || cu[warp + 1] <= r) {   // empty image or outside the buffer
    if (lane == 0 && (r < 0 || r > t_cap)) record_status(status, DORA_ERR_DEVICE_SEQLEN);
    for (int c = lane; c < dim; c += 32) ur[c] = 0;
    return;
  }
  const uint16_t* xr = x + static_cast<size_t>(r) * dim;
  float s = 0.f;
  for (int c = lane; c < dim; c += 32) s += __uint_as_float(static_cast<uint32_t>(xr[c]) << 16);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  const float mean = s / dim;
  float q = 0.f;
  for (int c = lane; c < dim; c += 32) {
    const float v = __uint_as_float(static_cast<uint32_t>(xr[c]) << 16) - mean;
    q += v * v;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
  const float rstd = rsqrtf(q / dim + eps);
  for (int c = lane; c < dim; c += 32) {
    const float v = (__uint_as_float(static_cast<uint32_t>(xr[c]) << 16) - mean) * rstd *
                        __uint_as_float(static_cast<uint32_t>(gam[c]) << 16) +
                    __uint_as_float(static_cast<uint32_t>(bet[c]) << 16);
    const __nv_bfloat16 hv = __float2bfloat16_rn(v);
    ur[c] = *reinterpret_cast<const uint16_t*>(&hv);
  }
}

// LC1 readout of one image per CTA: rows lo..hi-1 of x are layer-normalised
// (fp32, biased variance, row held in registers: dim <= 2048); the CLS row goes
// to u[i, 0:d], the others are summed per lane in registers and their mean goes to
// u[i, d:2d] (zero for an image without visual rows).
// Bound by the instructions and the shuffle chains of a row, not its bytes
// (256 images of 29 to 143 rows of 768: 34 MB, in L2): each warp takes two rows
// at a time, so that one row's shuffles cover the other's, in paired fp32, and
// keeps the centred row from the variance for the sum: 15.3 -> 11.8 us against one
// row at a time in scalar fp32 (16 warps of that: no faster).
constexpr int kLc1Warps = 8;
constexpr int kLc1MaxDim = 2048;

__device__ __forceinline__ uint64_t bf_pair(uint32_t w) { return f2_pack(lo_f(w), hi_f(w)); }
__device__ __forceinline__ float f2_sum(uint64_t v) {
  float a, b;
  f2_unpack(v, a, b);
  return a + b;
}

// kChunks = 16-byte pieces of a row per lane (dim <= 256 kChunks); R rows of a
// warp at a time.
template <int kChunks, int R>
__global__ void __launch_bounds__(kLc1Warps * 32)
    lc1_pool_kernel(const uint16_t* __restrict__ x, const int32_t* __restrict__ cu, int t_cap,
                    int dim, const uint16_t* __restrict__ gam, const uint16_t* __restrict__ bet,
                    float eps, uint16_t* __restrict__ u, int32_t* status) {
  extern __shared__ float acc[];                 // [kLc1Warps][dim]
  pdl_trigger();
  pdl_wait();
  const int img = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int d8 = dim / 8;
  const int lo = cu[img], hi = cu[img + 1];
  uint16_t* ur = u + static_cast<size_t>(img) * 2 * dim;
  const bool bad = lo < 0 || hi < lo || hi > t_cap;
  if (bad || hi == lo) {
    if (bad && threadIdx.x == 0) record_status(status, DORA_ERR_DEVICE_SEQLEN);
    for (int c = threadIdx.x; c < 2 * dim; c += blockDim.x) ur[c] = 0;
    return;
  }
  // Each lane owns the columns of its chunks c8 = lane + 32 i in every row,
  // so the visual rows' normalised values x^ = (x - mean) rstd are summed in
  // its registers; the affine map is applied once at the end, to the mean
  // (mean of g x^ + b = g mean(x^) + b).  Each warp walks rows lo + R warp ..
  // lo + R warp + R - 1 and on by R kLc1Warps; the next rows' loads are issued
  // before the current ones are reduced.
  uint64_t accr[kChunks][4];
#pragma unroll
  for (int i = 0; i < kChunks; ++i)
#pragma unroll
    for (int e = 0; e < 4; ++e) accr[i][e] = f2_pack(0.f, 0.f);
  uint4 nxt[R][kChunks];
  auto load_rows = [&](int j) {
#pragma unroll
    for (int k = 0; k < R; ++k) {
      const uint4* xr = reinterpret_cast<const uint4*>(x + static_cast<size_t>(j + k) * dim);
#pragma unroll
      for (int i = 0; i < kChunks; ++i) {
        const int c8 = lane + 32 * i;
        nxt[k][i] = (j + k < hi && c8 < d8) ? xr[c8] : make_uint4(0, 0, 0, 0);
      }
    }
  };
  // 1 / dim as the sum of two fp32 values, hi and what hi misses: with hi alone
  // (exact for few dims) 1.5e-4 of the means rounded to the wrong bf16 value at
  // dim 192 to 768, with both 1.1e-4, as with a division (0.7 us more a call).
  // An overflowed sum of squares stays infinite.
  const float fdim = static_cast<float>(dim), inv_hi = 1.f / fdim;
  const float inv_lo = fmaf(-inv_hi, fdim, 1.f) * inv_hi;
  auto over_dim = [&](float v) { return fmaf(v, inv_hi, fminf(v, FLT_MAX) * inv_lo); };
  load_rows(lo + R * warp);
  for (int j = lo + R * warp; j < hi; j += R * kLc1Warps) {
    uint64_t v[R][kChunks][4];
    float s[R];
#pragma unroll
    for (int k = 0; k < R; ++k) {
      uint64_t t = f2_pack(0.f, 0.f);
#pragma unroll
      for (int i = 0; i < kChunks; ++i) {
        const uint32_t w[4] = {nxt[k][i].x, nxt[k][i].y, nxt[k][i].z, nxt[k][i].w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          v[k][i][e] = bf_pair(w[e]);
          t = f2_add(t, v[k][i][e]);
        }
      }
      s[k] = f2_sum(t);
    }
    load_rows(j + R * kLc1Warps);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int k = 0; k < R; ++k) s[k] += __shfl_xor_sync(0xffffffffu, s[k], o);
    float q[R];
#pragma unroll
    for (int k = 0; k < R; ++k) {
      const float nm = -over_dim(s[k]);
      const uint64_t NM = f2_pack(nm, nm);
      uint64_t t = f2_pack(0.f, 0.f);
#pragma unroll
      for (int i = 0; i < kChunks; ++i) {
        if (lane + 32 * i >= d8) continue;             // (its pieces stay zero)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          v[k][i][e] = f2_add(v[k][i][e], NM);
          t = f2_fma(v[k][i][e], v[k][i][e], t);
        }
      }
      q[k] = f2_sum(t);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int k = 0; k < R; ++k) q[k] += __shfl_xor_sync(0xffffffffu, q[k], o);
#pragma unroll
    for (int k = 0; k < R; ++k) {
      if (j + k >= hi) continue;
      const float rstd = rsqrtf(over_dim(q[k]) + eps);
      if (j + k == lo) {                                 // CLS row: LN(x) itself
#pragma unroll
        for (int i = 0; i < kChunks; ++i) {
          const int c8 = lane + 32 * i;
          if (c8 >= d8) continue;
          const uint4 g4 = reinterpret_cast<const uint4*>(gam)[c8];
          const uint4 b4 = reinterpret_cast<const uint4*>(bet)[c8];
          const uint32_t gv[4] = {g4.x, g4.y, g4.z, g4.w}, bv[4] = {b4.x, b4.y, b4.z, b4.w};
          uint32_t o[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            float a, b;
            f2_unpack(v[k][i][e], a, b);
            o[e] = pack2(a * rstd * lo_f(gv[e]) + lo_f(bv[e]), b * rstd * hi_f(gv[e]) + hi_f(bv[e]));
          }
          reinterpret_cast<uint4*>(ur)[c8] = make_uint4(o[0], o[1], o[2], o[3]);
        }
      } else {
        const uint64_t RS = f2_pack(rstd, rstd);
#pragma unroll
        for (int i = 0; i < kChunks; ++i)
#pragma unroll
          for (int e = 0; e < 4; ++e) accr[i][e] = f2_fma(v[k][i][e], RS, accr[i][e]);
      }
    }
  }
#pragma unroll
  for (int i = 0; i < kChunks; ++i) {
    const int c8 = lane + 32 * i;
    if (c8 >= d8) continue;
    float f[8];
#pragma unroll
    for (int e = 0; e < 4; ++e) f2_unpack(accr[i][e], f[2 * e], f[2 * e + 1]);
    float4* dst = reinterpret_cast<float4*>(acc + warp * dim + c8 * 8);
    dst[0] = make_float4(f[0], f[1], f[2], f[3]);
    dst[1] = make_float4(f[4], f[5], f[6], f[7]);
  }
  __syncthreads();
  const int n_vis = hi - lo - 1;
  const float inv = n_vis > 0 ? 1.f / static_cast<float>(n_vis) : 0.f;
  for (int c = threadIdx.x; c < dim; c += blockDim.x) {
    float t = 0.f;
#pragma unroll
    for (int wp = 0; wp < kLc1Warps; ++wp) t += acc[wp * dim + c];
    const float g = __uint_as_float(static_cast<uint32_t>(gam[c]) << 16);
    const float b = __uint_as_float(static_cast<uint32_t>(bet[c]) << 16);
    const __nv_bfloat16 hv = __float2bfloat16_rn(n_vis > 0 ? t * inv * g + b : 0.f);
    ur[dim + c] = *reinterpret_cast<const uint16_t*>(&hv);
  }
}

// LayerScale fold: out[i, :] = bf16(gamma_i * w[i, :]) and bout[i] =
// bf16(gamma_i * b_i).  A product of two bf16 values is exact in fp32, so each
// output is the round-to-nearest-even of the exact product.
__global__ void layerscale_fold_kernel(const uint4* __restrict__ w, const uint16_t* __restrict__ b,
                                       const uint16_t* __restrict__ gam, int n, int k8,
                                       uint4* __restrict__ out, uint16_t* __restrict__ bout) {
  const long long total = static_cast<long long>(n) * k8;
  for (long long s = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; s < total;
       s += static_cast<long long>(gridDim.x) * blockDim.x) {
    const int row = static_cast<int>(s / k8);
    const float g = __uint_as_float(static_cast<uint32_t>(gam[row]) << 16);
    const uint4 v = w[s];
    out[s] = make_uint4(pack2(g * lo_f(v.x), g * hi_f(v.x)), pack2(g * lo_f(v.y), g * hi_f(v.y)),
                        pack2(g * lo_f(v.z), g * hi_f(v.z)), pack2(g * lo_f(v.w), g * hi_f(v.w)));
    if (b != nullptr && s % k8 == 0) {
      const __nv_bfloat16 hv = __float2bfloat16_rn(g * __uint_as_float(
                                                           static_cast<uint32_t>(b[row]) << 16));
      bout[row] = *reinterpret_cast<const uint16_t*>(&hv);
    }
  }
}

size_t up256(size_t v) { return (v + 255) & ~static_cast<size_t>(255); }

int grid_for(long long work) {
  const long long g = (work + 255) / 256;
  return static_cast<int>(g < 152LL * 16 ? (g > 0 ? g : 1) : 152LL * 16);
}

}  // namespace embed
}  // namespace dora

using namespace dora;

extern "C" {

size_t dora_embed_workspace_size(int32_t batch, int32_t channels, int32_t height, int32_t width,
                                 int32_t patch, int32_t dim) {
  if (batch < 0 || channels <= 0 || patch <= 0 || height <= 0 || width <= 0 || dim <= 0) return 0;
  const size_t tok = static_cast<size_t>(batch) * (height / patch) * (width / patch);
  const size_t k = static_cast<size_t>(channels) * patch * patch, kpad = (k + 63) / 64 * 64;
  const size_t wp = kpad != k ? embed::up256(static_cast<size_t>(dim) * kpad * 2) : 0;
  // the patch matrix with its CLS rows, or the patches and their embeddings: what the
  // size has always held, and what its callers and tests count on
  const size_t now = embed::up256((tok + batch) * kpad * 2);
  const size_t was = embed::up256(tok * kpad * 2) + embed::up256(tok * dim * 2);
  return 256 + (now > was ? now : was) + wp;
}

int dora_patch_embed(const dora_bf16* images, int32_t batch, int32_t channels, int32_t height,
                     int32_t width, int32_t patch, int32_t dim, const dora_bf16* w_pe,
                     const dora_bf16* b_pe, const dora_bf16* cls, const dora_bf16* pos,
                     dora_bf16* x0, void* workspace, size_t workspace_bytes,
                     dora_stream_t stream_) {
  if (batch < 0 || batch > 65535 || channels <= 0 || channels > 64 || patch <= 0 ||
      patch > 64 || height <= 0 || width <= 0 || height % patch != 0 || width % patch != 0 ||
      dim <= 0 || dim % 64 != 0 || dim > (1 << 16))
    return DORA_ERR_INVALID_ARG;
  const void* req[] = {images, w_pe, cls, pos, x0, workspace};
  for (const void* p : req)
    if (p == nullptr || (reinterpret_cast<uintptr_t>(p) & 15u) != 0) return DORA_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(b_pe) & 15u) != 0) return DORA_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return DORA_ERR_INVALID_ARG;
  if (workspace_bytes < dora_embed_workspace_size(batch, channels, height, width, patch, dim))
    return DORA_ERR_INVALID_ARG;
  const long long g = static_cast<long long>(height / patch) * (width / patch);
  const long long tok = static_cast<long long>(batch) * g;
  if (tok > (1 << 30)) return DORA_ERR_INVALID_ARG;
  const int dev = checked_device();
  if (dev == -1) return DORA_ERR_CUDA;
  if (dev < 0) return DORA_ERR_UNSUPPORTED;
  if (batch == 0) return DORA_OK;
  cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  int32_t* status = reinterpret_cast<int32_t*>(ws);
  const int k = channels * patch * patch, kpad = (k + 63) / 64 * 64;
  const long long rows = tok + batch;                  // a token row and a patch row each
  uint16_t* patches = reinterpret_cast<uint16_t*>(ws + 256);
  const uint16_t* w_gemm = w_pe;
  const long long pixels = static_cast<long long>(batch) * channels * height * width;
  if (patch % 8 == 0 && kpad == k && pixels < (1LL << 31) && rows * (k / 8) < (1LL << 31)) {
    const int v = patch % 16 == 0 ? 2 : 1;
    const long long items = pixels / (8 * v) + static_cast<long long>(batch) * (k / 8 / v);
    if (launch_pdl(v == 2 ? embed::patchify_kernel<2> : embed::patchify_kernel<1>,
                   dim3(embed::grid_for(items)), dim3(256), 0, stream,
                   reinterpret_cast<const uint4*>(images), batch, channels, height, width, patch,
                   reinterpret_cast<uint4*>(patches)) != cudaSuccess)
      return DORA_ERR_CUDA;
  } else {
    // K padded to a multiple of the GEMM's 64-wide K step: zero patch columns
    // and a zero-padded copy of the weights in the workspace
    uint16_t* wp = reinterpret_cast<uint16_t*>(ws + 256 + embed::up256(rows * kpad * 2));
    const long long items = rows * (kpad / 2), pieces = static_cast<long long>(dim) * (kpad / 8);
    const int band_smem = 3 * 14 * width * 2;
    bool padded = kpad == k;
    if (patch == 14 && channels == 3 && width % 8 == 0 && band_smem <= 160 * 1024 &&
        static_cast<long long>(batch) * (height / patch) + (pieces + 255) / 256 < (1LL << 31)) {
      auto kern = embed::patchify_band_kernel<14, 3>;
      if (band_smem > 48 * 1024 &&
          cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, band_smem) !=
              cudaSuccess)
        return DORA_ERR_CUDA;
      if (launch_pdl(kern,
                     dim3(static_cast<unsigned>(batch * (height / patch) + (pieces + 255) / 256)),
                     dim3(256), static_cast<size_t>(band_smem), stream,
                     reinterpret_cast<const uint4*>(images), batch, height / patch, width / patch,
                     height, width, reinterpret_cast<uint4*>(patches), w_pe, dim,
                     reinterpret_cast<uint4*>(wp)) != cudaSuccess)
        return DORA_ERR_CUDA;
      padded = true;
    } else if (patch % 2 == 0 && items < (1LL << 31) && pixels / 2 < (1LL << 31)) {
      if (launch_pdl(embed::patchify_even_kernel, dim3(embed::grid_for(items)), dim3(256), 0,
                     stream, reinterpret_cast<const uint32_t*>(images), batch, channels, height,
                     width, patch, kpad, reinterpret_cast<uint32_t*>(patches)) != cudaSuccess)
        return DORA_ERR_CUDA;
    } else {
      if (launch_pdl(embed::patchify_any_kernel, dim3(embed::grid_for(rows * (kpad / 8))),
                     dim3(256), 0, stream, images, batch, channels, height, width, patch, kpad,
                     reinterpret_cast<uint4*>(patches)) != cudaSuccess)
        return DORA_ERR_CUDA;
    }
    if (!padded && launch_pdl(embed::pad_cols_kernel,
                              dim3(static_cast<unsigned>((pieces + 255) / 256)), dim3(256), 0,
                              stream, w_pe, dim, k, kpad, reinterpret_cast<uint4*>(wp)) !=
                       cudaSuccess)
      return DORA_ERR_CUDA;
    if (kpad != k) w_gemm = wp;
  }
  // tokens: the convolution with bias, CLS and position embeddings in the epilogue
  LinearEpi ep;
  ep.bias = b_pe;
  ep.cls = cls;
  ep.pos = pos;
  ep.tokens = static_cast<int32_t>(g + 1);
  return launch_linear(patches, static_cast<int32_t>(rows), nullptr, kpad, w_gemm, dim, kEpiTokens,
                       ep, x0, status, stream) == cudaSuccess
             ? DORA_OK
             : DORA_ERR_CUDA;
}

size_t dora_head_workspace_size(int32_t batch, int32_t dim) {
  if (batch < 0 || dim <= 0) return 0;
  return 256 + embed::up256(static_cast<size_t>(batch) * dim * 2);
}

int dora_classifier_head(const dora_bf16* x, const int32_t* cu, int32_t batch, int32_t t_cap,
                         int32_t dim, const dora_bf16* norm_w, const dora_bf16* norm_b,
                         float eps, const dora_bf16* w_head, const dora_bf16* b_head,
                         int32_t classes, dora_bf16* logits, void* workspace,
                         size_t workspace_bytes, dora_stream_t stream_) {
  if (batch < 0 || batch > 65535 || t_cap < 0 || dim <= 0 || dim % 64 != 0 ||
      dim > (1 << 16) || classes <= 0 || classes % 32 != 0 || classes > (1 << 16) ||
      !(eps >= 0.f))
    return DORA_ERR_INVALID_ARG;
  const void* req[] = {x, cu, norm_w, norm_b, w_head, logits, workspace};
  for (const void* p : req)
    if (p == nullptr) return DORA_ERR_INVALID_ARG;
  const void* al[] = {x, norm_w, norm_b, w_head, b_head, logits};
  for (const void* p : al)
    if ((reinterpret_cast<uintptr_t>(p) & 15u) != 0) return DORA_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0 ||
      workspace_bytes < dora_head_workspace_size(batch, dim))
    return DORA_ERR_INVALID_ARG;
  const int dev = checked_device();
  if (dev == -1) return DORA_ERR_CUDA;
  if (dev < 0) return DORA_ERR_UNSUPPORTED;
  if (batch == 0) return DORA_OK;
  cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  int32_t* status = reinterpret_cast<int32_t*>(ws);
  uint16_t* u = reinterpret_cast<uint16_t*>(ws + 256);
  if (launch_pdl(embed::cls_ln_kernel, dim3((batch + 7) / 8), dim3(256), 0, stream, x, cu, batch,
                 t_cap, dim, norm_w, norm_b, eps, u, status) != cudaSuccess)
    return DORA_ERR_CUDA;
  LinearEpi ep;
  ep.bias = b_head;
  return launch_linear(u, batch, nullptr, dim, w_head, classes, DORA_EPI_BIAS, ep, logits, status,
                       stream) == cudaSuccess
             ? DORA_OK
             : DORA_ERR_CUDA;
}

size_t dora_head_lc1_workspace_size(int32_t batch, int32_t dim) {
  if (batch < 0 || dim <= 0) return 0;
  return 256 + embed::up256(static_cast<size_t>(batch) * 2 * dim * 2);
}

int dora_classifier_head_lc1(const dora_bf16* x, const int32_t* cu, int32_t batch, int32_t t_cap,
                             int32_t dim, const dora_bf16* norm_w, const dora_bf16* norm_b,
                             float eps, const dora_bf16* w_head, const dora_bf16* b_head,
                             int32_t classes, dora_bf16* logits, void* workspace,
                             size_t workspace_bytes, dora_stream_t stream_) {
  if (batch < 0 || batch > 65535 || t_cap < 0 || dim <= 0 || dim % 64 != 0 ||
      dim > embed::kLc1MaxDim || classes <= 0 || classes % 32 != 0 || classes > (1 << 16) ||
      !(eps >= 0.f))
    return DORA_ERR_INVALID_ARG;
  const void* req[] = {x, cu, norm_w, norm_b, w_head, logits, workspace};
  for (const void* p : req)
    if (p == nullptr) return DORA_ERR_INVALID_ARG;
  const void* al[] = {x, norm_w, norm_b, w_head, b_head, logits};
  for (const void* p : al)
    if ((reinterpret_cast<uintptr_t>(p) & 15u) != 0) return DORA_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0 ||
      workspace_bytes < dora_head_lc1_workspace_size(batch, dim))
    return DORA_ERR_INVALID_ARG;
  const int dev = checked_device();
  if (dev == -1) return DORA_ERR_CUDA;
  if (dev < 0) return DORA_ERR_UNSUPPORTED;
  if (batch == 0) return DORA_OK;
  cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  int32_t* status = reinterpret_cast<int32_t*>(ws);
  uint16_t* u = reinterpret_cast<uint16_t*>(ws + 256);
  const int smem = embed::kLc1Warps * dim * 4;
  const int chunks = (dim / 8 + 31) / 32;
  auto kern = chunks <= 1   ? embed::lc1_pool_kernel<1, 2>
              : chunks <= 2 ? embed::lc1_pool_kernel<2, 2>
              : chunks <= 3 ? embed::lc1_pool_kernel<3, 2>
              : chunks <= 4 ? embed::lc1_pool_kernel<4, 2>
                            : embed::lc1_pool_kernel<8, 1>;
  if (smem > 48 * 1024 &&
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) !=
          cudaSuccess)
    return DORA_ERR_CUDA;
  if (launch_pdl(kern, dim3(batch), dim3(embed::kLc1Warps * 32), static_cast<size_t>(smem), stream,
                 x, cu, t_cap, dim, norm_w, norm_b, eps, u, status) != cudaSuccess)
    return DORA_ERR_CUDA;
  LinearEpi ep;
  ep.bias = b_head;
  return launch_linear(u, batch, nullptr, 2 * dim, w_head, classes, DORA_EPI_BIAS, ep, logits,
                       status, stream) == cudaSuccess
             ? DORA_OK
             : DORA_ERR_CUDA;
}

int dora_fold_layerscale(const dora_bf16* w, const dora_bf16* b, const dora_bf16* gamma,
                         int32_t n, int32_t k, dora_bf16* w_out, dora_bf16* b_out,
                         dora_stream_t stream_) {
  if (n <= 0 || k <= 0 || k % 8 != 0 || static_cast<long long>(n) * k > (1LL << 34))
    return DORA_ERR_INVALID_ARG;
  const void* al[] = {w, gamma, w_out};
  for (const void* p : al)
    if (p == nullptr || (reinterpret_cast<uintptr_t>(p) & 15u) != 0) return DORA_ERR_INVALID_ARG;
  if ((b == nullptr) != (b_out == nullptr)) return DORA_ERR_INVALID_ARG;
  const int dev = checked_device();
  if (dev == -1) return DORA_ERR_CUDA;
  if (dev < 0) return DORA_ERR_UNSUPPORTED;
  cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
  embed::layerscale_fold_kernel<<<embed::grid_for(static_cast<long long>(n) * (k / 8)), 256, 0,
                                  stream>>>(reinterpret_cast<const uint4*>(w), b, gamma, n, k / 8,
                                            reinterpret_cast<uint4*>(w_out), b_out);
  return cudaGetLastError() == cudaSuccess ? DORA_OK : DORA_ERR_CUDA;
}

}  // extern "C"
