// The actor's encoder after its attention, in one kernel per 128-row tile:
//   Z1 = X + W_o O + b_o
//   Z  = Z1 + W_2 GELU(W_1 LayerNorm(Z1) + b_1) + b_2      (128 -> 256 -> 128)
//   S1 = W_s Z + b_s                                       (128 -> 64, the selector's first layer)
// O, X and Z are bf16 [rows, 128], S1 bf16 [rows, 64]; the LayerNorm is folded
// into W_1 (rstd (Z1 W_1'^T - mean c) + d, the moments from the rounded Z1).
//
// All four weights (176 KB) are loaded once per CTA and stay in shared memory
// beside one O tile; everything between the products stays on the SM: Z1, the
// GELU's output and Z go back into tensor memory as the next product's A
// operand, so of the intermediates only Z and S1 reach global memory.
//   warp 0      loads the weights, then each tile's O once the tile before it is
//               through its first product
//   warp 1      issues the four products of a tile
//   warp 2      tensor-memory allocation
//   warps 4-11  epilogues: two threads a row, half of its columns each; the two
//               halves' slice moments meet in shared memory
// Tensor memory: 0-127 the accumulators of W_o and W_2, 128-383 that of W_1,
// under which the GELU's output is written (columns 128 h + 64 of half h) and
// then the selector's accumulator, 384-447 Z1, then Z, as bf16.
//
// What bounds it: the chain of four products and epilogues of a tile, about
// 15,500 cycles (the GELU 4,300, the waits for the products 3,500 to 4,900, the
// other epilogues and the loads of X the rest), run 2.6 times by each SM at 256 x 197 tokens; the traffic (46 MB) would
// take 7 us.  As five launches (output projection, moments merge, fc1, fc2,
// selector linear), whose K = 128 tiles are all prologue and epilogue, the same
// took 60 us of device time, here 31; in the stream the actor's call went from
// 153.3 to 135.1 us, at 8 images of 384 columns from 71.4 to 55.6.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "dora_ptx.cuh"
#include "epilogue_math.cuh"
#include "token_ops.cuh"

namespace dora {
namespace actor_tail {

constexpr int BM = 128;
constexpr int W = 128;          // encoder width
constexpr int FF = 256;
constexpr int SH = 64;
constexpr int kThreads = 384;
constexpr int kEpiWarp0 = 4;
constexpr int kEpiWarps = 8;
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kD1 = 0, kD2 = 128, kZ = 384;

struct Smem {
  uint16_t o[2][BM * 64];       // a 64-column block of the O tile each, 128-byte swizzle
  uint16_t wo[2][W * 64];       // 64-column blocks of the weights
  uint16_t w1[2][FF * 64];
  uint16_t w2[4][W * 64];
  uint16_t ws[2][SH * 64];
  float c1[FF], d1[FF];         // folded LayerNorm of W_1
  float2 half_moments[2][BM];   // slice moments of Z1's two halves
  uint64_t w_full, o_full;
  uint64_t d_full[4];           // product i of the tile done
  uint64_t ready[3];            // Z1, GELU output, Z in tensor memory (one arrival a warp)
  uint64_t drain;
  uint32_t tmem_base;
  int abort_flag;
  int o_issued;
};
static_assert(sizeof(Smem) <= 227 * 1024, "shared memory");

struct Maps {
  CUtensorMap o, wo, w1, w2, ws;
};

// 32 packed values as two 16-column stores.
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
  tmem_st16(taddr, *reinterpret_cast<const uint32_t(*)[16]>(&r[0]));
  tmem_st16(taddr + 16, *reinterpret_cast<const uint32_t(*)[16]>(&r[16]));
}

// N packed values (16-byte aligned) to global memory, 32 bytes a store where
// `wide` says that the rows allow it.
template <int N>
__device__ __forceinline__ void store_row(uint16_t* p, const uint32_t (&r)[N], bool wide) {
  uint32_t* const d = reinterpret_cast<uint32_t*>(p);
  if (wide) {
#pragma unroll
    for (int j = 0; j < N; j += 8) st_global_32(d + j, &r[j]);
  } else {
#pragma unroll
    for (int j = 0; j < N; j += 4)
      *reinterpret_cast<uint4*>(d + j) = make_uint4(r[j], r[j + 1], r[j + 2], r[j + 3]);
  }
}

// A product of K = 16 * steps with A in tensor memory: 64-column blocks of B,
// `rows` rows each.  a_of(step) gives the column of the step's A.
template <int STEPS, int N, class AOf>
__device__ __forceinline__ void product_ts(uint32_t d, AOf a_of, const uint16_t* b) {
  constexpr uint32_t idesc = idesc_bf16(BM, N, false);
#pragma unroll
  for (int k = 0; k < STEPS; ++k)
    mma_bf16_ts(d, a_of(k), sdesc_sw128(smem_u32(b + (k / 4) * N * 64), 16, 1024) + 2 * (k % 4),
                idesc, k > 0 ? 1u : 0u);
}

__global__ void __launch_bounds__(kThreads, 1)
    actor_tail_kernel(const __grid_constant__ Maps mp, const TailArgs a, int m_cap,
                      const int32_t* __restrict__ m_dev, int32_t* status) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  pdl_trigger();
  if (smem_u32(smem_raw) & 1023u) {           // swizzled tiles need 1 KB alignment
    pdl_wait();
    if (threadIdx.x == 0) record_status(status, DORA_ERR_UNSUPPORTED);
    return;
  }
  Smem& s = *reinterpret_cast<Smem*>(smem_raw);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    mbar_init(&s.w_full, 1);
    mbar_init(&s.o_full, 1);
    for (int i = 0; i < 4; ++i) mbar_init(&s.d_full[i], 1);
    for (int i = 0; i < 3; ++i) mbar_init(&s.ready[i], kEpiWarps);
    mbar_init(&s.drain, 1);
    s.abort_flag = 0;
    s.o_issued = 0;
    fence_barrier_init();
  }
  if (warp == 2) tmem_alloc(&s.tmem_base, kTmemCols);
  // the set-up above overlaps the previous kernel; global memory waits for it
  pdl_wait();
  for (int i = threadIdx.x; i < FF; i += kThreads) {
    s.c1[i] = a.c1[i];
    s.d1[i] = a.d1[i];
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  int M = *m_dev;
  M = M < 0 ? 0 : (M > m_cap ? m_cap : M);
  const int tiles = (M + BM - 1) / BM;
  const uint32_t tmem = s.tmem_base;
  volatile int* abort = &s.abort_flag;

  if (warp == 0) {
    if (elect_one() && static_cast<int>(blockIdx.x) < tiles) {
      mbar_arrive_expect_tx(&s.w_full, sizeof(s.wo) + sizeof(s.w1) + sizeof(s.w2) + sizeof(s.ws));
      for (int k = 0; k < 2; ++k) tma_load_2d(s.wo[k], &mp.wo, &s.w_full, 64 * k, 0);
      for (int k = 0; k < 2; ++k) tma_load_2d(s.w1[k], &mp.w1, &s.w_full, 64 * k, 0);
      for (int k = 0; k < 4; ++k) tma_load_2d(s.w2[k], &mp.w2, &s.w_full, 64 * k, 0);
      for (int k = 0; k < 2; ++k) tma_load_2d(s.ws[k], &mp.ws, &s.w_full, 64 * k, 0);
      int it = 0;
      for (int t = blockIdx.x; t < tiles; t += gridDim.x, ++it) {
        if (it > 0 && !mbar_wait(&s.d_full[0], (it - 1) & 1, abort)) break;
        mbar_arrive_expect_tx(&s.o_full, sizeof(s.o));
        for (int k = 0; k < 2; ++k) tma_load_2d(s.o[k], &mp.o, &s.o_full, 64 * k, t * BM);
        s.o_issued = it + 1;
      }
    }
  } else if (warp == 1) {
    if (elect_one() && static_cast<int>(blockIdx.x) < tiles) {
      bool ok = mbar_wait(&s.w_full, 0, abort);
      int it = 0;
      for (int t = blockIdx.x; ok && t < tiles; t += gridDim.x, ++it) {
        const uint32_t ph = it & 1;
        // every accumulator's earlier contents were read before the arrivals
        // that the product before it waited for
        if (!(ok = mbar_wait(&s.o_full, ph, abort))) break;
        tc_fence_after();
        constexpr uint32_t id1 = idesc_bf16(BM, W, false);
#pragma unroll
        for (int k = 0; k < W / 16; ++k)
          mma_bf16_ss(tmem + kD1, sdesc_sw128(smem_u32(s.o[k / 4]), 16, 1024) + 2 * (k % 4),
                      sdesc_sw128(smem_u32(s.wo[k / 4]), 16, 1024) + 2 * (k % 4), id1,
                      k > 0 ? 1u : 0u);
        mma_commit(&s.d_full[0]);
        if (!(ok = mbar_wait(&s.ready[0], ph, abort))) break;
        tc_fence_after();
        product_ts<W / 16, FF>(tmem + kD2, [&](int k) { return tmem + kZ + 8u * k; }, s.w1[0]);
        mma_commit(&s.d_full[1]);
        if (!(ok = mbar_wait(&s.ready[1], ph, abort))) break;
        tc_fence_after();
        product_ts<FF / 16, W>(
            tmem + kD1, [&](int k) { return tmem + kD2 + 128u * (k / 8) + 8u * (k % 8); }, s.w2[0]);
        mma_commit(&s.d_full[2]);
        if (!(ok = mbar_wait(&s.ready[2], ph, abort))) break;
        tc_fence_after();
        product_ts<W / 16, SH>(tmem + kD2, [&](int k) { return tmem + kZ + 8u * k; }, s.ws[0]);
        mma_commit(&s.d_full[3]);
      }
      mma_commit(&s.drain);
      mbar_wait_limited(&s.drain, 0, kWaitLimitNs);
    }
  } else if (warp >= kEpiWarp0) {
    const int quarter = warp & 3, half = (warp - kEpiWarp0) >> 2;
    const int r = quarter * 32 + lane;
    const uint32_t lanes = tmem + (static_cast<uint32_t>(quarter * 32) << 16);
    const bool wide =
        ((reinterpret_cast<uintptr_t>(a.z) | reinterpret_cast<uintptr_t>(a.s1)) & 31u) == 0;
    const int c0 = 64 * half;                  // this thread's columns of a 128-wide row
    int it = 0;
    for (int t = blockIdx.x; t < tiles; t += gridDim.x, ++it) {
      const uint32_t ph = it & 1;
      const int row = t * BM + r;
      const bool live = row < M;
      // Z1 = X + O W_o^T + b_o, rounded
      uint4 x[8];
#pragma unroll
      for (int j = 0; j < 8; ++j)
        x[j] = live ? __ldg(reinterpret_cast<const uint4*>(a.x + static_cast<size_t>(row) * W + c0) + j)
                    : make_uint4(0u, 0u, 0u, 0u);
      uint32_t z1[32];
      float v[32];
      if (!mbar_wait_warp(&s.d_full[0], ph, abort)) break;
      tc_fence_after();
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint32_t acc[32];
        tmem_ld32(lanes + kD1 + c0 + 32 * h, acc);
        tmem_ld_wait();
#pragma unroll
        for (int e = 0; e < 32; ++e) v[e] = __uint_as_float(acc[e]);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          add_bf16x8(v + 8 * j, __ldg(reinterpret_cast<const uint4*>(a.bo + c0 + 32 * h) + j));
          add_bf16x8(v + 8 * j, x[4 * h + j]);
        }
        pack_row(v, *reinterpret_cast<uint32_t(*)[16]>(&z1[16 * h]));
      }
      const float2 mine = slice_moments(*reinterpret_cast<const uint32_t(*)[16]>(&z1[0]),
                                        *reinterpret_cast<const uint32_t(*)[16]>(&z1[16]));
      s.half_moments[half][r] = mine;
      tmem_st32(lanes + kZ + 32 * half, z1);
      tmem_st_wait();
      warp_arrive(&s.ready[0]);
      // GELU(W_1 LayerNorm(Z1) + b_1), over the accumulator columns already read
      if (!mbar_wait_warp(&s.ready[0], ph, abort)) break;
      const float2 other = s.half_moments[half ^ 1][r];
      const float2 lo = half ? other : mine, hi = half ? mine : other;
      const float2 mv = merge_two_slices(lo, hi);
      const float neg_mean = -mv.x, rstd = rsqrtf(mv.y + a.eps);
      if (!mbar_wait_warp(&s.d_full[1], ph, abort)) break;
      tc_fence_after();
#pragma unroll 1
      for (int i = 0; i < 4; ++i) {
        const int c = 128 * half + 32 * i;
        uint32_t acc[32], o[16];
        tmem_ld32(lanes + kD2 + c, acc);
        tmem_ld_wait();
#pragma unroll
        for (int e = 0; e < 32; ++e) v[e] = __uint_as_float(acc[e]);
        fold_layernorm(v, neg_mean, rstd, s.c1 + c, s.d1 + c);
#pragma unroll
        for (int e = 0; e < 32; e += 2) gelu_erf2(v[e], v[e + 1]);
        pack_row(v, o);
        tmem_st16(lanes + kD2 + 128 * half + 16 * i, o);
      }
      tmem_st_wait();
      warp_arrive(&s.ready[1]);
      // Z = Z1 + F W_2^T + b_2
      if (!mbar_wait_warp(&s.d_full[2], ph, abort)) break;
      tc_fence_after();
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint32_t acc[32];
        tmem_ld32(lanes + kD1 + c0 + 32 * h, acc);
        tmem_ld_wait();
#pragma unroll
        for (int e = 0; e < 32; ++e) v[e] = __uint_as_float(acc[e]);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          add_bf16x8(v + 8 * j, __ldg(reinterpret_cast<const uint4*>(a.b2 + c0 + 32 * h) + j));
          add_bf16x8(v + 8 * j, make_uint4(z1[16 * h + 4 * j], z1[16 * h + 4 * j + 1],
                                           z1[16 * h + 4 * j + 2], z1[16 * h + 4 * j + 3]));
        }
        pack_row(v, *reinterpret_cast<uint32_t(*)[16]>(&z1[16 * h]));
      }
      tmem_st32(lanes + kZ + 32 * half, z1);
      tmem_st_wait();
      warp_arrive(&s.ready[2]);
      if (live) store_row(a.z + static_cast<size_t>(row) * W + c0, z1, wide);
      // S1 = Z W_s^T + b_s
      if (!mbar_wait_warp(&s.d_full[3], ph, abort)) break;
      tc_fence_after();
      {
        uint32_t acc[32], o[16];
        tmem_ld32(lanes + kD2 + 32 * half, acc);
        tmem_ld_wait();
#pragma unroll
        for (int e = 0; e < 32; ++e) v[e] = __uint_as_float(acc[e]);
#pragma unroll
        for (int j = 0; j < 4; ++j)
          add_bf16x8(v + 8 * j, __ldg(reinterpret_cast<const uint4*>(a.bs + 32 * half) + j));
        pack_row(v, o);
        if (live) store_row(a.s1 + static_cast<size_t>(row) * SH + 32 * half, o, wide);
      }
    }
  }

  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (*abort) {
    if (threadIdx.x == 0) {
      record_status(status, DORA_ERR_TIMEOUT);
      // let the loads in flight land
      if (static_cast<int>(blockIdx.x) < tiles) mbar_wait_limited(&s.w_full, 0, 100ull * 1000 * 1000);
      if (s.o_issued > 0)
        mbar_wait_limited(&s.o_full, (s.o_issued - 1) & 1, 100ull * 1000 * 1000);
    }
    __syncthreads();
  }
  if (warp == 2) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

}  // namespace actor_tail

cudaError_t launch_actor_tail(const uint16_t* o, const uint16_t* wo, const uint16_t* w1,
                              const uint16_t* w2, const uint16_t* ws, const TailArgs& args,
                              int32_t m_cap, const int32_t* m_dev, int32_t* status,
                              cudaStream_t stream) {
  using namespace actor_tail;
  if (m_cap == 0) return cudaSuccess;
  Maps mp;
  auto map = [](CUtensorMap* m, const uint16_t* p, uint64_t cols, uint64_t rows, uint32_t box) {
    return encode_tmap_2d_bf16(m, p, cols, rows, cols * 2, 64, box) == 0;
  };
  if (!map(&mp.o, o, W, static_cast<uint64_t>(m_cap), BM) || !map(&mp.wo, wo, W, W, W) ||
      !map(&mp.w1, w1, W, FF, FF) || !map(&mp.w2, w2, FF, W, W) || !map(&mp.ws, ws, W, SH, SH))
    return cudaErrorInvalidValue;
  const cudaError_t e =
      cudaFuncSetAttribute(actor_tail_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           static_cast<int>(sizeof(Smem)));
  if (e != cudaSuccess) return e;
  const int tiles = (m_cap + BM - 1) / BM, cap = num_sms();
  return launch_pdl(actor_tail_kernel, dim3(tiles < cap ? tiles : cap), dim3(kThreads),
                    sizeof(Smem), stream, mp, args, m_cap, m_dev, status);
}

}  // namespace dora
