// The actor's encoder before its attention, in one kernel per 128-row tile:
//   X   = W_in K + b_in + e^C_l (+ W_h h_l on the CLS rows)       (d -> 128)
//   QKV = W_qkv LayerNorm1(X) + b_qkv                             (128 -> 384)
// K is read in place from the block's qkv rows; X and QKV are bf16 [rows, 128]
// and [rows, 384]; the LayerNorm is folded into W_qkv (rstd (X W'^T - mean c) + d,
// the moments from the rounded X, whose row a pair of threads holds whole).
//
// A ring of six 32 KB stages feeds both products: per tile d / 64 stages of 64
// columns of K (128 rows) and of W_in (128 rows), then three of 128 rows of W_qkv'.
//   warp 0      fills the ring (TMA)
//   warp 1      issues the products: X into columns 0-127 of tensor memory, QKV
//               into 128-511, with X as A (bf16, 32 columns of each half's
//               accumulator, which the half has read by then)
//   warp 2      tensor-memory allocation
//   warps 4-11  epilogues: two threads a row, half of its columns each; the two
//               halves' slice moments meet in shared memory.  Each row's image,
//               whose first row takes the history term, is searched for while the
//               product runs.
// The next tile's first product runs under the QKV epilogue of this one.
//
// What bounds it: the loads, which stop while a tile's X goes through its epilogue
// with the ring full (K alone is 77 MB from DRAM at 256 x 197 tokens, d = 768; with
// K served by L2 it would take 22 us, without storing QKV 26).  As a linear with
// slice moments, a launch for the history term and the QKV linear the same took
// 18.4 + 4.0 + 16.4 us, here 30.9 (profiler, caches cold); the actor's call went
// from 111.8 to 107.3.  Issuing a tile's QKV after the next tile's X, from a second
// accumulator, gave no more (107.9): the QKV's two buffers then hold the ring back.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "dora_ptx.cuh"
#include "epilogue_math.cuh"
#include "token_ops.cuh"

namespace dora {
namespace actor_front {

constexpr int BM = 128;
constexpr int BK = 64;
constexpr int W = 128;          // encoder width
constexpr int NQ = 3 * W;
constexpr int kStages = 6;
constexpr int kThreads = 384;
constexpr int kEpiWarp0 = 4;
constexpr int kEpiWarps = 8;
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kDX = 0, kDQ = 128;
constexpr uint32_t kStageBytes = 2 * BM * BK * 2;

struct Smem {
  uint16_t ring[kStages][2][BM * BK];   // two 128 x 64 blocks each, 128-byte swizzle
  float c[NQ], d[NQ];                   // folded LayerNorm of W_qkv
  float wh[3][W];                       // W_h, transposed
  float bias[W];
  // Slice moments of X's two halves, by tile parity.  A half reads the other's of
  // tile n after x_ready(n), and nothing orders the next tile's X (x_full(n + 1),
  // behind q_full[2](n) alone) after that read; x_full(n + 2) is behind
  // x_ready(n + 1), at which every warp arrives after its reads of tile n.  So one
  // buffer would let a late warp take the next tile's moments, two do not.
  float2 half_moments[2][2][BM];
  uint64_t full[kStages];
  uint64_t empty[kStages];
  uint64_t x_full;                      // first product of the tile done
  uint64_t x_ready;                     // X in tensor memory (one arrival a warp)
  uint64_t q_full[3];                   // 128 columns of QKV done
  uint64_t q_free;                      // QKV read out (one arrival a warp)
  uint64_t drain;
  uint32_t tmem_base;
  int abort_flag;
  int issued, consumed;
};
static_assert(sizeof(Smem) <= 227 * 1024, "shared memory");

struct Maps {
  CUtensorMap k, win, wqkv;
};

// 64 packed columns to global memory (32-byte aligned).
__device__ __forceinline__ void store64(uint16_t* p, const uint32_t (&r)[32]) {
#pragma unroll
  for (int j = 0; j < 32; j += 8) st_global_32(reinterpret_cast<uint32_t*>(p) + j, &r[j]);
}

__device__ __forceinline__ float bf16_value(uint16_t v) {
  return __uint_as_float(static_cast<uint32_t>(v) << 16);
}

// The image whose first row is `row`, or -1; cu ascends over `batch` images.
__device__ __forceinline__ int image_starting_at(const int32_t* __restrict__ cu, int batch,
                                                 int row) {
  int lo = 0, hi = batch;               // cu[lo] <= row < cu[hi], were they in range
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (__ldg(cu + mid) <= row) lo = mid;
    else hi = mid;
  }
  return __ldg(cu + lo) == row ? lo : -1;
}

__global__ void __launch_bounds__(kThreads, 1)
    actor_front_kernel(const __grid_constant__ Maps mp, const FrontArgs a, int m_cap, int k_blocks,
                       int32_t* status) {
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
    for (int i = 0; i < kStages; ++i) {
      mbar_init(&s.full[i], 1);
      mbar_init(&s.empty[i], 1);
    }
    mbar_init(&s.x_full, 1);
    mbar_init(&s.x_ready, kEpiWarps);
    for (int i = 0; i < 3; ++i) mbar_init(&s.q_full[i], 1);
    mbar_init(&s.q_free, kEpiWarps);
    mbar_init(&s.drain, 1);
    s.abort_flag = 0;
    s.issued = s.consumed = 0;
    fence_barrier_init();
  }
  if (warp == 2) tmem_alloc(&s.tmem_base, kTmemCols);
  // the set-up above overlaps the previous kernel; global memory waits for it
  pdl_wait();
  for (int i = threadIdx.x; i < NQ; i += kThreads) {
    s.c[i] = a.c[i];
    s.d[i] = a.d[i];
    s.wh[i % 3][i / 3] = bf16_value(a.w_h[i]);
  }
  if (threadIdx.x < W) s.bias[threadIdx.x] = bf16_value(a.bias[threadIdx.x]);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  int M = a.cu[a.batch];
  M = M < 0 ? 0 : (M > m_cap ? m_cap : M);
  const int tiles = (M + BM - 1) / BM;
  const uint32_t tmem = s.tmem_base;
  volatile int* abort = &s.abort_flag;

  if (warp == 0) {
    if (elect_one()) {
      int it = 0;
      bool ok = true;
      for (int t = blockIdx.x; ok && t < tiles; t += gridDim.x) {
        for (int kb = 0; kb < k_blocks + 3; ++kb) {
          const int st = it % kStages;
          if (!(ok = mbar_wait(&s.empty[st], ((it / kStages) & 1) ^ 1, abort))) break;
          mbar_arrive_expect_tx(&s.full[st], kStageBytes);
          if (kb < k_blocks) {
            tma_load_2d(s.ring[st][0], &mp.k, &s.full[st], kb * BK, t * BM);
            tma_load_2d(s.ring[st][1], &mp.win, &s.full[st], kb * BK, 0);
          } else {
            tma_load_2d(s.ring[st][0], &mp.wqkv, &s.full[st], 0, (kb - k_blocks) * W);
            tma_load_2d(s.ring[st][1], &mp.wqkv, &s.full[st], BK, (kb - k_blocks) * W);
          }
          s.issued = ++it;
        }
      }
    }
  } else if (warp == 1) {
    if (elect_one()) {
      constexpr uint32_t idesc = idesc_bf16(BM, W, false);
      int it = 0, n = 0;
      bool ok = true;
      for (int t = blockIdx.x; ok && t < tiles; t += gridDim.x, ++n) {
        const uint32_t ph = n & 1;
        // X's accumulator: the tile before has read it, and as A its products are done
        if (n > 0 && !(ok = mbar_wait(&s.q_full[2], ph ^ 1, abort))) break;
        for (int kb = 0; kb < k_blocks; ++kb, ++it) {
          const int st = it % kStages;
          if (!(ok = mbar_wait(&s.full[st], (it / kStages) & 1, abort))) break;
          tc_fence_after();
          const uint64_t ad = sdesc_sw128(smem_u32(s.ring[st][0]), 16, 1024);
          const uint64_t bd = sdesc_sw128(smem_u32(s.ring[st][1]), 16, 1024);
#pragma unroll
          for (int k = 0; k < BK / 16; ++k)
            mma_bf16_ss(tmem + kDX, ad + 2 * k, bd + 2 * k, idesc, (kb | k) != 0 ? 1u : 0u);
          mma_commit(&s.empty[st]);
        }
        if (!ok) break;
        mma_commit(&s.x_full);
        if (!(ok = mbar_wait(&s.x_ready, ph, abort))) break;
        if (n > 0 && !(ok = mbar_wait(&s.q_free, ph ^ 1, abort))) break;
        for (int j = 0; j < 3; ++j, ++it) {
          const int st = it % kStages;
          if (!(ok = mbar_wait(&s.full[st], (it / kStages) & 1, abort))) break;
          tc_fence_after();
#pragma unroll
          for (int k = 0; k < W / 16; ++k)
            mma_bf16_ts(tmem + kDQ + 128u * j, tmem + kDX + 64u * (k / 4) + 8u * (k % 4),
                        sdesc_sw128(smem_u32(s.ring[st][k / 4]), 16, 1024) + 2 * (k % 4), idesc,
                        k > 0 ? 1u : 0u);
          mma_commit(&s.empty[st]);
          mma_commit(&s.q_full[j]);
        }
      }
      s.consumed = it;
      mma_commit(&s.drain);
      mbar_wait_limited(&s.drain, 0, kWaitLimitNs);
    }
  } else if (warp >= kEpiWarp0) {
    const int quarter = warp & 3, half = (warp - kEpiWarp0) >> 2;
    const int r = quarter * 32 + lane;
    const uint32_t lanes = tmem + (static_cast<uint32_t>(quarter * 32) << 16);
    const int c0 = 64 * half;                  // this thread's columns of a 128-wide row
    int n = 0;
    for (int t = blockIdx.x; t < tiles; t += gridDim.x, ++n) {
      const uint32_t ph = n & 1;
      const int row = t * BM + r;
      const bool live = row < M;
      // the history term of this row, if it is an image's first
      const int img = live ? image_starting_at(a.cu, a.batch, row) : -1;
      bool cls = false;
      float h0 = 0.f, h1 = 0.f, h2 = 0.f;
      if (img >= 0) {
        const int end = __ldg(a.cu + img + 1);
        cls = row >= 0 && end <= m_cap && end > row;
        h0 = static_cast<float>(end - row - 1) / static_cast<float>(a.n0);
        h1 = a.rho[img];
        h2 = static_cast<float>(a.interventions[img]) / static_cast<float>(max(a.depth - 1, 1));
      }
      uint32_t x[32];
      float v[32];
      if (!mbar_wait_warp(&s.x_full, ph, abort)) break;
      tc_fence_after();
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint32_t acc[32];
        const int c = c0 + 32 * h;
        tmem_ld32(lanes + kDX + c, acc);
        tmem_ld_wait();
#pragma unroll
        for (int e = 0; e < 32; ++e) v[e] = __uint_as_float(acc[e]) + s.bias[c + e];
        uint32_t(&o)[16] = *reinterpret_cast<uint32_t(*)[16]>(&x[16 * h]);
        pack_row(v, o);
        if (__any_sync(0xffffffffu, cls)) {
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            const int k = c + 2 * e;
            const float lo = s.wh[0][k] * h0 + s.wh[1][k] * h1 + s.wh[2][k] * h2;
            const float hi = s.wh[0][k + 1] * h0 + s.wh[1][k + 1] * h1 + s.wh[2][k + 1] * h2;
            const uint32_t with = pack_bf16x2(bf16_lo(o[e]) + lo, bf16_hi(o[e]) + hi);
            o[e] = cls ? with : o[e];
          }
        }
      }
      const float2 mine = slice_moments(*reinterpret_cast<const uint32_t(*)[16]>(&x[0]),
                                        *reinterpret_cast<const uint32_t(*)[16]>(&x[16]));
      s.half_moments[n & 1][half][r] = mine;
      // X over this thread's own accumulator columns
      tmem_st16(lanes + kDX + c0, *reinterpret_cast<const uint32_t(*)[16]>(&x[0]));
      tmem_st16(lanes + kDX + c0 + 16, *reinterpret_cast<const uint32_t(*)[16]>(&x[16]));
      tmem_st_wait();
      warp_arrive(&s.x_ready);
      if (live) store64(a.x + static_cast<size_t>(row) * W + c0, x);
      if (!mbar_wait_warp(&s.x_ready, ph, abort)) break;
      const float2 other = s.half_moments[n & 1][half ^ 1][r];
      const float2 mv = merge_two_slices(half ? other : mine, half ? mine : other);
      const float neg_mean = -mv.x, rstd = rsqrtf(mv.y + a.eps);
      bool ok = true;
#pragma unroll 1
      for (int j = 0; j < 3; ++j) {
        if (!(ok = mbar_wait_warp(&s.q_full[j], ph, abort))) break;
        tc_fence_after();
        const int c = W * j + c0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t acc[32];
          tmem_ld32(lanes + kDQ + c + 32 * h, acc);
          tmem_ld_wait();
#pragma unroll
          for (int e = 0; e < 32; ++e) v[e] = __uint_as_float(acc[e]);
          fold_layernorm(v, neg_mean, rstd, s.c + c + 32 * h, s.d + c + 32 * h);
          pack_row(v, *reinterpret_cast<uint32_t(*)[16]>(&x[16 * h]));
        }
        if (j == 2) warp_arrive(&s.q_free);
        if (live) store64(a.qkv + static_cast<size_t>(row) * NQ + c, x);
      }
      if (!ok) break;
    }
  }

  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (*abort) {
    if (threadIdx.x == 0) {
      record_status(status, DORA_ERR_TIMEOUT);
      // let every load that was issued but never consumed land
      for (int it = s.consumed; it < s.issued; ++it)
        mbar_wait_limited(&s.full[it % kStages], (it / kStages) & 1, 100ull * 1000 * 1000);
    }
    __syncthreads();
  }
  if (warp == 2) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

}  // namespace actor_front

cudaError_t launch_actor_front(const uint16_t* keys, int32_t pitch, int32_t dim,
                               const uint16_t* w_in, const uint16_t* w_qkv, const FrontArgs& args,
                               int32_t m_cap, int32_t* status, cudaStream_t stream) {
  using namespace actor_front;
  if (m_cap == 0) return cudaSuccess;
  Maps mp;
  auto map = [](CUtensorMap* m, const uint16_t* p, uint64_t cols, uint64_t rows, uint64_t ld) {
    return encode_tmap_2d_bf16(m, p, cols, rows, ld * 2, BK, BM) == 0;
  };
  if (!map(&mp.k, keys, dim, m_cap, pitch) || !map(&mp.win, w_in, dim, W, dim) ||
      !map(&mp.wqkv, w_qkv, W, NQ, W))
    return cudaErrorInvalidValue;
  const cudaError_t e =
      cudaFuncSetAttribute(actor_front_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           static_cast<int>(sizeof(Smem)));
  if (e != cudaSuccess) return e;
  const int tiles = (m_cap + BM - 1) / BM, cap = num_sms();
  return launch_pdl(actor_front_kernel, dim3(tiles < cap ? tiles : cap), dim3(kThreads),
                    sizeof(Smem), stream, mp, args, m_cap, dim / BK, status);
}

}  // namespace dora
