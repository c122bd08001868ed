// Dense bf16 GEMM with fused epilogues on the 5th-generation tensor cores:
//   Y[M, N] = epi(X[M, K] W[N, K]^T + b)      (nn.Linear layout)
// used for the QKV, projection and MLP linears of the pruned block (Eq. 1).
// The LayerNorm before the QKV and fc1 linears is folded in: with W' = W
// diag(gamma) (bf16), c = W' 1 and d = W beta + b,
//   LayerNorm(x) W^T + b = rstd (x W'^T - mean c) + d,
// so the GEMM reads the raw rows and the epilogue applies each row's mean and
// rstd = 1/sqrt(var + eps) from the row moments (mean, var) written with the
// rows; the residual epilogue writes the 64-column slice moments they are
// merged from.
//
// Design (one persistent CTA per SM, CTAs working in pairs):
//   The two CTAs of a pair work on vertically adjacent output tiles (M-tiles
//   2p and 2p+1 of the same N-tile), so they need the same W tile.  With
//   256-wide tiles a pair is a cluster; narrower tiles need nothing from the
//   neighbour but its L2 reads, and launching them without clusters takes
//   0.5-0.7 us off each (two cluster barriers and the cluster's scheduling):
//   197 x 192 to 576 columns 4.5 -> 4.0 us, 768 to 192 6.2 -> 5.5.
//   warp 0     TMA producer: the CTA's own 128x64 X tile and its part of the
//              BNx64 W tile, per stage of a shared-memory ring (128-byte
//              swizzle).  256-wide tiles run as a CTA pair (below), each CTA
//              loading half of W; narrower tiles load the whole W tile in each
//              CTA (both CTAs of a pair read the same W tile, so the second
//              read is an L2 hit).
//   warp 1     MMA issuer: one thread issues tcgen05.mma (M=128, N=BN, K=16,
//              or M=256 across the pair) into one of two TMEM accumulators
//              (2 x BN fp32 columns), so the epilogue of tile t overlaps the
//              main loop of tile t+1.
//   epilogue warps (2 .. 1 + kEpiWarps): tcgen05.ld the accumulator (each
//              thread owns one row; the warps of a TMEM lane quarter split the
//              columns), release it once in registers, add bias, GELU or
//              residual, round to bf16, stage each 32x32 chunk in shared
//              memory (64-byte swizzle) and write it with a TMA tensor store.
//              The residual epilogue gives each chunk its own buffer, into
//              which a TMA load brings the residual chunk while the tile's
//              MMAs still run; the result is written over it in place (a
//              long-K linear keeps two buffers a warp and reloads them within
//              the tile, for one more stage).  The patch embedding's epilogue
//              is the same with the position embeddings as the residual, boxes
//              of one image's rows shared by every image.  The tile that
//              straddles the live row count stores row by row.
// The live row count M may come from device memory (rows left after a
// deletion); tiles past it are never scheduled.  Every wait is bounded.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "dora_ptx.cuh"
#include "epilogue_math.cuh"
#include "token_ops.cuh"

namespace dora {
namespace gemm {

constexpr int BM = 128;
constexpr int BK = 64;
constexpr int kCluster = 2;
constexpr int kStageChunk = 32 * 32;   // one warp's 32 rows x 32 columns, bf16
constexpr int kSmemLimit = 227 * 1024;
// The residual epilogue of a long-K linear (K >= kLongK, fc2): two staging
// buffers per epilogue warp instead of one per chunk, so the stage ring gets
// one more stage.  The residual of a tile's first two chunks is loaded a tile
// ahead as in the plain residual epilogue; that of the other two is loaded
// into the first two's buffers once their stores have read them, inside an
// epilogue that a long main loop leaves mostly idle.
constexpr int kEpiResidualLongK = 5;
constexpr int kLongK = 2048;

// Per-instantiation layout.
// Pair mode: one MMA of M = 256 spans both CTAs of the cluster, each holding
// its own 128 rows of X and one half of the W tile, so a stage is 32 KB
// instead of 48; the shared memory read per MMA drops by a third.  Otherwise
// one MMA per CTA on a whole W tile of its own.
// Epilogue warps: a multiple of 4 (one per TMEM lane quarter); the ALU-heavy
// plain GELU epilogue gets 16, the others 8 with two staging buffers per warp
// (the residual epilogue one per chunk).  The stages fill what shared memory is left.
template <int BN, int EPI, bool PAIR>
struct Cfg {
  static constexpr bool kPair = PAIR;
  static constexpr int kBRows = kPair ? BN / 2 : BN;   // W rows held per CTA
  // The tiles of a last wave that would leave half of the clusters idle are cut
  // into two column halves, one a cluster (same bits).  us at 129 x 3 tile pairs on
  // 76 clusters (5.09 waves): fc2 106 -> 100, QKV (15.3) 75.8 -> 73.8, fc1 (20.4)
  // 116 -> 115; ViT-L's fc2 at 59 x 4 (3.1) 91 -> 84; no change where the last
  // wave is fuller.  Quarters gave no more, and cost fc2 1.3 % everywhere.
  // Not in the short-K residual epilogue, which fills its main loop: the
  // run-time column count costs it more (47.4 -> 48.6 us) than the halves give.
  static constexpr bool kSplit = PAIR && EPI != DORA_EPI_BIAS_RESIDUAL;
  static constexpr bool kLn = EPI == kEpiLn || EPI == kEpiLnGelu;
  static constexpr bool kResTma =
      EPI == DORA_EPI_BIAS_RESIDUAL || EPI == kEpiResidualLongK || EPI == kEpiTokens;
  // slice moments of the output rows, where the caller takes them
  static constexpr bool kMoments = kResTma && EPI != kEpiTokens;
  // the two GELU epilogues are ALU-bound: 16 warps; so is the patch embedding's
  // on 256 columns, with its short K (128 images of 16 x 16 patches, the call: 55.0
  // -> 51.8 us); the others 8 (the residual's spills with 16: 61.5 -> 67.6 us at
  // 50432 x 768 x 768, and the plain LayerNorm's runs 108.5 -> 113.0).  A 64-wide
  // tile has 32 columns for each of 8 warps; the residual's need whole
  // 64-column slices: 4
  static constexpr int kEpiWarps =
      BN == 64 ? (kResTma ? 4 : 8)
               : ((EPI == DORA_EPI_BIAS_GELU || EPI == kEpiLnGelu ||
                   (EPI == kEpiTokens && BN == 256))
                      ? 16
                      : 8);
  static constexpr int kColGroups = kEpiWarps / 4;
  static constexpr int kCols = BN / kColGroups;         // columns per epilogue warp
  static constexpr int kChunks = kCols / 32;
  // chunks per TMEM load: two (64 registers) unless 16 warps cap registers at
  // 96, or a long K hides the loads anyway (two would spill)
  static constexpr int kBatch =
      (kEpiWarps == 16 || EPI == kEpiResidualLongK) ? 1 : (kChunks < 2 ? kChunks : 2);
  // staging buffers per epilogue warp: one per chunk for the residual (its
  // TMA load lands there; two for a long K), one with 16 warps or the folded
  // LayerNorm, else two
  static constexpr int kBufs =
      kResTma ? (EPI == kEpiResidualLongK && kChunks > 2 ? 2 : kChunks)
              : ((kEpiWarps == 16 || kLn) ? 1 : 2);
  // folded LayerNorm: each epilogue warp's c and d columns, staged per tile
  static constexpr int kCdCols = kLn ? kCols : 1;
  static constexpr int kThreads = 64 + 32 * kEpiWarps;
  static constexpr int kStageBytes = (BM + kBRows) * BK * 2;
  static constexpr int kOutBytes = kEpiWarps * (kBufs * kStageChunk * 2 + 2 * kCdCols * 4);
  static constexpr int kFit = (kSmemLimit - 1024 - kOutBytes) / kStageBytes;
  static constexpr int kStages = kFit < 6 ? kFit : 6;
  static_assert(kStages >= 2, "shared memory");
};
constexpr uint16_t kPairMask = 0x3;

template <int BN, int EPI, bool PAIR>
struct Smem {
  using C = Cfg<BN, EPI, PAIR>;
  uint16_t a[C::kStages][BM * BK];                  // 16 KB per stage
  uint16_t b[C::kStages][C::kBRows * BK];           // 16 or 32 KB per stage
  uint16_t out[C::kEpiWarps][C::kBufs][kStageChunk];   // 2 KB each
  float cd[C::kEpiWarps][2][C::kCdCols];            // colsum, colbias of the warp's columns
  uint64_t full[C::kStages];
  uint64_t empty[C::kStages];
  uint64_t res_full[C::kEpiWarps][C::kResTma ? C::kBufs : 1];
  uint64_t cd_full[C::kEpiWarps];
  uint64_t acc_full[2];
  uint64_t acc_empty[2];
  uint64_t drain;
  uint32_t tmem_base;
  int abort_flag;
  int issued;
  int consumed;
};

// Bias (or the folded LayerNorm) and GELU of one 32-column chunk of one row,
// in fp32.
// For the folded LayerNorm, c and d of the chunk's 32 columns come from
// shared memory (cs, cb).
template <int EPI>
__device__ __forceinline__ void epilogue_math(const uint32_t (&r)[32], float (&v)[32],
                                              const LinearEpi& ep, int gcol, float neg_mean,
                                              float rstd, const float* cs, const float* cb) {
#pragma unroll
  for (int e = 0; e < 32; ++e) v[e] = __uint_as_float(r[e]);
  if constexpr (EPI == kEpiLn || EPI == kEpiLnGelu) {
    fold_layernorm(v, neg_mean, rstd, cs, cb);
  } else if (EPI != kEpiTokens && ep.bias != nullptr) {
    const uint4* bp = reinterpret_cast<const uint4*>(ep.bias + gcol);
#pragma unroll
    for (int q = 0; q < 4; ++q) add_bf16x8(v + 8 * q, __ldg(bp + q));
  }
  if constexpr (EPI == DORA_EPI_BIAS_GELU || EPI == kEpiLnGelu) {
#pragma unroll
    for (int e = 0; e < 32; e += 2) gelu_erf2(v[e], v[e + 1]);
  }
}

template <int BN, int EPI, bool PAIR>
__global__ void __launch_bounds__(Cfg<BN, EPI, PAIR>::kThreads, 1)
    gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                const __grid_constant__ CUtensorMap tmBt,
                const __grid_constant__ CUtensorMap tmY, const __grid_constant__ CUtensorMap tmR,
                uint16_t* __restrict__ Y, const LinearEpi ep, int m_cap,
                const int32_t* __restrict__ m_dev, int N, int K, int32_t* status) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  pdl_trigger();
  if (smem_u32(smem_raw) & 1023u) {           // swizzled tiles need 1 KB alignment
    pdl_wait();
    if (threadIdx.x == 0) record_status(status, DORA_ERR_UNSUPPORTED);
    return;
  }
  Smem<BN, EPI, PAIR>& s = *reinterpret_cast<Smem<BN, EPI, PAIR>*>(smem_raw);
  using C = Cfg<BN, EPI, PAIR>;
  constexpr int kEpiWarps = C::kEpiWarps;
  constexpr int kBufs = C::kBufs;
  constexpr int kStages = C::kStages;
  constexpr bool kPair = C::kPair;
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  // Work is a list of tile pairs: pair p covers M-tiles 2*(p / n_tiles) and
  // 2*(p / n_tiles) + 1 of N-tile p % n_tiles (row pairs counted from the
  // last with ep.m_reverse); CTA `rank` of CTA pair c takes the M-tile
  // 2*(p / n_tiles) + rank of pairs c, c + clusters, ...
  // Both CTAs of a cluster (pair mode) walk the same pairs in lockstep.
  const int rank =
      kPair ? static_cast<int>(cluster_ctarank()) : static_cast<int>(blockIdx.x % kCluster);
  const int cid = blockIdx.x / kCluster;
  const int n_clusters = gridDim.x / kCluster;
  const int n_tiles = (N + BN - 1) / BN;
  const int kb_count = K / BK;
  constexpr uint32_t kTmemCols = 2 * BN;
  constexpr int kHalfB = BN / 2;

  if (threadIdx.x == 0) {
    for (int i = 0; i < kStages; ++i) {
      mbar_init(&s.full[i], 1);
      // pair mode: the first CTA's MMAs release both CTAs' stages; otherwise
      // each CTA's own MMAs release its stage
      mbar_init(&s.empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&s.acc_full[i], 1);
      // pair mode: the epilogues of both CTAs hand the accumulator back to the first
      mbar_init(&s.acc_empty[i], kPair ? 2 * kEpiWarps : kEpiWarps);
    }
    for (int w = 0; w < kEpiWarps; ++w) {
      for (int c = 0; c < (C::kResTma ? C::kBufs : 1); ++c) mbar_init(&s.res_full[w][c], 1);
      mbar_init(&s.cd_full[w], 1);
    }
    mbar_init(&s.drain, 1);
    s.abort_flag = 0;
    s.issued = 0;
    s.consumed = 0;
    fence_barrier_init();
    tma_prefetch_desc(&tmA);
    tma_prefetch_desc(&tmB);
    tma_prefetch_desc(&tmY);
    if (C::kResTma) tma_prefetch_desc(&tmR);
  }
  if (warp == 1) {
    if constexpr (kPair) tmem_alloc_pair(&s.tmem_base, kTmemCols);
    else tmem_alloc(&s.tmem_base, kTmemCols);
  }
  tc_fence_before();
  // peers' barriers are initialised before any remote signal
  if constexpr (kPair) cluster_sync();
  else __syncthreads();
  tc_fence_after();
  // the set-up above overlaps the previous kernel; global memory waits for it
  pdl_wait();
  int M = m_cap;
  if (m_dev != nullptr) {
    const int v = *m_dev;
    M = v < 0 ? 0 : (v > m_cap ? m_cap : v);
  }
  const int m_pairs = (M + 2 * BM - 1) / (2 * BM);
  const int num_pairs = m_pairs * n_tiles;
  // Work items: the tile pairs, those of a sparse last wave as column halves.
  int full = num_pairs;                         // tile pairs left whole
  if constexpr (C::kSplit) {
    const int rest = num_pairs % n_clusters;
    if (2 * rest <= n_clusters) full -= rest;
  }
  const int items = full + 2 * (num_pairs - full);
  struct Item {
    int pair, n0, cols;                         // tile pair, first output column, columns
  };
  auto item = [&](int w) -> Item {
    if (!C::kSplit || w < full) return {w, (w % n_tiles) * BN, BN};
    const int p = full + ((w - full) >> 1);
    return {p, (p % n_tiles) * BN + ((w - full) & 1) * (BN / 2), BN / 2};
  };
  const uint32_t tmem = s.tmem_base;
  volatile int* abort = &s.abort_flag;
  // row pair of work item p; m_reverse walks them from the last, so that a
  // linear reading the output of one that walked forward starts on the rows
  // written last, still in L2
  auto mpair = [&](int p) {
    const int q0 = p / n_tiles;
    return ep.m_reverse ? m_pairs - 1 - q0 : q0;
  };

  if (warp == 0) {
    if (elect_one()) {
      int it = 0;
      bool ok = true;
      for (int w = cid; ok && w < items; w += n_clusters) {
        const Item t = item(w);
        const int mt = 2 * mpair(t.pair) + rank;
        for (int kb = 0; kb < kb_count; ++kb) {
          const int st = it % kStages;
          const uint32_t ph = (it / kStages) & 1;
          if (!mbar_wait(&s.empty[st], ph ^ 1, abort)) {
            ok = false;
            break;
          }
          if constexpr (kPair) {
            // this CTA's X rows and half of the W tile; the bytes of both CTAs
            // are counted on the first CTA's barrier, which its MMA waits on
            // (half a tile loads boxes half as high)
            const bool whole = !C::kSplit || t.cols == BN;
            if (rank == 0)
              mbar_arrive_expect_tx(&s.full[st],
                                    2 * (BM + (whole ? kHalfB : kHalfB / 2)) * BK * 2);
            tma_load_2d_pair(s.a[st], &tmA, &s.full[st], 0, kb * BK, mt * BM);
            tma_load_2d_pair(s.b[st], whole ? &tmB : &tmBt, &s.full[st], 0, kb * BK,
                             t.n0 + rank * (t.cols >> 1));
          } else {
            // the X tile and both halves of the W tile (the map's box is BN/2 rows)
            mbar_arrive_expect_tx(&s.full[st], (BM + BN) * BK * 2);
            tma_load_2d(s.a[st], &tmA, &s.full[st], kb * BK, mt * BM);
            tma_load_2d(s.b[st], &tmB, &s.full[st], kb * BK, t.n0);
            tma_load_2d(s.b[st] + kHalfB * BK, &tmB, &s.full[st], kb * BK, t.n0 + kHalfB);
          }
          ++it;
        }
      }
      s.issued = it;
    }
  } else if (warp == 1) {
    const bool issuer = elect_one();
    if (issuer && kPair && rank == 0) {
      // pair MMA issuer: M = 256 over both CTAs, D in both CTAs' TMEM
      int it = 0, ti = 0;
      bool ok = true;
      for (int w = cid; ok && w < items; w += n_clusters, ++ti) {
        const uint32_t idesc = idesc_bf16(2 * BM, C::kSplit && w >= full ? BN / 2 : BN, false);
        const int acc = ti & 1;
        const uint32_t aph = (ti >> 1) & 1;
        if (!mbar_wait(&s.acc_empty[acc], aph ^ 1, abort)) break;
        tc_fence_after();
        const uint32_t d = tmem + static_cast<uint32_t>(acc * BN);
        for (int kb = 0; kb < kb_count; ++kb) {
          const int st = it % kStages;
          const uint32_t ph = (it / kStages) & 1;
          if (!mbar_wait(&s.full[st], ph, abort)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint64_t ad = sdesc_sw128(smem_u32(s.a[st]), 16, 1024);
          const uint64_t bd = sdesc_sw128(smem_u32(s.b[st]), 16, 1024);
#pragma unroll
          for (int k = 0; k < BK / 16; ++k)
            mma_bf16_ss_pair(d, ad + 2 * k, bd + 2 * k, idesc, (kb | k) != 0 ? 1u : 0u);
          mma_commit_pair(&s.empty[st], kPairMask);        // both CTAs' stages free
          ++it;
        }
        if (ok) mma_commit_pair(&s.acc_full[acc], kPairMask);
      }
      s.consumed = it;
      mma_commit_pair(&s.drain, 0x1);
      mbar_wait_limited(&s.drain, 0, kWaitLimitNs);
    } else if (issuer) {
     if constexpr (!kPair) {
      constexpr uint32_t idesc = idesc_bf16(BM, BN, false);
      int it = 0, ti = 0;
      bool ok = true;
      for (int w = cid; ok && w < items; w += n_clusters, ++ti) {
        const int acc = ti & 1;
        const uint32_t aph = (ti >> 1) & 1;
        if (!mbar_wait(&s.acc_empty[acc], aph ^ 1, abort)) break;
        tc_fence_after();
        const uint32_t d = tmem + static_cast<uint32_t>(acc * BN);
        for (int kb = 0; kb < kb_count; ++kb) {
          const int st = it % kStages;
          const uint32_t ph = (it / kStages) & 1;
          if (!mbar_wait(&s.full[st], ph, abort)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint64_t ad = sdesc_sw128(smem_u32(s.a[st]), 16, 1024);
          const uint64_t bd = sdesc_sw128(smem_u32(s.b[st]), 16, 1024);
#pragma unroll
          for (int k = 0; k < BK / 16; ++k)
            mma_bf16_ss(d, ad + 2 * k, bd + 2 * k, idesc, (kb | k) != 0 ? 1u : 0u);
          mma_commit(&s.empty[st]);                        // this CTA's stage free
          ++it;
        }
        if (ok) mma_commit(&s.acc_full[acc]);
      }
      s.consumed = it;
      mma_commit(&s.drain);
      mbar_wait_limited(&s.drain, 0, kWaitLimitNs);
     }
    }
  } else {
    constexpr int kBatch = C::kBatch;              // chunks per TMEM load
    const int ew = warp - 2;                      // epilogue warp index
    const int q = warp & 3;                       // TMEM lanes this warp may read
    const int slot = ew >> 2;                     // which column slice
    // chunks of 32 columns of each warp in an item
    auto warp_chunks = [&](const Item& t) {
      return !C::kSplit || t.cols == BN ? C::kChunks : C::kChunks / 2;
    };
    const uint32_t lane_sel = static_cast<uint32_t>(q * 32) << 16;
    int buf = 0;                                  // staging buffer to write next
    uint32_t res_pend = 0;                        // staging buffers with a residual load in flight
    uint32_t res_par = 0;                         // their next completion parity
    // Residual chunk `c` of the warp's 32 rows from row0, column col0 on, into
    // staging buffer c % kBufs (whose previous store must have read it).
    // The patch embedding's residual is its token's position embedding: the
    // box starts at the first row's token, and lanes past the image's last
    // token (where the box reads zeros) fetch theirs from the next image's start.
    auto residual_row = [&](int row_, int gcol) {
      const int r_ = EPI == kEpiTokens ? row_ % ep.tokens : row_;
      return reinterpret_cast<const uint4*>((EPI == kEpiTokens ? ep.pos : ep.residual) +
                                            static_cast<size_t>(r_) * N + gcol);
    };
    auto load_residual = [&](int c, int row0, int col0) {
      const int b = c % kBufs;
      if (lane == 0) {
        mbar_arrive_expect_tx(&s.res_full[ew][b], kStageChunk * 2);
        tma_load_2d(s.out[ew][b], &tmR, &s.res_full[ew][b], col0 + c * 32,
                    EPI == kEpiTokens ? row0 % ep.tokens : row0);
      }
      res_pend |= 1u << b;
    };
    // Residual of the warp's whole 32-row chunks of tile pair `p` (the first
    // kBufs chunks), once the stores of the previous tile have read the buffers.
    auto prefetch_residual = [&](int w) {
      const Item t = item(w);
      const int row0 = (2 * mpair(t.pair) + rank) * BM + q * 32;
      if (row0 + 32 > M) return;
      const int chunks = warp_chunks(t);
      const int col0 = t.n0 + slot * 32 * chunks;
      if (lane == 0) bulk_wait_group_read0();
      __syncwarp();
#pragma unroll
      for (int c = 0; c < kBufs; ++c) {
        if (c >= chunks || col0 + c * 32 >= N) break;
        load_residual(c, row0, col0);
      }
    };
    // Slice moments of the rounded output row: the first chunk of a 64-column
    // slice is kept packed until the second is done.
    uint32_t first_half[16];
    auto emit_moments = [&](const uint32_t(&o)[16], int row_, int gcol) {
      if ((gcol & 32) == 0) {
#pragma unroll
        for (int e = 0; e < 16; ++e) first_half[e] = o[e];
      } else {
        reinterpret_cast<float2*>(ep.stats_out)[static_cast<size_t>(gcol >> 6) * m_cap + row_] =
            slice_moments(first_half, o);
      }
    };
    // Folded LayerNorm: c and d of the warp's columns of tile pair `p`, one
    // bulk copy each into the warp's buffer, after the warp's reads of the
    // previous tile's values.
    bool cd_pend = false;
    uint32_t cd_par = 0;
    auto prefetch_cd = [&](int w) {
      const Item t = item(w);
      const int mine = 32 * warp_chunks(t);
      const int col0 = t.n0 + slot * mine;
      const int cols = N - col0 < mine ? N - col0 : mine;
      if (cols <= 0) return;
      __syncwarp();                               // every lane's reads of the buffer are done
      if (lane == 0) {
        fence_proxy_async_smem();
        mbar_arrive_expect_tx(&s.cd_full[ew], 2u * 4u * static_cast<uint32_t>(cols));
        bulk_load(s.cd[ew][0], ep.colsum + col0, 4u * cols, &s.cd_full[ew]);
        bulk_load(s.cd[ew][1], ep.colbias + col0, 4u * cols, &s.cd_full[ew]);
      }
      cd_pend = true;
    };
    // Folded LayerNorm: (mean, var) of this lane's row, loaded a tile ahead
    // (a warp's 32 rows are one 256-byte load).
    float2 mv = make_float2(0.f, 0.f);
    auto load_mv = [&](int w) {
      const int row_p = (2 * mpair(item(w).pair) + rank) * BM + q * 32 + lane;
      if (row_p >= M) return;
      const float2* p = reinterpret_cast<const float2*>(ep.stats_in) + row_p;
      if (BN < 256 && ep.slices_in > 0) mv = merge_slice_moments(p, m_cap, ep.slices_in);
      else mv = __ldg(p);
    };
    if constexpr (C::kLn)
      if (cid < items) {
        prefetch_cd(cid);
        load_mv(cid);
      }
    if constexpr (C::kResTma)
      if (cid < items) prefetch_residual(cid);
    int ti = 0;
    bool ok = true;
    for (int w = cid; ok && w < items; w += n_clusters, ++ti) {
      const int acc = ti & 1;
      const uint32_t aph = (ti >> 1) & 1;
      const Item t = item(w);
      const int mt = 2 * mpair(t.pair) + rank;
      const int chunks = warp_chunks(t);
      const int wcol0 = slot * 32 * chunks;       // this warp's first column of the tile
      const int row0 = mt * BM + q * 32;          // first row of this warp
      const int row = row0 + lane;
      const bool whole = row0 + 32 <= M;          // all 32 rows live: TMA store
      const bool past_image = EPI == kEpiTokens && row0 % ep.tokens + lane >= ep.tokens;
      float neg_mean = 0.f, rstd = 0.f;           // folded LayerNorm of this row
      if constexpr (C::kLn) {
        neg_mean = -mv.x;
        rstd = rsqrtf(mv.y + ep.eps);
        if (w + n_clusters < items) load_mv(w + n_clusters);
      }
      if (!mbar_wait_warp(&s.acc_full[acc], aph, abort)) break;
      tc_fence_after();
      if constexpr (C::kLn) {
        if (cd_pend) {
          if (!mbar_wait_warp(&s.cd_full[ew], cd_par, abort)) break;
          cd_par ^= 1u;
          cd_pend = false;
        }
      }
#pragma unroll 1
      for (int cb = 0; cb < chunks; cb += kBatch) {
        uint32_t r[kBatch][32];
#pragma unroll
        for (int c = 0; c < kBatch; ++c)
          tmem_ld32(tmem + lane_sel +
                        static_cast<uint32_t>(acc * BN + wcol0 + (cb + c) * 32),
                    r[c]);
        tmem_ld_wait();
        if (cb + kBatch == chunks) {
          // the accumulator is in registers: hand it back to the MMA warp
          tc_fence_before();
          __syncwarp();
          if (lane == 0) {
            if (kPair && rank != 0) mbar_arrive_remote(&s.acc_empty[acc], 0);
            else mbar_arrive(&s.acc_empty[acc]);
          }
        }
#pragma unroll
        for (int c = 0; c < kBatch; ++c) {
          const int gcol = t.n0 + wcol0 + (cb + c) * 32;
          if (gcol >= N || row0 >= M) continue;    // warp-uniform
          float v[32];
          uint32_t o[16];
          epilogue_math<EPI>(r[c], v, ep, gcol, neg_mean, rstd,
                             &s.cd[ew][0][((cb + c) * 32) % C::kCdCols],
                             &s.cd[ew][1][((cb + c) * 32) % C::kCdCols]);
          if constexpr (EPI == kEpiTokens) {
            // bias, or the CLS token, whose row takes nothing from its (zero) patch
            const bool is_cls = row % ep.tokens == 0;
            const uint16_t* add = is_cls ? ep.cls : ep.bias;
#pragma unroll
            for (int e = 0; e < 32; ++e) v[e] = is_cls ? 0.f : v[e];
            if (add != nullptr) {
#pragma unroll
              for (int j = 0; j < 4; ++j)
                add_bf16x8(v + 8 * j, __ldg(reinterpret_cast<const uint4*>(add + gcol) + j));
            }
          }
          if (whole) {
            // row `lane` of the 32x32 chunk, 64-byte swizzle: 16-byte piece j
            // of row l sits at piece j ^ ((l >> 1) & 3).
            uint16_t* stage;
            if constexpr (C::kResTma) {
              const int rb = (cb + c) % kBufs;
              stage = s.out[ew][rb];
              if (!mbar_wait_warp(&s.res_full[ew][rb], (res_par >> rb) & 1u, abort)) {
                ok = false;
                break;
              }
              res_par ^= 1u << rb;
              res_pend &= ~(1u << rb);
            } else {
              // the store issued kBufs chunks ago from this buffer must have read it
              stage = s.out[ew][buf];
              if (lane == 0) {
                if constexpr (kBufs == 2) bulk_wait_group_read1();
                else bulk_wait_group_read0();
              }
              __syncwarp();
              buf = (buf + 1) % kBufs;
            }
            uint8_t* rowp = reinterpret_cast<uint8_t*>(stage) + lane * 64;
            if constexpr (C::kResTma) {
#pragma unroll
              for (int j = 0; j < 4; ++j)
                add_bf16x8(v + 8 * j,
                           past_image ? __ldg(residual_row(row, gcol) + j)
                                      : *reinterpret_cast<const uint4*>(
                                            rowp + ((j ^ ((lane >> 1) & 3)) << 4)));
            }
            pack_row(v, o);
            if constexpr (C::kMoments)
              if (ep.stats_out != nullptr) emit_moments(o, row, gcol);
#pragma unroll
            for (int j = 0; j < 4; ++j)
              *reinterpret_cast<uint4*>(rowp + ((j ^ ((lane >> 1) & 3)) << 4)) =
                  make_uint4(o[4 * j], o[4 * j + 1], o[4 * j + 2], o[4 * j + 3]);
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
              tma_store_2d(&tmY, stage, gcol, row0);
              bulk_commit_group();
            }
            if constexpr (C::kResTma && kBufs < C::kChunks) {
              // the chunk kBufs on goes into this buffer once the store has read it
              const int nc = cb + c + kBufs;
              const int col0 = t.n0 + wcol0;
              if (nc < chunks && col0 + nc * 32 < N) {
                if (lane == 0) bulk_wait_group_read0();
                __syncwarp();
                load_residual(nc, row0, col0);
              }
            }
          } else if (row < M) {
            if constexpr (C::kResTma) {
              const uint4* rp = residual_row(row, gcol);
#pragma unroll
              for (int j = 0; j < 4; ++j) add_bf16x8(v + 8 * j, __ldg(rp + j));
            }
            pack_row(v, o);
            if constexpr (C::kMoments)
              if (ep.stats_out != nullptr) emit_moments(o, row, gcol);
            uint4* yp = reinterpret_cast<uint4*>(Y + static_cast<size_t>(row) * N + gcol);
#pragma unroll
            for (int j = 0; j < 4; ++j)
              yp[j] = make_uint4(o[4 * j], o[4 * j + 1], o[4 * j + 2], o[4 * j + 3]);
          }
        }
        if (!ok) break;
      }
      if constexpr (C::kResTma)
        if (ok && w + n_clusters < items) prefetch_residual(w + n_clusters);
      if constexpr (C::kLn)
        if (ok && w + n_clusters < items) prefetch_cd(w + n_clusters);
    }
    if (lane == 0) {
      bulk_wait_group0();                         // stores done before the CTA exits
      // after an abort: residual loads issued but never consumed land first
      for (int c = 0; c < kBufs; ++c)
        if (res_pend & (1u << c))
          mbar_wait_limited(&s.res_full[ew][c], (res_par >> c) & 1u, 100ull * 1000 * 1000);
      if (cd_pend) mbar_wait_limited(&s.cd_full[ew], cd_par, 100ull * 1000 * 1000);
    }
    __syncwarp();
  }

  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (*abort) {
    if (threadIdx.x == 0) {
      record_status(status, DORA_ERR_TIMEOUT);
      // let every TMA load that was issued but never consumed land first
      if (!kPair || rank == 0)
        for (int it = s.consumed; it < s.issued; ++it)
          mbar_wait_limited(&s.full[it % kStages], (it / kStages) & 1, 100ull * 1000 * 1000);
    }
    __syncthreads();
  }
  if (warp == 1) {
    tc_fence_after();
    if constexpr (kPair) tmem_dealloc_pair(tmem, kTmemCols);
    else tmem_dealloc(tmem, kTmemCols);
  }
  // no CTA leaves while its peer may still signal it
  if constexpr (kPair) cluster_sync();
}

template <int BN, int EPI, bool PAIR>
static cudaError_t launch_bn_epi(const CUtensorMap& ta, const CUtensorMap& tb,
                                 const CUtensorMap& tbt, const CUtensorMap& ty,
                                 const CUtensorMap& tr, uint16_t* y, const LinearEpi& ep,
                                 int m_cap, const int32_t* m_dev, int n, int k, int32_t* status,
                                 cudaStream_t stream) {
  static_assert(sizeof(Smem<BN, EPI, PAIR>) <= kSmemLimit, "shared memory");
  const size_t smem = sizeof(Smem<BN, EPI, PAIR>);
  auto kern = gemm_kernel<BN, EPI, PAIR>;
  cudaError_t e =
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = kCluster;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.blockDim = dim3(Cfg<BN, EPI, PAIR>::kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = attr + 1;
  cfg.numAttrs = PAIR ? 1 : 0;
  // as many co-resident clusters as fit, capped by the tile pairs of m_cap
  static int max_clusters[64] = {0};   // per instantiation and device
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) dev = 0;
  if (max_clusters[dev] == 0) {
    cfg.gridDim = dim3(kCluster * (num_sms() / kCluster));
    int c = num_sms() / kCluster;
    if (PAIR) {
      e = cudaOccupancyMaxActiveClusters(&c, kern, &cfg);
      if (e != cudaSuccess) return e;
    }
    max_clusters[dev] = c > 0 ? c : 1;
  }
  const long pairs =
      static_cast<long>((m_cap + 2 * BM - 1) / (2 * BM)) * ((n + BN - 1) / BN);
  const long clusters = pairs < max_clusters[dev] ? pairs : max_clusters[dev];
  cfg.gridDim = dim3(static_cast<unsigned>(kCluster * clusters));
  if (pdl_enabled()) {                           // dependent launch (the kernel waits)
    cfg.attrs = attr;
    ++cfg.numAttrs;
  }
  return cudaLaunchKernelEx(&cfg, kern, ta, tb, tbt, ty, tr, y, ep, m_cap, m_dev, n, k, status);
}

// BN = 256 tiles run in pair mode.
template <int BN>
static cudaError_t launch_bn(const CUtensorMap& ta, const CUtensorMap& tb,
                             const CUtensorMap& tbt, const CUtensorMap& ty, const CUtensorMap& tr,
                             uint16_t* y, const LinearEpi& ep, int epi, int m_cap,
                             const int32_t* m_dev, int n, int k, int32_t* status,
                             cudaStream_t stream) {
  constexpr bool kPair = BN == 256;
  const auto launch = [&](auto kernel) {
    return kernel(ta, tb, tbt, ty, tr, y, ep, m_cap, m_dev, n, k, status, stream);
  };
  switch (epi) {
    case DORA_EPI_BIAS_GELU:
      return launch(launch_bn_epi<BN, DORA_EPI_BIAS_GELU, kPair>);
    case DORA_EPI_BIAS_RESIDUAL:
      return launch(launch_bn_epi<BN, DORA_EPI_BIAS_RESIDUAL, kPair>);
    case kEpiResidualLongK:                        // only wide tiles
      if constexpr (BN == 256) return launch(launch_bn_epi<BN, kEpiResidualLongK, kPair>);
      return cudaErrorInvalidValue;
    case kEpiTokens:
      return launch(launch_bn_epi<BN, kEpiTokens, kPair>);
    case kEpiLn:
      return launch(launch_bn_epi<BN, kEpiLn, kPair>);
    case kEpiLnGelu:
      return launch(launch_bn_epi<BN, kEpiLnGelu, kPair>);
    default:
      return launch(launch_bn_epi<BN, DORA_EPI_BIAS, kPair>);
  }
}

// Whether one wave of CTA pairs holds every tile pair of that width.
static bool one_wave(int32_t m_cap, int32_t n, int bn) {
  const long row_pairs = (static_cast<long>(m_cap) + 2 * BM - 1) / (2 * BM);
  return row_pairs * ((n + bn - 1) / bn) <= num_sms() / kCluster;
}

}  // namespace gemm

// In one wave a CTA merges its rows' moments once, under the loads and MMAs of
// its only tile; in more, every tile would again, and the wide tiles' epilogues
// have no registers for it (a forward of 256 DeiT-B images 4.91 -> 5.23 ms).
bool linear_merges(int32_t m_cap, int32_t n) { return gemm::one_wave(m_cap, n, 128); }

cudaError_t launch_linear(const uint16_t* x, int32_t m_cap, const int32_t* m_dev, int32_t k,
                          const uint16_t* w, int32_t n, int32_t epilogue, const LinearEpi& ep,
                          uint16_t* y, int32_t* status, cudaStream_t stream) {
  if (m_cap == 0) return cudaSuccess;
  // A tile's main loop and epilogue get shorter with its width, so while one
  // wave of clusters holds all of them the narrowest tile finishes first; past
  // that the widest feeds the tensor cores best.  256 x 1536 to 1024 columns
  // (DINOv2's head) on 16 clusters instead of 4, us with the pooling: 29.2 -> 25.2; a
  // DeiT-B block on one image 70.2 -> 53.2 and on eight 74.3 -> 63.1, DeiT-Tiny's on
  // eight 47.1 -> 43.8.
  int bn = (n % 256 == 0) ? 256 : 128;
  if (gemm::one_wave(m_cap, n, 64)) bn = 64;
  else if (gemm::one_wave(m_cap, n, 128)) bn = 128;
  CUtensorMap ta, tb, tbt, ty, tr;
  if (encode_tmap_2d_bf16(&ta, x, static_cast<uint64_t>(k), static_cast<uint64_t>(m_cap),
                          static_cast<uint64_t>(k) * 2, gemm::BK, gemm::BM) != 0)
    return cudaErrorInvalidValue;
  if (encode_tmap_2d_bf16(&tb, w, static_cast<uint64_t>(k), static_cast<uint64_t>(n),
                          static_cast<uint64_t>(k) * 2, gemm::BK, static_cast<uint32_t>(bn / 2)) != 0)
    return cudaErrorInvalidValue;
  // the same with boxes half as high, for column halves of a tile (unused otherwise)
  tbt = tb;
  if (bn == 256 &&
      encode_tmap_2d_bf16(&tbt, w, static_cast<uint64_t>(k), static_cast<uint64_t>(n),
                          static_cast<uint64_t>(k) * 2, gemm::BK, 64) != 0)
    return cudaErrorInvalidValue;
  if (encode_tmap_2d_bf16(&ty, y, static_cast<uint64_t>(n), static_cast<uint64_t>(m_cap),
                          static_cast<uint64_t>(n) * 2, 32, 32, 64) != 0)
    return cudaErrorInvalidValue;
  // the residual [m_cap, n] in the output's 32 x 32 chunks (unused otherwise)
  tr = ty;
  const bool tokens = epilogue == kEpiTokens;          // the position embeddings
  if ((epilogue == DORA_EPI_BIAS_RESIDUAL || tokens) &&
      encode_tmap_2d_bf16(&tr, tokens ? ep.pos : ep.residual, static_cast<uint64_t>(n),
                          static_cast<uint64_t>(tokens ? ep.tokens : m_cap),
                          static_cast<uint64_t>(n) * 2, 32, 32, 64) != 0)
    return cudaErrorInvalidValue;
  if (bn == 256) {
    const int epi = (epilogue == DORA_EPI_BIAS_RESIDUAL && k >= gemm::kLongK)
                        ? gemm::kEpiResidualLongK
                        : epilogue;
    return gemm::launch_bn<256>(ta, tb, tbt, ty, tr, y, ep, epi, m_cap, m_dev, n, k, status,
                                stream);
  }
  if (bn == 64)
    return gemm::launch_bn<64>(ta, tb, tbt, ty, tr, y, ep, epilogue, m_cap, m_dev, n, k, status,
                               stream);
  return gemm::launch_bn<128>(ta, tb, tbt, ty, tr, y, ep, epilogue, m_cap, m_dev, n, k, status,
                              stream);
}

}  // namespace dora
