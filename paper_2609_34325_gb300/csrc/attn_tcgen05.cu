// Packed variable-length multi-head self-attention on tcgen05 tensor cores.
// For image i (rows [cu[i], cu[i+1]) of the packed buffer) and head h:
//     O = softmax(Q K^T * scale) V
// with no attention across images and no padding (Sec. 3.5 "Inference").
//
// Work unit = (image, pair of heads, 128-row query tile); a unit walks its keys
// in chunks of up to 96 ("steps"), the image's 32-key blocks dealt evenly over
// the fewest chunks (197 tokens: 96 + 64 + 37).  One persistent CTA per SM owns
// a contiguous range of units, split by estimated cost.  The two heads of a
// unit run on two groups, each with its own softmax warps (one thread per query
// row), PV issuer and half of tensor memory, so that the exponentials of one
// cover the barriers and tensor-memory loads of the other:
//   warp 0       walks the CTA's units, loads the Q tiles of both heads with one
//                TMA box, and per chunk K and V of both heads with one box each
//                (boxes of the rows needed, rounded up to 32), and publishes a
//                descriptor per step and per unit.  Everything a unit needs is
//                the same for both heads but the column, so this one thread
//                keeps up with units of 65 tokens (1,300 cycles each; walking
//                one head a unit it took 2,000 and was the limit there).
//   warp 1       issues S(j) = Q K^T (M=128, N=keys rounded to 16, K=64) of both
//                groups into their S/P buffers j mod 2, once PV(j - 2) is done.
//   warps 2, 3   issue O (+)= P(j) V of group 0 and 1, P read from the buffer that
//                S(j) was in.
//   warps 4-11   softmax, four warps per group: the maximum comes with the loads
//                of S (tcgen05.ld.red), then S is read again 32 columns at a time
//                for 2^x, the row sum and P (bf16), written over columns already
//                read.  Within a unit the reference maximum is only raised when
//                a later chunk exceeds it by more than 2^8, and then O is rescaled
//                in TMEM; otherwise P stays below 2^8 in the old frame, which bf16
//                and fp32 hold exactly as well.  The softmax also zeroes the V rows
//                of a chunk's last 16-key group that lie past the image.
//   warps 12-15  epilogue of both groups: when a unit's last PV is done, O / row
//                sum, each thread storing its row's 128 bytes.
// A last head without a partner (odd head counts) is a unit of its own whose second
// group loads, multiplies and stores nothing of use; its softmax is skipped, so that
// the first one's exponentials have the MUFU alone: 256 x 197 tokens x 1 head 18.6 ->
// 16.6 us, 64 x 577 x 1 28.4 -> 24.1, 87 x 577 x 3 51.3 -> 49.5 (one head a unit, in
// the kernel before: 15.0, 27.0, 48.6).  Skipping its MMAs too gave no more.
// TMEM (256 columns a group): S/P buffers at 0 and 96, O at 192.  Rows past the
// image are computed but never stored; keys past it are masked, and V rows past
// it are zeroed so stale data cannot leak through 0 * NaN.
//
// What bounds it: the serial chain of a step (about 1,700 cycles for 80 keys: the
// maximum 350, the exponentials 1,100 with both groups on the MUFU, the hand-offs
// the rest) and the instruction cache.  The roles' code together must stay in
// it: a softmax unrolled per chunk length (64 KB more code) ran 238 us where this
// loop over 32 columns runs 77, and the inlined waits of all roles are why the
// loader and issuers have one call site for each.  Measured against the kernel
// before it (two threads a row exchanging maxima, MMAs issued from a lane-0
// branch, one query tile at a time), us: 256 x 197 tokens x 12 heads 93.7 ->
// 77.4, the same after one and three deletions 69.9 -> 49.8 and 33.0 -> 25.8, 64 x
// 577 x 12 136.9 -> 107.5, 128 x 257 x 12 91.0 -> 65.0.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "dora_ptx.cuh"
#include "token_ops.cuh"

namespace dora {
namespace attn {

constexpr int BQ = 128;         // query rows per unit
constexpr int KC = 96;          // keys per step, at most
constexpr int kDescRing = 8;    // step descriptors in flight
constexpr int kUnitRing = 4;    // unit descriptors in flight
constexpr int kThreads = 512;   // 16 warps, 128 registers a thread at launch
constexpr int kSoftRegs = 152;  // softmax warps (4-11)
constexpr int kOtherRegs = 96;  // the other eight
constexpr int kSoftWarp0 = 4;
constexpr int kEpiWarp0 = 12;
constexpr uint32_t kTmemCols = 512;
constexpr float kRescaleLog2 = 8.f;    // raise the reference maximum past 2^8
constexpr uint32_t kSleepNs = 200000;  // waiting threads sleep instead of spinning
static_assert(8 * 32 * (kSoftRegs + kOtherRegs) <= kThreads * 128, "registers");

__device__ __forceinline__ uint32_t tmem_sp(int g, int b) {
  return 256u * static_cast<uint32_t>(g) + 96u * static_cast<uint32_t>(b);
}
__device__ __forceinline__ uint32_t tmem_o(int g) { return 256u * static_cast<uint32_t>(g) + 192u; }

// Tensor maps of the packed qkv buffer as [3 heads][t_cap rows][64 columns]:
// m[i] has boxes of 32 (i + 1) rows of two neighbouring heads.
struct QkvMaps {
  CUtensorMap m[BQ / 32];
};

// Step descriptor (one 32-bit word).
constexpr uint32_t kDStage = 0x7u;        // K/V stage
constexpr uint32_t kDKvPar = 1u << 3;     // phase parity of that stage's load
constexpr uint32_t kDFirst = 1u << 4;     // first key chunk of a unit
constexpr uint32_t kDLast = 1u << 5;      // last key chunk of a unit
constexpr uint32_t kDLone = 1u << 6;      // the unit's second head does not exist
constexpr uint32_t kDEnd = 1u << 31;      // no more steps
__device__ __forceinline__ int d_kc(uint32_t d) { return static_cast<int>((d >> 8) & 0x7Fu); }
__device__ __forceinline__ int d_blocks(uint32_t d) { return (d_kc(d) + 31) >> 5; }
__device__ __forceinline__ int d_rows(uint32_t d) { return static_cast<int>((d >> 16) & 0xFFu); }

// HD: head width, 64 or 32 (rows of 128 or 64 bytes, swizzled as wide).
template <int HD>
struct Smem {
  static constexpr int kStages = HD == 64 ? 3 : 6;   // K/V chunk ring, two heads' chunks each
  uint16_t q[2][2][BQ * HD];    // 16 KB each (HD 64): by unit parity and group
  uint16_t k[kStages][2][KC * HD];   // 12 KB each (HD 64): by stage and group
  uint16_t v[kStages][2][KC * HD];
  float lsum[2][4][BQ];         // row sums, by group and unit mod 4
  uint64_t q_full[2];
  uint64_t q_empty[2];
  uint64_t kv_full[kStages];
  uint64_t kv_empty[kStages];   // one arrival per group
  uint64_t s_full[2][2];        // S of a step in the group's S/P buffer b
  uint64_t p_full[2][2];        // P written over it (one arrival per softmax warp)
  uint64_t p_free[2][2];        // PV of buffer b done
  uint64_t o_done[2];           // last PV of a unit done
  uint64_t o_free[2];           // O read out (one arrival per epilogue warp)
  uint64_t l_full[2][4];        // row sums of a unit (one arrival per softmax warp)
  uint64_t sd_full[kDescRing];  // step descriptor published
  uint64_t sd_empty[kDescRing]; // ... read by the three issuers and the eight softmax warps
  uint64_t ud_full[kUnitRing];  // unit descriptor published
  uint64_t ud_empty[kUnitRing]; // ... read by the four epilogue warps
  uint64_t drain[3];
  uint32_t sdesc[kDescRing];
  uint32_t urow[kUnitRing];     // first output row of the unit
  uint32_t uhead[kUnitRing];    // first head | rows << 16
  uint32_t tmem_base;
  int abort_flag;
  int img_begin, unit_begin, img_end, unit_end;   // the CTA's units
  int q_issued, kv_issued;
};
static_assert(sizeof(Smem<64>) <= 227 * 1024 && sizeof(Smem<32>) <= 227 * 1024, "shared memory");

// Descriptor of a tile of HD-wide rows as TMA wrote it, swizzled over 8 rows.
template <int HD>
__device__ __forceinline__ uint64_t tile_desc(uint32_t saddr, uint32_t lbo) {
  return HD == 64 ? sdesc_sw128(saddr, lbo, 1024) : sdesc_sw64(saddr, lbo, 512);
}

// The map's box from row y of heads z and z + 1, one behind the other in dst.
__device__ __forceinline__ void tma_load_heads(void* dst, const CUtensorMap* map, uint64_t* bar,
                                               int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(0), "r"(y), "r"(z), "r"(smem_u32(bar))
      : "memory");
}

// Rows of the image with bounds [b0, b1), clamped to the buffer (0 when its
// start lies outside); lo receives its first row.
__device__ __forceinline__ int clamp_rows(int b0, int b1, int t_cap, int& lo) {
  lo = b0;
  const int n = b1 - b0;
  if (lo < 0 || lo > t_cap) {
    lo = 0;
    return 0;
  }
  return n < 0 ? 0 : (n > t_cap - lo ? t_cap - lo : n);
}

// Query tiles of an image of n rows, and the estimated cost of one: its 16-key
// groups plus a fixed part (about four groups' worth of hand-offs, Q load and
// output).
__device__ __forceinline__ int tiles_of(int n) { return (n + BQ - 1) / BQ; }
__device__ __forceinline__ int unit_cost(int n) { return (n + 15) / 16 + 4; }

// A CTA's units, in image-major, head, query-tile order.  The next image's end
// is fetched an image ahead.
struct Walker {
  const int32_t* cu;
  int batch, pairs, t_cap, img_end, unit_end;
  int img, unit, pair, qt, n, nqt, lo, hi, ahead;
  __device__ __forceinline__ void load_image() {
    const int b0 = hi;
    hi = ahead;
    if (img + 2 <= batch) ahead = __ldg(cu + img + 2);
    n = clamp_rows(b0, hi, t_cap, lo);
    nqt = tiles_of(n);
  }
  __device__ __forceinline__ bool done() const {
    return img > img_end || (img == img_end && unit >= unit_end) || img >= batch;
  }
  __device__ __forceinline__ void settle() {      // to an image with a unit at `unit`
    while (!done() && unit >= pairs * nqt) {
      ++img;
      unit = pair = qt = 0;
      if (img < batch) load_image();
    }
  }
  __device__ __forceinline__ void start(const int32_t* c, int b, int p, int tc, int ib, int ub,
                                        int ie, int ue) {
    cu = c;
    batch = b;
    pairs = p;
    t_cap = tc;
    img = ib;
    unit = ub;
    img_end = ie;
    unit_end = ue;
    pair = qt = n = nqt = lo = hi = ahead = 0;
    if (img >= batch) return;
    hi = __ldg(cu + img);
    ahead = __ldg(cu + img + 1);
    load_image();
    if (nqt > 0) {
      pair = unit / nqt;
      qt = unit - pair * nqt;
    }
    settle();
  }
  __device__ __forceinline__ void next() {
    ++unit;
    if (++qt == nqt) {
      qt = 0;
      ++pair;
    }
    settle();
  }
};

// Whole warp: the first of the CTA's units (end = 0) or the first past them
// (end = 1), as (image, unit of the image).  A unit belongs to CTA
// floor(C * grid / total), C being the cost of the units before it; CTA 0 also
// checks every image against the buffer and max_seqlen.  Each lane owns a
// contiguous block of images whose bounds it reads as one batch of independent
// loads, so the whole search costs about two memory round trips for any batch.
// It is the head of the kernel's latency (2,800 cycles when one warp found both
// bounds in turn): two warps find one each, which takes 0.4-0.8 us off (64 x 197
// x 6 heads 16.1 -> 15.7 us, 64 x 577 x 12 109.3 -> 107.7).
__device__ inline void find_bound(const int32_t* cu, int batch, int pairs, int t_cap,
                                  int max_seqlen, int32_t* status, int end, int& img_at,
                                  int& unit_at) {
  const int lane = threadIdx.x & 31;
  const int per = (batch + 31) / 32;
  const int i0 = min(batch, lane * per), i1 = min(batch, i0 + per);
  long long mine = 0;                   // this lane's images: cost, one head pair
  int c_last = 0;                       // its last unit's cost
#pragma unroll 1
  for (int k0 = i0; k0 < i1; k0 += 8) {
    int bnd[9];
#pragma unroll
    for (int t = 0; t < 9; ++t) bnd[t] = (k0 + t <= i1) ? __ldg(cu + k0 + t) : 0;
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      if (k0 + t < i1) {
        int lo;
        const int n = clamp_rows(bnd[t], bnd[t + 1], t_cap, lo);
        if (n > 0) {
          c_last = unit_cost(n);
          mine += static_cast<long long>(tiles_of(n)) * c_last;
        }
        if (blockIdx.x == 0 && end == 0) {
          const int l0 = bnd[t], len = bnd[t + 1] - l0;
          if (l0 < 0 || l0 > t_cap || len > t_cap - l0 || len > max_seqlen)
            record_status(status, DORA_ERR_DEVICE_SEQLEN);
        }
      }
    }
  }
  long long incl = mine;                // one head pair's cost up to this lane's last image
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  const long long one_pair = __shfl_sync(0xffffffffu, incl, 31);
  const long long total = one_pair * pairs, G = gridDim.x, bx = blockIdx.x;
  // first unit with C * G >= x ((batch, 0) if none): C grows along the order, so
  // it lies in the first lane whose last unit reaches x, found by that lane
  // walking its own images (their bounds are in L1 by now)
  auto locate = [&](long long x, int& img, int& unit) {
    const bool has = c_last > 0 && (pairs * incl - c_last) * G >= x;
    const unsigned m = __ballot_sync(0xffffffffu, has);
    img = batch;
    unit = 0;
    if (m == 0u) return;
    const int owner = __ffs(m) - 1;
    if (lane == owner) {
      long long pre = pairs * (incl - mine);      // cost of the units before image i0
      for (int i = i0; i < i1; ++i) {
        int lo;
        const int n = clamp_rows(cu[i], cu[i + 1], t_cap, lo);
        if (n == 0) continue;
        const int nqt = tiles_of(n);
        const long long c = unit_cost(n), u = static_cast<long long>(pairs) * nqt;
        if ((pre + (u - 1) * c) * G >= x) {
          const long long need = x - pre * G;
          long long w = need > 0 ? (need + c * G - 1) / (c * G) : 0;
          img = i;
          unit = static_cast<int>(w);
          break;
        }
        pre += u * c;
      }
    }
    img = __shfl_sync(0xffffffffu, img, owner);
    unit = __shfl_sync(0xffffffffu, unit, owner);
  };
  img_at = batch;
  unit_at = 0;
  if (one_pair > 0 && bx + end < G) locate((bx + end) * total, img_at, unit_at);
}

__device__ __forceinline__ bool wait_one(uint64_t* bar, uint32_t parity, volatile int* abort) {
  return mbar_wait_sleep(bar, parity, abort, kSleepNs);
}
__device__ __forceinline__ bool wait_warp(uint64_t* bar, uint32_t parity, volatile int* abort) {
  return __all_sync(0xffffffffu, wait_one(bar, parity, abort)) != 0;
}

// -infinity in `count` (1 to 15) columns from taddr on, of this lane's row.
__device__ __forceinline__ void mask_columns(uint32_t taddr, int count) {
  const uint32_t v = __float_as_uint(-INFINITY);
  if (count & 8) {
    const uint32_t v8[8] = {v, v, v, v, v, v, v, v};
    tmem_st8(taddr, v8);
    taddr += 8;
  }
  if (count & 4) {
    tmem_st4(taddr, v);
    taddr += 4;
  }
  if (count & 2) {
    tmem_st2(taddr, v);
    taddr += 2;
  }
  if (count & 1) tmem_st1(taddr, v);
  tmem_st_wait();
}

// p = 2^(s scale - m) of N values, packed to bf16.  The sum (l0 + l1, fp32) is that
// of the rounded values, which are the weights that V gets: their rounding then
// cancels in O / sum for what the rows of V share.  Against 64 bits, relative
// (2-norm), the sum of the values before rounding -> this one: 197 tokens 2.17e-3 ->
// 2.10e-3, 577 2.28e-3 -> 2.23e-3 (the kernels before, whose largest weight was 1 more
// often and so not rounded, 2.12e-3 and 2.26e-3).  The fp32 + bf16 adds cost 0-0.6 %
// of the kernel against paired fp32 adds; unpacking the values for those 1-3.6 %.
template <int N>
__device__ __forceinline__ void exp_pack(const uint32_t (&a)[N], uint32_t (&p)[N / 2], uint64_t sc,
                                         uint64_t nm, float& l0, float& l1) {
#pragma unroll
  for (int e = 0; e < N; e += 2) {
    float x0, x1;
    f2_unpack(f2_fma(f2_pack(__uint_as_float(a[e]), __uint_as_float(a[e + 1])), sc, nm), x0, x1);
    p[e >> 1] = pack_bf16x2(ex2_approx(x0), ex2_approx(x1));
    add_bf16x2(l0, l1, p[e >> 1]);
  }
}

// A grid with a CTA for every possible unit needs no search: CTA b has query
// tile b mod tiles of pair (b / tiles) mod pairs of image b / (tiles pairs), if
// the image is that long (the last one also has what lies past max_seqlen, and
// each image's first CTA checks it).  One thread, and 1.1 us less than the
// search: 1 x 197 x 3 heads 8.6 -> 7.5 us, 8 images 8.9 -> 7.9.
__device__ __forceinline__ void own_unit(const int32_t* cu, int pairs, int tiles, int t_cap,
                                         int max_seqlen, int32_t* status, int& ib, int& ub,
                                         int& ie, int& ue) {
  const int row = static_cast<int>(blockIdx.x) / tiles;
  const int qt = static_cast<int>(blockIdx.x) - row * tiles;
  ib = ie = row / pairs;
  const int pair = row - ib * pairs;
  const int b0 = __ldg(cu + ib), b1 = __ldg(cu + ib + 1);
  int lo;
  const int nqt = tiles_of(clamp_rows(b0, b1, t_cap, lo));
  ub = pair * nqt + min(qt, nqt);
  ue = pair * nqt + (qt == tiles - 1 ? nqt : min(qt + 1, nqt));
  if (pair == 0 && qt == 0) {
    const int len = b1 - b0;
    if (b0 < 0 || b0 > t_cap || len > t_cap - b0 || len > max_seqlen)
      record_status(status, DORA_ERR_DEVICE_SEQLEN);
  }
}

template <int HD>
__global__ void __launch_bounds__(kThreads, 1)
    varlen_attn_kernel(const __grid_constant__ QkvMaps mp, const int32_t* __restrict__ cu,
                       int batch, int max_seqlen, int t_cap, int heads, float scale_log2,
                       uint16_t* __restrict__ out, int32_t* status) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  pdl_trigger();
  if (smem_u32(smem_raw) & 1023u) {
    pdl_wait();
    if (threadIdx.x == 0) record_status(status, DORA_ERR_UNSUPPORTED);
    return;
  }
  Smem<HD>& s = *reinterpret_cast<Smem<HD>*>(smem_raw);
  constexpr int kStages = Smem<HD>::kStages;
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int dim = heads * HD;

  if (threadIdx.x == 64) {
    for (int g = 0; g < 2; ++g) {
      for (int b = 0; b < 2; ++b) {
        mbar_init(&s.s_full[g][b], 1);
        mbar_init(&s.p_full[g][b], 4);
        mbar_init(&s.p_free[g][b], 1);
      }
      mbar_init(&s.q_full[g], 1);
      mbar_init(&s.q_empty[g], 1);
      mbar_init(&s.o_done[g], 1);
      mbar_init(&s.o_free[g], 4);
      for (int i = 0; i < 4; ++i) mbar_init(&s.l_full[g][i], 4);
      mbar_init(&s.drain[g], 1);
    }
    for (int i = 0; i < kDescRing; ++i) {
      mbar_init(&s.sd_full[i], 1);
      mbar_init(&s.sd_empty[i], 11);
    }
    for (int i = 0; i < kStages; ++i) {
      mbar_init(&s.kv_full[i], 1);
      mbar_init(&s.kv_empty[i], 2);
    }
    for (int i = 0; i < kUnitRing; ++i) {
      mbar_init(&s.ud_full[i], 1);
      mbar_init(&s.ud_empty[i], 4);
    }
    mbar_init(&s.drain[2], 1);
    s.abort_flag = 0;
    s.q_issued = s.kv_issued = 0;
    fence_barrier_init();
  }
  if (warp == 3) tmem_alloc(&s.tmem_base, kTmemCols);
  // the set-up above overlaps the previous kernel; global memory waits for it
  pdl_wait();
  const int pairs = (heads + 1) / 2, tiles = tiles_of(max_seqlen);
  if (static_cast<long long>(batch) * pairs * tiles == gridDim.x) {
    if (threadIdx.x == 0)
      own_unit(cu, pairs, tiles, t_cap, max_seqlen, status, s.img_begin, s.unit_begin, s.img_end,
               s.unit_end);
  } else if (warp < 2) {
    int img, unit;
    find_bound(cu, batch, pairs, t_cap, max_seqlen, status, warp, img, unit);
    if (lane == 0) {
      (warp == 0 ? s.img_begin : s.img_end) = img;
      (warp == 0 ? s.unit_begin : s.unit_end) = unit;
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s.tmem_base;
  volatile int* abort = &s.abort_flag;

  if (warp < kSoftWarp0) {
    setmaxnreg_dec<kOtherRegs>();
    if (warp == 0) {
      // ---------------- scheduler + TMA producer ----------------
      if (elect_one()) {
        Walker wk;
        wk.start(cu, batch, (heads + 1) / 2, t_cap, s.img_begin, s.unit_begin, s.img_end,
                 s.unit_end);
        int loads = 0, stg = 0;
        uint32_t par = 0;                       // chunks loaded; their stage and its phase parity
        int dn = 0;                             // steps published
        int u = 0;                              // units begun
        bool ok = true;
        int n_of = -1, nch = 0, base = 0, more = 0;   // chunks of images of n_of rows
        auto desc = [&](uint32_t d) -> bool {
          const int i = dn % kDescRing;
          if (!wait_one(&s.sd_empty[i], ((dn / kDescRing) & 1) ^ 1, abort)) return false;
          s.sdesc[i] = d;
          mbar_arrive(&s.sd_full[i]);
          ++dn;
          return true;
        };
        for (; ok && !wk.done(); wk.next(), ++u) {
          // the unit's Q tiles and its descriptor
          const int i = u % kUnitRing, qb = u & 1, row = wk.lo + wk.qt * BQ;
          const int rows = min(BQ, wk.n - wk.qt * BQ), r32 = (rows + 31) >> 5;
          if (!(ok = wait_one(&s.q_empty[qb], ((u >> 1) & 1) ^ 1, abort))) break;
          mbar_arrive_expect_tx(&s.q_full[qb], 2 * r32 * 32 * HD * 2);
          tma_load_heads(s.q[qb], &mp.m[r32 - 1], &s.q_full[qb], row, 2 * wk.pair);
          s.q_issued = u + 1;
          if (!(ok = wait_one(&s.ud_empty[i], ((u / kUnitRing) & 1) ^ 1, abort))) break;
          s.urow[i] = static_cast<uint32_t>(row);
          s.uhead[i] = static_cast<uint32_t>(2 * wk.pair) | (static_cast<uint32_t>(rows) << 16);
          mbar_arrive(&s.ud_full[i]);
          // its K/V chunks: the 32-key blocks dealt over the fewest chunks
          if (wk.n != n_of) {
            n_of = wk.n;
            const int blocks = (n_of + 31) >> 5;
            nch = (blocks + KC / 32 - 1) / (KC / 32);
            base = blocks / nch;
            more = blocks - base * nch;
          }
          int off = 0;
          for (int c = 0; c < nch; ++c) {
            const int cb = base + (c < more ? 1 : 0);       // 32-key blocks of the chunk
            if (!(ok = wait_one(&s.kv_empty[stg], par ^ 1, abort))) break;
#ifdef DORA_TEST_WITHHOLD_KV_LOAD
            // timeout-path test library only: CTA 0 never issues its first K/V
            // load nor its expected bytes, so the S issuer's bounded wait on
            // that stage runs out with no copy in flight
            const bool withhold = blockIdx.x == 0 && loads == 0;
#else
            constexpr bool withhold = false;
#endif
            if (!withhold) {
              mbar_arrive_expect_tx(&s.kv_full[stg], 4 * cb * 32 * HD * 2);
              tma_load_heads(s.k[stg], &mp.m[cb - 1], &s.kv_full[stg], wk.lo + off,
                             heads + 2 * wk.pair);
              tma_load_heads(s.v[stg], &mp.m[cb - 1], &s.kv_full[stg], wk.lo + off,
                             2 * (heads + wk.pair));
            }
            s.kv_issued = ++loads;
            ok = desc(static_cast<uint32_t>(stg) | (par ? kDKvPar : 0u) | (c == 0 ? kDFirst : 0u) |
                      (c == nch - 1 ? kDLast : 0u) | (2 * wk.pair + 1 == heads ? kDLone : 0u) |
                      (static_cast<uint32_t>(min(32 * cb, n_of - off)) << 8) |
                      (static_cast<uint32_t>(rows) << 16));
            if (!ok) break;
            if (++stg == kStages) {
              stg = 0;
              par ^= 1u;
            }
            off += 32 * cb;
          }
        }
        if (ok && desc(kDEnd)) {
          const int i = u % kUnitRing;          // no more units
          if (wait_one(&s.ud_empty[i], ((u / kUnitRing) & 1) ^ 1, abort)) {
            s.uhead[i] = 0xFFFFFFFFu;
            mbar_arrive(&s.ud_full[i]);
          }
        }
      }
    } else if (warp == 1) {
      // ---------------- S issuer of both groups ----------------
      // S(j) = Q K^T of a group goes into S/P buffer j mod 2 once PV(j - 2) has read
      // its P there.
      if (elect_one()) {
        int u = 0;                              // units whose S are all issued
        bool ok = true;
        for (int j = 0; ok; ++j) {
          const int i = j % kDescRing, b = j & 1, qb = u & 1;
          if (!wait_one(&s.sd_full[i], (j / kDescRing) & 1, abort)) break;
          const uint32_t d = s.sdesc[i];
          mbar_arrive(&s.sd_empty[i]);
          if (d & kDEnd) break;
          const int stg = static_cast<int>(d & kDStage), groups = (d_kc(d) + 15) >> 4;
          if (!wait_one(&s.kv_full[stg], (d & kDKvPar) ? 1u : 0u, abort)) break;
          if ((d & kDFirst) && !wait_one(&s.q_full[qb], (u >> 1) & 1, abort)) break;
          const uint32_t id_s = idesc_bf16(BQ, 16 * groups, false);
          // a load of two heads puts the second right behind the first
          const int q_step = ((d_rows(d) + 31) & ~31) * HD, k_step = 32 * d_blocks(d) * HD;
#pragma unroll 1
          for (int g = 0; g < 2; ++g) {
            if (j >= 2 && !(ok = wait_one(&s.p_free[g][b], ((j >> 1) - 1) & 1, abort))) break;
            tc_fence_after();
            const uint64_t qd = tile_desc<HD>(smem_u32(&s.q[qb][0][0] + g * q_step), 16);
            const uint64_t kd = tile_desc<HD>(smem_u32(&s.k[stg][0][0] + g * k_step), 16);
            const uint32_t dt = tmem + tmem_sp(g, b);
#pragma unroll
            for (int k = 0; k < HD / 16; ++k)
              mma_bf16_ss(dt, qd + 2 * k, kd + 2 * k, id_s, k > 0 ? 1u : 0u);
            mma_commit(&s.s_full[g][b]);
          }
          if (d & kDLast) {
            mma_commit(&s.q_empty[qb]);
            ++u;
          }
        }
        mma_commit(&s.drain[2]);
        mbar_wait_limited(&s.drain[2], 0, kWaitLimitNs);
      }
    } else {
      // ---------------- PV issuer of group g ----------------
      // O (+)= P(j) V once P(j) is written and, on a unit's first chunk, the
      // epilogue has read the group's previous O.
      if (elect_one()) {
        const int g = warp - 2;
        int up = 0;                             // units whose PVs are all issued
        for (int j = 0;; ++j) {
          const int i = j % kDescRing, b = j & 1;
          if (!wait_one(&s.sd_full[i], (j / kDescRing) & 1, abort)) break;
          const uint32_t d = s.sdesc[i];
          mbar_arrive(&s.sd_empty[i]);
          if (d & kDEnd) break;
          const int nk = (d_kc(d) + 15) >> 4, stg = static_cast<int>(d & kDStage);
          const uint64_t vd =
              tile_desc<HD>(smem_u32(&s.v[stg][0][0] + g * 32 * d_blocks(d) * HD), 16 * HD);
          const uint32_t ot = tmem + tmem_o(g), at = tmem + tmem_sp(g, b);
          constexpr uint32_t id_o = idesc_bf16(BQ, HD, true);
          if ((d & kDFirst) && up > 0 && !wait_one(&s.o_free[g], (up - 1) & 1, abort)) break;
          if (!wait_one(&s.p_full[g][b], (j >> 1) & 1, abort)) break;
          tc_fence_after();
          mma_bf16_ts(ot, at, vd, id_o, (d & kDFirst) ? 0u : 1u);
#pragma unroll
          for (int kk = 1; kk < KC / 16; ++kk)   // 16 keys: 2 HD 16-byte pieces of V, 8 P columns
            if (kk < nk) mma_bf16_ts(ot, at + 8u * kk, vd + 2u * HD * kk, id_o, 1u);
          mma_commit(&s.p_free[g][b]);
          if (d & kDLast) {
            mma_commit(&s.o_done[g]);
            ++up;
          }
          mma_commit(&s.kv_empty[stg]);
        }
        mma_commit(&s.drain[g]);
        mbar_wait_limited(&s.drain[g], 0, kWaitLimitNs);
      }
    }
  } else if (warp < kEpiWarp0) {
    // ---------------- softmax: one thread per query row ----------------
    setmaxnreg_inc<kSoftRegs>();
    const int g = (warp - kSoftWarp0) >> 2;
    const int quarter = warp & 3;
    const int r = quarter * 32 + lane;                   // query row of the tile (TMEM lane)
    const uint32_t lane_sel = static_cast<uint32_t>(quarter * 32) << 16;
    const uint64_t sc = f2_pack(scale_log2, scale_log2);
    const uint32_t lone = g == 1 ? kDLone : 0u;
    float m_ref = 0.f, l = 0.f;                          // reference (log2 units), row sum
    int u = 0;                                           // units finished
    auto step = [&](int j, uint32_t d) -> bool {
      const int kc = d_kc(d), groups = (kc + 15) >> 4, b = j & 1;
      // warp-uniform: rows of the tile, and not the head that a lone last one lacks
      const bool live = quarter * 32 < d_rows(d) && !(d & lone);
      const uint32_t tsp = tmem + lane_sel + tmem_sp(g, b);
      if (!wait_warp(&s.s_full[g][b], (j >> 1) & 1, abort)) return false;
      tc_fence_after();
      if (kc & 15) {
        // the last 16-key group reaches past the image: mask its S columns, and
        // zero its V rows (S is done, so the chunk's load landed; whole rows)
        const int past = 16 * groups - kc;
        if (live) mask_columns(tsp + static_cast<uint32_t>(kc), past);
        constexpr int kRow16 = HD / 8;                   // 16-byte pieces of a row
        if (r < past * kRow16)
          reinterpret_cast<uint4*>(&s.v[d & kDStage][0][0] +
                                   g * 32 * d_blocks(d) * HD)[kc * kRow16 + r] =
              make_uint4(0u, 0u, 0u, 0u);
        fence_proxy_async_smem();
      }
      if (live) {
        const int blocks = groups >> 1;                  // 32 columns each; then half a block
        const uint32_t tail = tsp + 32u * static_cast<uint32_t>(blocks);
        const bool first = (d & kDFirst) != 0;
        // the maximum is formed by the loads themselves
        float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
        uint32_t sv[KC];                                 // read again below, 32 at a time
#pragma unroll
        for (int i = 0; i < KC / 32; ++i)
          if (i < blocks)
            tmem_ld_max32(tsp + 32u * i, *reinterpret_cast<uint32_t(*)[32]>(&sv[32 * i]), mx[i]);
        if (groups & 1) {
          uint32_t a[16];
          tmem_ld_max16(tail, a, mx[3]);
        }
        tmem_ld_wait();
        const float mc = max3f(mx[0], mx[1], fmaxf(mx[2], mx[3])) * scale_log2;
        float alpha = 1.f;
        if (first) {
          m_ref = mc;
          l = 0.f;
        } else if (mc > m_ref + kRescaleLog2) {
          alpha = ex2_approx(m_ref - mc);
          l *= alpha;
          m_ref = mc;
        }
        // a chunk of -infinities alone (only from infinite inputs) weighs nothing
        const float neg_m = m_ref == -INFINITY ? 0.f : -m_ref;
        const uint64_t nm = f2_pack(neg_m, neg_m);
        float l0 = l, l1 = 0.f;
#pragma unroll 1
        for (int i = 0; i < blocks; ++i) {
          uint32_t a[32], p[16];
          tmem_ld32(tsp + 32u * i, a);
          tmem_ld_wait();
          exp_pack<32>(a, p, sc, nm, l0, l1);
          tmem_st16(tsp + 16u * i, p);                   // over columns already read
        }
        if (groups & 1) {
          uint32_t a[16], p[8];
          tmem_ld16(tail, a);
          tmem_ld_wait();
          exp_pack<16>(a, p, sc, nm, l0, l1);
          tmem_st8(tsp + 16u * blocks, p);
        }
        l = l0 + l1;
        if (__any_sync(0xffffffffu, alpha != 1.f)) {
          // O holds the chunks before this one once their PV is done: bring it
          // to the raised reference before this chunk's PV
          if (!wait_warp(&s.p_free[g][b ^ 1], ((j - 1) >> 1) & 1, abort)) return false;
          tc_fence_after();
          const uint32_t to = tmem + lane_sel + tmem_o(g);
#pragma unroll 1
          for (int h = 0; h < HD / 16; ++h) {
            uint32_t o[16];
            tmem_ld16(to + 16u * h, o);
            tmem_ld_wait();
#pragma unroll
            for (int e = 0; e < 16; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * alpha);
            tmem_st16(to + 16u * h, o);
          }
        }
        tmem_st_wait();
      }
      if (d & kDLast) s.lsum[g][u & 3][r] = l;
      warp_arrive(&s.p_full[g][b]);
      if (d & kDLast) {
        if (lane == 0) mbar_arrive(&s.l_full[g][u & 3]);
        ++u;
      }
      return true;
    };
    for (int j = 0;; ++j) {
      const int i = j % kDescRing;
      if (!wait_warp(&s.sd_full[i], (j / kDescRing) & 1, abort)) break;
      const uint32_t d = s.sdesc[i];
      __syncwarp();
      if (lane == 0) mbar_arrive(&s.sd_empty[i]);
      if ((d & kDEnd) || !step(j, d)) break;
    }
  } else {
    // ---------------- epilogue: O / row sum ----------------
    setmaxnreg_dec<kOtherRegs>();
    const int quarter = warp & 3;
    const int r = quarter * 32 + lane;
    const uint32_t lane_sel = static_cast<uint32_t>(quarter * 32) << 16;
    const bool whole = (reinterpret_cast<uintptr_t>(out) & 31u) == 0;   // 32-byte stores
#pragma unroll 1
    for (int u = 0;; ++u) {
      const int i = u % kUnitRing;
      // one descriptor per unit, then an end marker
      if (!wait_warp(&s.ud_full[i], (u / kUnitRing) & 1, abort)) break;
      const uint32_t row0 = s.urow[i], hd = s.uhead[i];
      __syncwarp();
      if (lane == 0) mbar_arrive(&s.ud_empty[i]);
      if (hd == 0xFFFFFFFFu) break;
      const int rows = static_cast<int>(hd >> 16), head = static_cast<int>(hd & 0xFFFFu);
      bool ok = true;
#pragma unroll 1
      for (int g = 0; g < 2; ++g) {
        if (!(ok = wait_warp(&s.l_full[g][u & 3], (u >> 2) & 1, abort))) break;
        const bool live = quarter * 32 < rows && head + g < heads;   // warp-uniform
        const float inv = live ? 1.0f / s.lsum[g][u & 3][r] : 1.f;
        if (!(ok = wait_warp(&s.o_done[g], u & 1, abort))) break;
        tc_fence_after();
        uint16_t* const dst = out + static_cast<size_t>(row0 + r) * dim + (head + g) * HD;
#pragma unroll 1
        for (int h = 0; h < HD / 32; ++h) {
          uint32_t o[32], w[16];
          if (live) {
            tmem_ld32(tmem + lane_sel + tmem_o(g) + 32u * h, o);
            tmem_ld_wait();
          }
          if (h == HD / 32 - 1) warp_arrive(&s.o_free[g]);
          if (live && r < rows) {
#pragma unroll
            for (int e = 0; e < 16; ++e)
              w[e] = pack_bf16x2(__uint_as_float(o[2 * e]) * inv,
                                 __uint_as_float(o[2 * e + 1]) * inv);
            uint32_t* const d = reinterpret_cast<uint32_t*>(dst + 32 * h);
            if (whole) {
              st_global_32(d, &w[0]);
              st_global_32(d + 8, &w[8]);
            } else {
#pragma unroll
              for (int c = 0; c < 4; ++c)
                reinterpret_cast<uint4*>(d)[c] =
                    make_uint4(w[4 * c], w[4 * c + 1], w[4 * c + 2], w[4 * c + 3]);
            }
          }
        }
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
      // let the last TMA load of every buffer land (earlier ones were consumed)
      for (int u = max(0, s.q_issued - 2); u < s.q_issued; ++u)
        mbar_wait_limited(&s.q_full[u & 1], (u >> 1) & 1, 100ull * 1000 * 1000);
      for (int c = max(0, s.kv_issued - kStages); c < s.kv_issued; ++c)
        mbar_wait_limited(&s.kv_full[c % kStages], (c / kStages) & 1, 100ull * 1000 * 1000);
    }
    __syncthreads();
  }
  if (warp == 3) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

}  // namespace attn

namespace attn {
template <int HD>
static cudaError_t launch(const uint16_t* qkv, const int32_t* cu, int32_t batch,
                          int32_t max_seqlen, int32_t t_cap, int32_t heads, float scale,
                          uint16_t* out, int32_t* status, cudaStream_t stream) {
  QkvMaps mp;
  for (int i = 0; i < BQ / 32; ++i)
    if (encode_tmap_heads(&mp.m[i], qkv, static_cast<uint64_t>(t_cap),
                          static_cast<uint64_t>(3) * heads, HD, 32u * (i + 1)) != 0)
      return cudaErrorInvalidValue;
  const size_t smem = sizeof(Smem<HD>);
  const cudaError_t e =
      cudaFuncSetAttribute(varlen_attn_kernel<HD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  // Any bound is accepted; a length past t_cap is flagged as one past the buffer.
  if (max_seqlen > t_cap) max_seqlen = t_cap;
  const long long units = static_cast<long long>(batch) * ((heads + 1) / 2) *
                          ((static_cast<long long>(max_seqlen) + BQ - 1) / BQ);
  const long long cap = num_sms();
  const int grid = static_cast<int>(units < cap ? units : cap);
  return launch_pdl(varlen_attn_kernel<HD>, dim3(grid), dim3(kThreads), smem, stream, mp, cu,
                    batch, max_seqlen, t_cap, heads, scale * 1.4426950408889634f, out, status);
}
}  // namespace attn

cudaError_t launch_varlen_attn(const uint16_t* qkv, const int32_t* cu, int32_t batch,
                               int32_t max_seqlen, int32_t t_cap, int32_t heads, float scale,
                               uint16_t* out, int32_t* status, cudaStream_t stream,
                               int32_t head_dim) {
  if (batch == 0 || t_cap == 0 || max_seqlen == 0) return cudaSuccess;
  return head_dim == 32 ? attn::launch<32>(qkv, cu, batch, max_seqlen, t_cap, heads, scale, out,
                                           status, stream)
                        : attn::launch<64>(qkv, cu, batch, max_seqlen, t_cap, heads, scale, out,
                                           status, stream);
}

}  // namespace dora
