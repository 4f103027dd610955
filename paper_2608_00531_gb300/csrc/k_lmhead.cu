// Stage 5 fused with the target's LM head (Sec. 3.5, Eq. 4; greedy decoding,
// Sec. 4.1): the target's greedy token at every tree node computed from the
// node's final hidden state, as the epilogue of the LM-head contraction
//   logits[r][v] = hidden[r] . w_lm[v],   targ[r] = first argmax_v logits[r][v],
// so that the rows x vocab logits never reach HBM.
//
// The contraction runs on the tcgen05 tensor cores in pairs of SMs
// (cta_group::2): a pair owns one N tile of hidden rows (up to 256 columns of
// the accumulator) and a contiguous range of the vocabulary, taken 256 ids at a
// time as the M = 256 operand, 128 per CTA.  The pairs that share a vocab range
// run side by side, so each weight tile is read from HBM about once and served
// to the other N tiles from L2.
//   warp 0   producer (each CTA): TMA loads of the 64-wide K slices of its 128
//            weight rows and of its half of the hidden tile (128-byte swizzle)
//            into a ring of up to 12 stages; both CTAs' copies complete on the
//            first CTA's barrier;
//   warp 1   MMA issuer (an elected lane of the first CTA): per K slice four
//            M256 N<=256 K16 bf16 products accumulating in float32 in both
//            CTAs' TMEM; two accumulators alternate between vocab tiles;
//   warps 2-9 epilogue (each CTA): a TMEM lane is a vocab id, a column a hidden
//            row; the warp takes each column's maximum and its first lane (a
//            float redux and a ballot), and the lane that keeps the column replaces
//            its running (max, id) when strictly greater, so the lowest id
//            wins ties.
// The pair merges its 8 lane quarters through the first CTA's shared memory and
// writes one (max, id) per row for its vocab range; a second kernel takes the
// first maximum over the ranges.  Waits are bounded: on expiry a CTA flags
// CURE_DEVERR_TIMEOUT, drains its copies and products, frees its TMEM and
// leaves, and its pair reports no maximum for the range.
//
// What bounds it: with one tile of rows the weight's bytes (21 x 4096 x 128256:
// 159 us, 6.6 TB/s); with several the tensor pipe at the clock that the power
// limit leaves (817 x 4096 x 151936: 640 us, 448 cycles a K slice of 224
// columns, the products' own time, at 1.44 GHz; the pipe is 94 % busy in an
// isolated launch of 583 us).  With hidden rows as the N operand 817 rows pad to
// 896 columns of four tiles that use every SM, and a few rows to 32 instead of a
// 128-row operand; pairing halves each SM's share of the hidden tile, so the
// ring holds 7 to 12 slices.  Before (one SM per 128 hidden rows x 256 ids, 4
// slices): 192 us and 684 us at these shapes, 28.1 instead of 11.5 us for 9 x
// 1024 x 32000 (its reduction over the ranges was a serial loop per row), 103
// instead of 86 for 257 x 2048 x 100001.  The epilogue's maxima are float redux
// instructions: with integer keys made of the values it outlasted the products
// at short K (1000 x 1024 x 33000 45.8 us, now 39.0).
#include <cudaTypedefs.h>
#include <limits.h>

#include <algorithm>
#include <atomic>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace cure {
namespace {

using namespace tc;

constexpr int BV = 128;            // vocab ids per CTA (TMEM lanes); 256 per pair
constexpr int BN = 256;            // most hidden rows per tile (accumulator columns)
constexpr int BK = 64;             // K slice: one 128-byte swizzled row
constexpr int kMaxStages = 12;
constexpr int kThreads = 320;      // 10 warps
constexpr int kEpiWarps = 8;
constexpr uint32_t kTmemCols = 512;
constexpr int kABytes = BV * BK * 2;  // 16 KiB
enum { B_FULL = 0, B_EMPTY = kMaxStages, B_ACCFULL = 2 * kMaxStages, B_ACCEMPTY = B_ACCFULL + 2,
       B_DRAIN = B_ACCEMPTY + 2, B_NEVER = B_DRAIN + 1, kNumBars = B_NEVER + 1 };
constexpr int kOffBars = 0;
constexpr int kOffTmemSlot = 8 * kNumBars;
constexpr int kOffAbort = kOffTmemSlot + 4;
constexpr int kOffRing = 1024;     // stages start 1024-byte aligned
constexpr int kSmemMax = 232448 - 1024;  // less the room to align the base
static_assert(kOffAbort + 4 <= kOffRing, "barriers fit below the ring");

constexpr int stage_bytes(int nt) { return kABytes + nt / 2 * BK * 2; }
constexpr int stages_of(int nt) {
  const int n = (kSmemMax - kOffRing) / stage_bytes(nt);
  return n < kMaxStages ? n : kMaxStages;
}

struct LmArgs {
  int M, d, V;
  int nt, n_tiles;          // hidden rows per tile, tiles
  int groups, v_tiles;      // vocab ranges, 256-id vocab tiles
  int stages;
  float* part_val;          // [groups][M] maxima
  int32_t* part_idx;        // [groups][M]
  int* err;
  int expire_rank;          // self-test: this CTA of each pair lets an epilogue wait run out (-1: none)
  long long expire_limit;   // after this many cycles
};

// The warp's maximum (NaNs passed over), in every lane: one instruction.
__device__ __forceinline__ float warp_max(float x) {
  float m;
  asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(m) : "f"(x));
  return m;
}

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The address of this shared-memory variable in the pair's first CTA.
__device__ __forceinline__ uint32_t in_first_cta(uint32_t addr) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(addr));
  return r;
}
__device__ __forceinline__ void arrive_cluster(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void st_cluster(uint32_t addr, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

// All lanes of the warp wait; the warp proceeds only if every lane succeeded.
__device__ __forceinline__ bool wait_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* err) {
  const bool ok = wait_bounded(bar, parity, abort_flag, err, true);
  return __all_sync(0xffffffffu, ok);
}
// One lane of the (converged) warp.  The issuing warp runs as a whole and elects
// the lane inside the asm (four products then take 124 cycles to issue; behind a
// branch to lane 0 they took 265).
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred el;\n\telect.sync _|el, 0xffffffff;\n\tselp.u32 %0, 1, 0, el;\n\t}\n" : "=r"(p));
  return p != 0;
}

// A copy into this CTA that completes on a barrier of either CTA of the pair.
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2"
      " [%0], [%1, {%3, %4}], [%2];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1)
      : "memory");
}

// Four M256 K16 products of the pair over one 64-wide K slice (descriptors step
// by 32 bytes, 2 in 16-byte units, inside the 128-byte swizzled rows).
__device__ __forceinline__ void mma_kslice(uint32_t d, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p0, pt, el;\n\t.reg .b64 a, b;\n\t"
      "elect.sync _|el, 0xffffffff;\n\t"
      "setp.ne.b32 p0, %4, 0;\n\t"
      "setp.eq.b32 pt, %4, %4;\n\t"
      "@el tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p0;\n\t"
      "add.s64 a, %1, 2;\n\tadd.s64 b, %2, 2;\n\t"
      "@el tcgen05.mma.cta_group::2.kind::f16 [%0], a, b, %3, pt;\n\t"
      "add.s64 a, %1, 4;\n\tadd.s64 b, %2, 4;\n\t"
      "@el tcgen05.mma.cta_group::2.kind::f16 [%0], a, b, %3, pt;\n\t"
      "add.s64 a, %1, 6;\n\tadd.s64 b, %2, 6;\n\t"
      "@el tcgen05.mma.cta_group::2.kind::f16 [%0], a, b, %3, pt;\n\t}\n" ::"r"(d),
      "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
      : "memory");
}
// Arrive on `bar` in both CTAs once the pair's products issued so far are done.
__device__ __forceinline__ void commit_pair(uint32_t bar) {
  asm volatile(
      "{\n\t.reg .pred el;\n\telect.sync _|el, 0xffffffff;\n\t"
      "@el tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n\t}\n" ::"r"(bar),
      "h"((uint16_t)3)
      : "memory");
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
lm_head_argmax_kernel(const __grid_constant__ CUtensorMap mh, const __grid_constant__ CUtensorMap mw,
                      const LmArgs A) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t sb = (raw + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (sb - raw);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  auto bar = [&](int i) { return sb + kOffBars + 8u * (uint32_t)i; };
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + kOffAbort);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + kOffTmemSlot);

  const int rank = (int)cluster_rank();
  const int pair = (int)blockIdx.x >> 1;
  const int n0 = (pair % A.n_tiles) * A.nt;  // first hidden row of the tile
  const int g = pair / A.n_tiles;
  const int t_lo = (int)((int64_t)g * A.v_tiles / A.groups);
  const int t_hi = (int)((int64_t)(g + 1) * A.v_tiles / A.groups);
  const int ntl = t_hi - t_lo;
  const int KS = A.d / BK, NS = A.stages;
  const int stage = kABytes + A.nt / 2 * BK * 2;

  if (threadIdx.x == 0) {
    for (int s = 0; s < NS; ++s) {
      mbar_init(bar(B_FULL + s), 1);
      mbar_init(bar(B_EMPTY + s), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(bar(B_ACCFULL + a), 1);
      mbar_init(bar(B_ACCEMPTY + a), 2 * kEpiWarps);  // one arrival per epilogue warp of the pair
    }
    mbar_init(bar(B_DRAIN), 1);
    mbar_init(bar(B_NEVER), 1);  // nothing arrives on it
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 0 && lane == 0) {
    tma_prefetch_desc(&mh);
    tma_prefetch_desc(&mw);
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sb + kOffTmemSlot),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // both CTAs' barriers and TMEM are ready
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_begin();

  if (warp == 0) {
    // ---------------------------------------------------------------- producer
    if (lane == 0) {
      // ring position: stage s, round parity ph (no division by the stage
      // count: the issuing lanes' instructions set the pace of a slice)
      int s = 0, it = 0;
      uint32_t ph = 0, st = sb + kOffRing;
      const uint32_t full0 = in_first_cta(bar(B_FULL));
      const int h0 = n0 + rank * (A.nt / 2);
      bool ok = true;
      for (int t = t_lo; t < t_hi && ok; ++t) {
        const int v0 = (2 * t + rank) * BV;
        for (int k = 0; k < KS; ++k) {
          // (the first round's wait returns at once: the barrier's phase before)
          if (!wait_bounded(bar(B_EMPTY + s), ph ^ 1u, abort_flag, A.err, true)) {
            ok = false;
            break;
          }
          if (rank == 0) mbar_arrive_expect_tx(bar(B_FULL + s), 2 * stage);  // both CTAs' copies
          tma_load_2d(st, &mw, full0 + 8u * s, k * BK, v0);
          tma_load_2d(st + kABytes, &mh, full0 + 8u * s, k * BK, h0);
          ++it;
          st += stage;
          if (++s == NS) {
            s = 0;
            ph ^= 1u;
            st = sb + kOffRing;
          }
        }
      }
      if (!ok) {  // let the copies in flight land before the CTA's smem goes away
        if (rank == 0) {
          for (int j = max(0, it - NS); j < it; ++j)
            wait_bounded(bar(B_FULL + j % NS), (j / NS) & 1, abort_flag, A.err, false);
        } else {  // they complete on the other CTA's barriers: a time far above a copy's
          const long long t0 = clock64();
          while (clock64() - t0 < (1 << 20)) {
          }
        }
      }
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer
    if (rank == 0) {
      const uint32_t idesc = idesc_bf16_f32(2 * BV, A.nt, false);
      int s = 0;
      uint32_t ph = 0;
      const uint64_t ad0 = sdesc_sw128(sb + kOffRing, 16, 1024), bd0 = sdesc_sw128(sb + kOffRing + kABytes, 16, 1024);
      uint32_t off = 0;  // of the stage, in the descriptors' 16-byte units
      bool ok = true;
      for (int t = 0; t < ntl && ok; ++t) {
        const int a = t & 1;
        if (t >= 2 && !wait_warp(bar(B_ACCEMPTY + a), ((t >> 1) & 1) ^ 1, abort_flag, A.err)) {
          ok = false;
          break;
        }
        tc_fence_after();
        for (int k = 0; k < KS; ++k) {
          if (!wait_warp(bar(B_FULL + s), ph, abort_flag, A.err)) {
            ok = false;
            break;
          }
          tc_fence_after();
          mma_kslice(tmem + a * BN, ad0 + off, bd0 + off, idesc, k > 0 ? 1u : 0u);
          commit_pair(bar(B_EMPTY + s));
          off += (uint32_t)stage >> 4;
          if (++s == NS) {
            s = 0;
            ph ^= 1u;
            off = 0;
          }
        }
        if (ok) commit_pair(bar(B_ACCFULL + a));
      }
      // every product issued has completed before TMEM is freed
      if (elect_one())
        asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar(B_DRAIN))
                     : "memory");
      __syncwarp();
      wait_bounded(bar(B_DRAIN), 0, abort_flag, A.err, false);
    }
  } else {
    // ---------------------------------------------------------------- epilogue
    const int q = warp & 3;            // TMEM lane quarter this warp may access
    const int half = (warp - 2) >> 2;  // takes the 32-column chunks of this parity
    float best[BN / 64];               // this lane's column of each chunk: running maximum
    int bi[BN / 64];
#pragma unroll
    for (int j = 0; j < BN / 64; ++j) {
      best[j] = -INFINITY;
      bi[j] = -1;
    }
    bool ok = true;
    for (int t = 0; t < ntl; ++t) {
      const int a = t & 1;
      ok = wait_bounded(bar(B_ACCFULL + a), (t >> 1) & 1, abort_flag, A.err, true);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      const int v0 = (2 * (t_lo + t) + rank) * BV + q * 32;  // id of the warp's first lane
      const bool full = v0 + 32 <= A.V;
#pragma unroll
      for (int j = 0; j < BN / 64; ++j) {
        const int c = 2 * j + half;
        if (c * 32 < A.nt) {
          uint32_t r[32];
          tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + a * BN + c * 32, r);
          tmem_wait_ld();
          if (!full) {  // the vocabulary ends inside the warp's ids
#pragma unroll
            for (int i = 0; i < 32; ++i)
              if (v0 + lane >= A.V) r[i] = 0xff800000u;  // -inf
          }
          float mx = -INFINITY;  // this lane's column: its maximum and the lanes that hold it
          uint32_t who = 0u;
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            const float x = __uint_as_float(r[i]);
            const float m = warp_max(x);
            const uint32_t eq = __ballot_sync(0xffffffffu, x == m);
            if (lane == i) {
              mx = m;
              who = eq;
            }
          }
          if (mx > best[j]) {  // (a NaN or -inf never is)
            best[j] = mx;
            bi[j] = v0 + __ffs(who) - 1;
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) arrive_cluster(in_first_cta(bar(B_ACCEMPTY + a)));
    }
    if (A.expire_rank == rank)
      ok = __all_sync(0xffffffffu, wait_bounded(bar(B_NEVER), 0, abort_flag, A.err, true, A.expire_limit));
    // the pair's maxima meet in the first CTA's ring, which nothing writes or
    // reads any more once the last accumulator is complete: [8 quarters][256]
    // maxima, then ids
    if (ok) {
      const uint32_t base = in_first_cta(sb + kOffRing) + (rank * 4 + q) * BN * 4;
#pragma unroll
      for (int j = 0; j < BN / 64; ++j) {
        const int c = 2 * j + half;
        if (c * 32 < A.nt) {
          st_cluster(base + (c * 32 + lane) * 4, __float_as_uint(best[j]));
          st_cluster(base + 8 * BN * 4 + (c * 32 + lane) * 4, (uint32_t)bi[j]);
        }
      }
    } else if (lane == 0) {
      // the pair gives up together: with a wait run out in either CTA (whatever its
      // role, that CTA's epilogue stops) the ring need not hold maxima, and the
      // range reports none, so that no stale word becomes a token
      st_cluster(in_first_cta(sb + kOffAbort), 1u);
    }
  }

  __syncwarp();
  tc_fence_before();
  __syncthreads();
  cluster_sync();
  if (rank == 0 && (int)threadIdx.x < A.nt && n0 + (int)threadIdx.x < A.M) {
    const bool whole = !*abort_flag;
    const float* vals = reinterpret_cast<const float*>(smem + kOffRing) + threadIdx.x;
    const int* ids = reinterpret_cast<const int*>(vals) + 8 * BN;
    float best = -INFINITY;
    int b = -1;
#pragma unroll
    for (int p = 0; p < 8; ++p) {
      const float v = vals[p * BN];
      const int i = ids[p * BN];
      if (whole && i >= 0 && (v > best || (v == best && i < b))) {
        best = v;
        b = i;
      }
    }
    A.part_val[(int64_t)g * A.M + n0 + threadIdx.x] = best;
    A.part_idx[(int64_t)g * A.M + n0 + threadIdx.x] = b;
  }
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}

// The first maximum over the vocab ranges, a warp per row.
__global__ void __launch_bounds__(256)
lm_head_reduce_kernel(const float* __restrict__ part_val, const int32_t* __restrict__ part_idx, int groups, int M,
                      int32_t* __restrict__ out, const int32_t* __restrict__ out_index) {
  pdl_begin();
  const int r = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (r >= M) return;
  float best = -INFINITY;
  int b = INT_MAX;
  for (int g = lane; g < groups; g += 32) {
    const int i = part_idx[(int64_t)g * M + r];  // -1: no logit of the range was above -inf
    const float v = part_val[(int64_t)g * M + r];
    if (i >= 0 && v > best) {  // ranges come in id order
      best = v;
      b = i;
    }
  }
  const float m = warp_max(best);
  const int id = __reduce_min_sync(0xffffffffu, best == m ? b : INT_MAX);
  if (lane == 0) out[out_index ? out_index[r] : r] = id == INT_MAX ? 0 : id;
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::atomic<bool> tried{false};
  if (!fn && !tried.exchange(true)) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}

// [rows][d] bf16, K-major: boxes of 64 (K) x box_rows, 128-byte swizzle.
bool make_rows_map(CUtensorMap* m, const void* base, uint64_t rows, int d, int box_rows) {
  auto fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {(cuuint64_t)d, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)d * 2};
  cuuint32_t box[2] = {BK, (cuuint32_t)box_rows};
  cuuint32_t es[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

// Tiles of up to 256 hidden rows, a multiple of 32; the pairs left over by the
// tiles split the vocabulary.  Of the tile counts at and just above the fewest,
// the one with the least work on the busiest pair is taken, counted as its
// vocab tiles x (columns + 100): measured at 817 rows, a vocab tile of 64 K
// slices takes 19.7 / 17.6 / 15.0 / 14.0 / 13.2 us with 224 / 192 / 160 / 128 /
// 96 columns, since below about 150 columns a slice costs what its barriers
// and issue cost.  (1400 x 151936: 6 tiles of 256 1111 us, 10 of 160 1172; 257 x
// 100001 x 2048: 2 of 160 90 us, 3 of 96 139.)
LmPlan plan_lm_head(int rows, int vocab) {
  LmPlan p;
  p.v_tiles = (vocab + 2 * BV - 1) / (2 * BV);
  const int pairs = std::max(1, num_sms() / 2);
  const int fewest = std::max(1, (rows + BN - 1) / BN);
  double least = 0;
  for (int n = fewest; n < fewest + 8; ++n) {
    const int nt = ((rows + n - 1) / n + 31) / 32 * 32;
    const int tiles = std::max(1, (rows + nt - 1) / nt);
    const int groups = std::min(std::max(1, pairs / tiles), p.v_tiles);
    const int waves = (tiles * groups + pairs - 1) / pairs;
    const double cost = (double)waves * ((p.v_tiles + groups - 1) / groups) * (std::max(nt, 128) + 100);
    if (n == fewest || cost < least) {
      least = cost;
      p.nt = std::max(32, nt);
      p.n_tiles = tiles;
      p.groups = groups;
    }
  }
  p.ws_bytes = ((size_t)p.groups * rows * (sizeof(float) + sizeof(int32_t)) + 255) / 256 * 256;
  return p;
}

cudaError_t launch_lm_head_argmax(const LmPlan& p, const uint16_t* hidden, const uint16_t* w_lm, int rows, int d,
                                  int vocab, int32_t* out, const int32_t* out_index, void* workspace, int* err,
                                  cudaStream_t s, int expire_rank, long long expire_limit) {
  if (rows == 0) return cudaSuccess;
  static std::atomic<uint64_t> attr_done{0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const uint64_t bit = 1ull << (dev & 63);
  if (!(attr_done.load() & bit)) {
    e = cudaFuncSetAttribute(lm_head_argmax_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax + 1024);
    if (e != cudaSuccess) return e;
    attr_done.fetch_or(bit);
  }
  CUtensorMap mh, mw;
  if (!make_rows_map(&mh, hidden, (uint64_t)rows, d, p.nt / 2) || !make_rows_map(&mw, w_lm, (uint64_t)vocab, d, BV))
    return cudaErrorInvalidValue;
  LmArgs a;
  a.M = rows;
  a.d = d;
  a.V = vocab;
  a.nt = p.nt;
  a.n_tiles = p.n_tiles;
  a.groups = p.groups;
  a.v_tiles = p.v_tiles;
  a.stages = stages_of(p.nt);
  a.part_val = static_cast<float*>(workspace);
  a.part_idx = reinterpret_cast<int32_t*>(static_cast<char*>(workspace) + (size_t)p.groups * rows * sizeof(float));
  a.err = err;
  a.expire_rank = expire_rank;
  a.expire_limit = expire_limit;
  e = launch_pdl(lm_head_argmax_kernel, dim3(2 * p.n_tiles * p.groups), dim3(kThreads),
                 1024 + kOffRing + a.stages * stage_bytes(p.nt), s, mh, mw, a);
  if (e != cudaSuccess) return e;
  e = launch_pdl(lm_head_reduce_kernel, dim3((rows + 7) / 8), dim3(256), 0, s, a.part_val, a.part_idx, p.groups,
                 rows, out, out_index);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace cure
