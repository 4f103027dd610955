// Stage 1 (Sec. 3.3, Eq. 2) and the target argmax of stage 5 (Sec. 3.5, greedy
// decoding): one streaming pass over bf16 vocabulary rows.
//
// A row is scanned by one CTA, or split over a thread-block cluster of S CTAs
// when there are too few rows to fill the GPU.  Top-k lists are ordered by
// (value desc, id asc); stage 1 also keeps a base-2 log-sum-exp (lazily raised
// base + sum).  No global scratch is used.  Two ways to feed the lanes:
//  - register streaming (stage 1): every thread loads 16-byte vectors (8 bf16
//    logits) with non-allocating loads, the next vectors loaded while the
//    current ones are consumed; the log-sum-exp work per logit wants the many
//    resident warps this allows;
//  - a ring (the target argmax): a producer warp streams the CTA's part of
//    the row into three 8 KiB shared-memory stages with bulk copies
//    (cp.async.bulk, completing on an mbarrier per stage), so the bytes in
//    flight do not depend on registers; four consumer warps read their
//    vectors from it and free each stage once they hold them.  Ring waits
//    are bounded: on expiry a CTA flags CURE_DEVERR_TIMEOUT, lets its copies
//    land and still takes part in the merge.
#include <cooperative_groups.h>
#include <float.h>
#include <limits.h>

#include <type_traits>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace cg = cooperative_groups;

namespace cure {
namespace {

constexpr int kThreads = 128;              // consumer threads (4 warps)
constexpr int kWarps = kThreads / 32;
constexpr int kCtaThreads = kThreads + 32; // plus one producer warp
constexpr int kUnroll = 2;                 // vectors per consumer lane per step (ring-fed scan)
constexpr int kChunkVec = 512;             // 16-byte vectors per ring stage (8 KiB)
constexpr int kStages = 3;
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

using tc::smem_u32;
using tc::wait_bounded;

// One bulk copy of `bytes` (a multiple of 16) from global memory into this
// CTA's shared memory, completing on `bar`.
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
      "l"(src), "r"(bytes), "r"(bar)
      : "memory");
}
__device__ __forceinline__ uint4 ld_shared_v4(uint32_t a) {
  uint4 r;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "r"(a));
  return r;
}

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ uint4 ld_stream(const uint4* p) {
  uint4 r;
  asm volatile("ld.global.nc.L1::no_allocate.L2::256B.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
               : "l"(p));
  return r;
}

__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

__device__ __forceinline__ bool better(float a, int ia, float b, int ib) {
  return a > b || (a == b && ia < ib);
}

template <int KT>
struct TopK {
  float v[KT];
  int i[KT];
  __device__ __forceinline__ void init() {
#pragma unroll
    for (int k = 0; k < KT; ++k) {
      v[k] = -INFINITY;
      i[k] = INT_MAX;
    }
  }
  __device__ __forceinline__ void insert(float x, int ix) {
    if (!better(x, ix, v[KT - 1], i[KT - 1])) return;
    bool placed = false;
#pragma unroll
    for (int k = KT - 1; k > 0; --k) {
      const bool up = better(x, ix, v[k - 1], i[k - 1]);
      if (!placed) {
        if (up) {
          v[k] = v[k - 1];
          i[k] = i[k - 1];
        } else {
          v[k] = x;
          i[k] = ix;
          placed = true;
        }
      }
    }
    if (!placed) {
      v[0] = x;
      i[0] = ix;
    }
  }
  __device__ __forceinline__ void merge_shfl(int offset) {
    float pv[KT];
    int pi[KT];
#pragma unroll
    for (int k = 0; k < KT; ++k) {
      pv[k] = __shfl_xor_sync(0xffffffffu, v[k], offset);
      pi[k] = __shfl_xor_sync(0xffffffffu, i[k], offset);
    }
#pragma unroll
    for (int k = 0; k < KT; ++k) insert(pv[k], pi[k]);
  }
};

// Base-2 log-sum-exp state: sum of 2^(x*log2e - mb).
struct Lse2 {
  float mb;  // base: the running max * log2e, as used in the exponents
  float s;
};

__device__ __forceinline__ void lse_merge(Lse2& a, float mb2, float s2) {
  const float m = fmaxf(a.mb, mb2);
  if (m == -INFINITY) return;
  a.s = a.s * ex2(a.mb - m) + s2 * ex2(mb2 - m);
  a.mb = m;
}

__device__ __forceinline__ float max3f(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// Pairs of floats in one 64-bit register pair, for the packed f32x2
// arithmetic of sm_100 and later (two lanes of work per instruction).
__device__ __forceinline__ uint64_t f2_pack(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void f2_unpack(uint64_t r, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r));
}
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t f2_add(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t f2_mul(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, off));
  return v;
}

// Order-preserving unsigned keys of floats (both zeros map to one key), for
// warp maxima by one redux instruction instead of five shuffles.  Key 0 lies
// below every value's, and stands for a NaN too.
__device__ __forceinline__ uint32_t order_key(float x) {
  const uint32_t b = __float_as_uint(x + 0.f);
  if (x != x) return 0u;
  return b ^ ((uint32_t)((int32_t)b >> 31) | 0x80000000u);
}
__device__ __forceinline__ float key_value(uint32_t k) {
  if (k < 0x007fffffu) return -INFINITY;  // keys below every value's
  return __uint_as_float(k ^ ((k >> 31) ? 0x80000000u : 0xffffffffu));
}
__device__ __forceinline__ float warp_max_key(float v) {
  return key_value(__reduce_max_sync(0xffffffffu, order_key(v)));
}

// A lower bound on the warp's k-th best value, the same in every lane: the
// largest lane-local k-th best (that lane holds k values at or above it) and
// the k-th largest of the lane maxima (k lanes each hold one value at or
// above it; a lane that ties the current maximum drops out with it, which can
// only lower the bound).
template <int KT>
__device__ __forceinline__ uint32_t warp_kth_key(const TopK<KT>& tk) {
  uint32_t t = __reduce_max_sync(0xffffffffu, order_key(tk.v[KT - 1]));
  uint32_t m = order_key(tk.v[0]);
#pragma unroll
  for (int k = 0; k < KT; ++k) {
    const uint32_t mk = __reduce_max_sync(0xffffffffu, m);
    if (k == KT - 1) t = max(t, mk);
    if (m == mk) m = 0u;
  }
  return t;
}
// A warp's top-k list, the same in every lane: values (as order keys, 0 =
// empty) and ids, best first.
template <int KT>
struct WarpTop {
  uint32_t key[KT];
  int id[KT];
};

// The warp's list from the lanes' sorted lists: round k takes the best head
// (largest value, lowest id on ties), and the lane that held it moves on.
template <int KT>
__device__ __forceinline__ void warp_merge(TopK<KT>& tk, WarpTop<KT>& out) {
#pragma unroll
  for (int k = 0; k < KT; ++k) {
    const uint32_t x = tk.i[0] == INT_MAX ? 0u : order_key(tk.v[0]);
    out.key[k] = __reduce_max_sync(0xffffffffu, x);
    out.id[k] = __reduce_min_sync(0xffffffffu, x == out.key[k] ? tk.i[0] : INT_MAX);
    if (x == out.key[k] && tk.i[0] == out.id[k]) {
#pragma unroll
      for (int q = 0; q + 1 < KT; ++q) {
        tk.v[q] = tk.v[q + 1];
        tk.i[q] = tk.i[q + 1];
      }
      tk.v[KT - 1] = -INFINITY;
      tk.i[KT - 1] = INT_MAX;
    }
  }
}

// The log-sum-exp of the warp's lanes, in every lane.
__device__ __forceinline__ void warp_lse(Lse2& ls) {
  const float m = warp_max_key(ls.mb);
  float sum = m == -INFINITY ? 0.f : ls.s * ex2(ls.mb - m);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
  ls.mb = m;
  ls.s = sum;
}

__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// The target argmax (ring-fed: its light work per logit leaves the loads in
// flight as the limit).  grid (S, rows) with cluster (S, 1, 1).  Rows are
// (b, j) of a [batch][n_max] tree and only j < n_nodes[b] are scanned.
__global__ void __launch_bounds__(kCtaThreads, 6)
vocab_ring_kernel(const uint16_t* __restrict__ logits, int vocab, int n_max, const int32_t* __restrict__ n_nodes,
                  int32_t* __restrict__ targ, int* err) {
  pdl_begin();  // (accept_walk_kernel counts on the wait in here coming before the trigger)
  const int64_t row = blockIdx.y;
  const int S = gridDim.x;
  const int c = blockIdx.x;  // rank within the cluster
  const int tid = threadIdx.x;
  const int b = (int)(row / n_max);
  const int j = (int)(row % n_max);
  if (j >= n_nodes[b]) {  // uniform over the cluster: every CTA leaves
    if (c == 0 && tid == 0) targ[row] = -1;
    return;
  }

  const uint16_t* rowp = logits + row * (int64_t)vocab;
  const int mis = (int)((reinterpret_cast<uintptr_t>(rowp) >> 1) & 7);
  const int a0 = min((8 - mis) & 7, vocab);
  const int nvec = (vocab - a0) >> 3;
  const int tail0 = a0 + (nvec << 3);
  const int per = (nvec + S - 1) / S;
  const int vb = c * per;
  const int ve = min(nvec, vb + per);

  TopK<1> tk;
  tk.init();
  if (c == 0 && tid < a0) tk.insert(bf16_lo(rowp[tid]), tid);
  if (c == S - 1 && tid < vocab - tail0) tk.insert(bf16_lo(rowp[tail0 + tid]), tail0 + tid);

  const uint4* vp = reinterpret_cast<const uint4*>(rowp + a0);  // 16-byte aligned
  // The CTA's vectors [vb, ve) stream through a ring of kStages shared-memory
  // stages of kChunkVec vectors, filled by bulk copies that the producer warp
  // issues (bytes in flight do not depend on registers); each consumer warp
  // frees a stage once it has its vectors in registers.
  __shared__ __align__(128) uint4 ring[kStages][kChunkVec];
  __shared__ __align__(8) uint64_t full_bar[kStages], empty_bar[kStages];
  __shared__ int abort_s;
  volatile int* abort_flag = &abort_s;
  const int lane = tid & 31, warp = tid >> 5;
  const int nloc = max(0, ve - vb);
  const int nchunks = (nloc + kChunkVec - 1) / kChunkVec;
  if (tid == 0) {
    for (int st = 0; st < kStages; ++st) {
      tc::mbar_init(smem_u32(&full_bar[st]), 1);
      tc::mbar_init(smem_u32(&empty_bar[st]), kWarps);
    }
    abort_s = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();

  // thr: the warp's maximum so far.  A logit below it cannot be the row's
  // argmax, so the lanes' best change only in the rare steps with a logit at
  // or above it, after which thr is recomputed (the trip count is uniform over
  // the warp, and all lanes take part).
  float thr = warp_max(tk.v[0]);
  // One step: kUnroll vectors per lane, r[u] at vector index gi[u] (vb-based);
  // FULL when every lane's vectors are in range, so that no check is needed.
  auto step = [&](const uint4 (&r)[kUnroll], const int (&gi)[kUnroll], bool first, auto full_tag) {
    constexpr bool FULL = decltype(full_tag)::value;
    float lo[kUnroll][4], hi[kUnroll][4];
    float gmv[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      const uint32_t w[4] = {r[u].x, r[u].y, r[u].z, r[u].w};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        lo[u][q] = bf16_lo(w[q]);
        hi[u][q] = bf16_hi(w[q]);
      }
      const float g = fmaxf(max3f(lo[u][0], hi[u][0], lo[u][1]),
                            max3f(max3f(hi[u][1], lo[u][2], hi[u][2]), lo[u][3], hi[u][3]));
      gmv[u] = (FULL || gi[u] < nloc) ? g : -INFINITY;
    }
    // a warp does not start by inserting every logit it sees
    if (first) thr = fmaxf(thr, warp_max(fmaxf(gmv[0], gmv[1])));
    bool cand = false;
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) cand |= (FULL || gi[u] < nloc) && gmv[u] >= thr;
    if (__any_sync(0xffffffffu, cand)) {
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) {
        if ((FULL || gi[u] < nloc) && gmv[u] >= thr) {
          const int idx = a0 + ((vb + gi[u]) << 3);
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            if (lo[u][q] >= thr) tk.insert(lo[u][q], idx + 2 * q);
            if (hi[u][q] >= thr) tk.insert(hi[u][q], idx + 2 * q + 1);
          }
        }
      }
      thr = warp_max(tk.v[0]);
    }
  };

  if (warp == kWarps) {
    // ---------------------------------------------------------------- producer
    if (lane == 0) {
      int issued = 0;
      for (int ch = 0; ch < nchunks; ++ch, ++issued) {
        const int st = ch % kStages;
        if (ch >= kStages &&
            !wait_bounded(smem_u32(&empty_bar[st]), ((ch / kStages) & 1) ^ 1, abort_flag, err, true))
          break;
        const uint32_t bytes = (uint32_t)min(kChunkVec, nloc - ch * kChunkVec) * 16u;
        tc::mbar_arrive_expect_tx(smem_u32(&full_bar[st]), bytes);
        bulk_load(smem_u32(&ring[st][0]), vp + vb + ch * kChunkVec, bytes, smem_u32(&full_bar[st]));
      }
      // the copies in flight land before the CTA's shared memory goes away
      for (int ch = max(0, issued - kStages); ch < issued; ++ch)
        wait_bounded(smem_u32(&full_bar[ch % kStages]), (ch / kStages) & 1, abort_flag, err, false);
    }
  } else {
    // ---------------------------------------------------------------- consumers
    bool first = true;
    for (int ch = 0; ch < nchunks; ++ch) {
      const int st = ch % kStages;
      const bool ok = wait_bounded(smem_u32(&full_bar[st]), (ch / kStages) & 1, abort_flag, err, true);
      if (!__all_sync(0xffffffffu, ok)) break;
      const int cb = ch * kChunkVec;              // chunk's first vector (vb-based)
      const bool full = cb + kChunkVec <= nloc;
      // the warp's two steps of this chunk: vectors warp*32 + lane + u*128,
      // u = 0..3; the stage is freed once the second step's vectors are read
      uint4 r[kUnroll];
      int gi[kUnroll];
      constexpr int kSteps = kChunkVec / (kThreads * kUnroll);  // steps per chunk
#pragma unroll
      for (int half = 0; half < kSteps; ++half) {
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
          const int o = warp * 32 + lane + (half * kUnroll + u) * (kThreads);
          gi[u] = cb + o;
          if (full || gi[u] < nloc) r[u] = ld_shared_v4(smem_u32(&ring[st][o]));
        }
        if (half == kSteps - 1) {
          __syncwarp();
          if (lane == 0) tc::mbar_arrive(smem_u32(&empty_bar[st]));  // this warp's vectors are in registers
        }
        if (full) step(r, gi, first && half == 0, std::integral_constant<bool, true>());
        else step(r, gi, first && half == 0, std::integral_constant<bool, false>());
      }
      first = false;
    }
  }

  // ---- warp, CTA and (rank 0 reading its peers' results) cluster merge
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) tk.merge_shfl(off);
  __shared__ float warp_v[kWarps], cta_v;
  __shared__ int warp_i[kWarps], cta_i;
  if (lane == 0 && warp < kWarps) {
    warp_v[warp] = tk.v[0];
    warp_i[warp] = tk.i[0];
  }
  __syncthreads();
  if (tid == 0) {
#pragma unroll
    for (int w = 1; w < kWarps; ++w) tk.insert(warp_v[w], warp_i[w]);
    cta_v = tk.v[0];
    cta_i = tk.i[0];
  }
  if (S > 1) {
    cg::cluster_group cluster = cg::this_cluster();
    cluster.sync();
    if (c == 0 && tid == 0) {
      for (int r = 1; r < S; ++r) tk.insert(*cluster.map_shared_rank(&cta_v, r), *cluster.map_shared_rank(&cta_i, r));
    }
    cluster.sync();
  }
  if (c == 0 && tid == 0) targ[row] = tk.i[0];
}

// Register-streaming variant (used for stage 1, whose log-sum-exp work per
// logit wants many resident warps): every thread streams 16-byte vectors with
// non-allocating loads, the next vectors loaded while the current ones are
// consumed.  grid (S, rows) with cluster (S, 1, 1), T threads per CTA.
//
// What bounds it: at 512 rows x 151936 the stream (30.4 us graph-replayed,
// 5.1 TB/s; 22.9 us at the copy rate); with few rows the latency of a warp's
// chain of steps and of the merge.  So the rare part of a step and the merge
// are kept short: warp maxima are one redux instruction on order keys instead
// of five shuffles; a warp's threshold is shared with the CTA's other warps,
// so that fewer logits enter a list; every warp writes its result straight
// into rank 0's shared memory, one cluster barrier follows, and one warp
// merges all parts at once (before: a merge per CTA, two barriers, and a
// serial walk over the peers' shared memory by one thread).  Each lane keeps its
// own list, so that several logits enter at once.  Up to top-4 the 24 inserts of
// a step are unrolled; above, a lane loops over a mask of its candidates, since
// 24 unrolled inserts of an 8-deep list do not fit the instruction cache (top-6
// of 512 x 151936: 44.8 us; unrolled 133; one list per warp, entered one logit
// at a time, 65).
// Before these changes and the launch shapes of pick_scan: 512 x 151936 top-3
// 36.7 us, top-6 306 us (now 44.8), 16 x 128256 12.0 us, 128 x 151936 33.6 us (now 14).
//
// Vectors per lane per step: three 16-byte loads in flight per lane (70
// registers up to top-3, still one wave of the grid).
constexpr int kUnrollS = 3;
constexpr int kMaxSplit = 8;  // portable cluster size

template <int KT>
struct ScanPart {
  uint32_t key[KT];
  int id[KT];
  float mb, s;
};

// One of the few ids at the row's ends, outside its whole vectors (a NaN there is
// passed over).
__device__ __forceinline__ void lse_add(Lse2& ls, float x) {
  lse_merge(ls, fmaxf(x, -INFINITY) * kLog2e, 1.f);  // (a NaN as -inf)
}

template <int KT, int T>
__global__ void __launch_bounds__(T)
vocab_scan_kernel(const uint16_t* __restrict__ logits, int vocab, int k_out,
                  int32_t* __restrict__ top_ids, float* __restrict__ top_vals, float* __restrict__ margin,
                  float* __restrict__ logp1) {
  constexpr int W = T / 32;
  __shared__ ScanPart<KT> part[kMaxSplit * W];  // rank 0's holds every warp of the cluster
  __shared__ uint32_t thr_s;  // the largest k-th best of the CTA's warps, as an order key
  const int64_t row = blockIdx.y;
  const int S = gridDim.x;
  const int c = blockIdx.x;  // rank within the cluster
  const int tid = threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5;
  if (tid == 0) thr_s = 0u;
  __syncthreads();
  // every CTA of the cluster has started once this barrier completes (waited
  // for before the first write to rank 0's shared memory)
  if (S > 1) cluster_arrive();
  pdl_begin();

  const uint16_t* rowp = logits + row * (int64_t)vocab;
  const int mis = (int)((reinterpret_cast<uintptr_t>(rowp) >> 1) & 7);
  const int a0 = min((8 - mis) & 7, vocab);
  const int nvec = (vocab - a0) >> 3;
  const int tail0 = a0 + (nvec << 3);
  const int per = (nvec + S - 1) / S;
  const int vb = c * per;
  const int ve = min(nvec, vb + per);

  const uint4* vp = reinterpret_cast<const uint4*>(rowp + a0);
  const int wb0 = vb + (tid & ~31);
  uint4 r[kUnrollS];
#pragma unroll
  for (int u = 0; u < kUnrollS; ++u) {
    const int vi = wb0 + lane + u * T;
    if (vi < ve) r[u] = ld_stream(vp + vi);
  }

  TopK<KT> ll;
  ll.init();
  Lse2 ls{-INFINITY, 0.f};
  if (c == 0 && warp == 0 && a0 > 0) {  // the ids before the first 16-byte boundary
    const float x = lane < a0 ? bf16_lo(rowp[lane]) : 0.f;
    if (lane < a0) lse_add(ls, x);
    if (lane < a0) ll.insert(x, lane);
  }

  // The trip count is uniform over the warp: the threshold and the log-sum-exp
  // base are warp-wide values that all lanes take part in.
  //  - tkey: the order key of a lower bound on the row's k-th best: the largest
  //    bound of the CTA's warps so far (a warp publishes its own when its lists
  //    change, and reads the CTA's best once a step).  A logit below it cannot
  //    be in the row's top k, so lists change only in rare steps.
  //  - mbw: base-2 exponent base of the lane sums (sum of 2^(x log2e - mbw));
  //    raised, with the sums rescaled, only when some lane sees a logit more
  //    than 2^8 above it, so the sums stay below 2^8 per term and the rescale
  //    is rare and uniform.
  uint32_t tkey = 0u;
  float mbw = -INFINITY;
  uint64_t sacc = f2_pack(0.f, 0.f);  // two lane sums, as one f32x2 pair
  // one step: kUnrollS vectors per lane; FULL when every lane's vectors are in
  // range (all but a warp's last step), so that no per-vector check is needed
  auto step = [&](int wb, auto full_tag) {
    constexpr bool FULL = decltype(full_tag)::value;
    uint4 nx[kUnrollS];
#pragma unroll
    for (int u = 0; u < kUnrollS; ++u) {
      const int vi = wb + lane + (kUnrollS + u) * T;
      if (vi < ve) nx[u] = ld_stream(vp + vi);
    }
    uint64_t xp[kUnrollS][4];  // (lo, hi) logit pairs of each 32-bit word
    float gmv[kUnrollS];
#pragma unroll
    for (int u = 0; u < kUnrollS; ++u) {
      const uint32_t w[4] = {r[u].x, r[u].y, r[u].z, r[u].w};
      float lo[4], hi[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        lo[q] = bf16_lo(w[q]);
        hi[q] = bf16_hi(w[q]);
        xp[u][q] = f2_pack(lo[q], hi[q]);
      }
      const float g = fmaxf(max3f(lo[0], hi[0], lo[1]), max3f(max3f(hi[1], lo[2], hi[2]), lo[3], hi[3]));
      gmv[u] = (FULL || wb + lane + u * T < ve) ? g : -INFINITY;
    }
    float gl = gmv[0];
#pragma unroll
    for (int u = 1; u < kUnrollS; ++u) gl = fmaxf(gl, gmv[u]);
    if (__any_sync(0xffffffffu, gl * kLog2e > mbw + 8.f)) {
      const float nb = warp_max_key(gl) * kLog2e;
      if (mbw != -INFINITY) {
        const float sc = ex2(mbw - nb);
        sacc = f2_mul(sacc, f2_pack(sc, sc));
      }
      mbw = nb;
    }
    if (mbw != -INFINITY) {
      const uint64_t l2 = f2_pack(kLog2e, kLog2e), nb2 = f2_pack(-mbw, -mbw);
#pragma unroll
      for (int u = 0; u < kUnrollS; ++u) {
        if (FULL || wb + lane + u * T < ve) {
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            float a, b;
            f2_unpack(f2_fma(xp[u][q], l2, nb2), a, b);
            sacc = f2_add(sacc, f2_pack(ex2(a), ex2(b)));
          }
        }
      }
    }
    tkey = max(tkey, *reinterpret_cast<volatile uint32_t*>(&thr_s));
    if (wb == wb0) {
      // first step: the k-th largest of the lanes' maxima of this step is a
      // valid threshold already, so that a warp does not start by inserting
      // every logit it sees
      float gm = gl;
#pragma unroll
      for (int k = 0; k < KT; ++k) {
        const uint32_t mk = __reduce_max_sync(0xffffffffu, order_key(gm));
        if (k == KT - 1) tkey = max(tkey, mk);
        if (gm == key_value(mk)) gm = -INFINITY;
      }
    }
    const float thr = key_value(tkey);
    if (__any_sync(0xffffffffu, gl >= thr)) {
      if constexpr (KT <= 4) {
#pragma unroll
        for (int u = 0; u < kUnrollS; ++u) {
          if ((FULL || wb + lane + u * T < ve) && gmv[u] >= thr) {
            const int idx = a0 + ((wb + lane + u * T) << 3);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              float a, b;
              f2_unpack(xp[u][q], a, b);
              if (a >= thr) ll.insert(a, idx + 2 * q);
              if (b >= thr) ll.insert(b, idx + 2 * q + 1);
            }
          }
        }
      } else {
        uint32_t cand = 0u;  // this lane's logits at or above it, in id order
#pragma unroll
        for (int u = 0; u < kUnrollS; ++u) {
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            float a, b;
            f2_unpack(xp[u][q], a, b);
            const bool in = FULL || wb + lane + u * T < ve;
            if (in && a >= thr) cand |= 1u << (8 * u + 2 * q);
            if (in && b >= thr) cand |= 2u << (8 * u + 2 * q);
          }
        }
#pragma unroll 1
        while (cand) {
          const int e = __ffs(cand) - 1;
          cand &= cand - 1u;
          uint32_t w = 0u;  // the word of logit e (masks, not an indexed array)
#pragma unroll
          for (int u = 0; u < kUnrollS; ++u) {
            const uint32_t wu[4] = {r[u].x, r[u].y, r[u].z, r[u].w};
#pragma unroll
            for (int q = 0; q < 4; ++q) w |= wu[q] & (0u - (uint32_t)((e >> 1) == 4 * u + q));
          }
          ll.insert((e & 1) ? bf16_hi(w) : bf16_lo(w), a0 + ((wb + lane + (e >> 3) * T) << 3) + (e & 7));
        }
        __syncwarp();
      }
      tkey = max(tkey, warp_kth_key(ll));
      if (lane == 0) atomicMax(&thr_s, tkey);
    }
#pragma unroll
    for (int u = 0; u < kUnrollS; ++u) r[u] = nx[u];
  };
  int wb = wb0;
  for (; wb + 31 + (kUnrollS - 1) * T < ve; wb += kUnrollS * T) step(wb, std::integral_constant<bool, true>());
  for (; wb < ve; wb += kUnrollS * T) step(wb, std::integral_constant<bool, false>());
  float sa, sb2;
  f2_unpack(sacc, sa, sb2);
  lse_merge(ls, mbw, sa + sb2);
  if (c == S - 1 && warp == W - 1 && tail0 < vocab) {  // the ids after the last 16-byte boundary
    const int i = tail0 + lane;
    const float x = i < vocab ? bf16_lo(rowp[i]) : 0.f;
    if (i < vocab) lse_add(ls, x);
    if (i < vocab) ll.insert(x, i);
  }
  WarpTop<KT> tk;
  warp_merge(ll, tk);

  // ---- every warp's result goes to rank 0's shared memory
  warp_lse(ls);
  if (S > 1) cluster_wait();  // rank 0 has started
  if (lane == 0) {
    ScanPart<KT>* pp = &part[c * W + warp];
    if (S > 1) pp = cg::this_cluster().map_shared_rank(pp, 0);
#pragma unroll
    for (int k = 0; k < KT; ++k) {
      pp->key[k] = tk.key[k];
      pp->id[k] = tk.id[k];
    }
    pp->mb = ls.mb;
    pp->s = ls.s;
  }
  __syncwarp();
  if (S > 1) {
    cluster_arrive();
    cluster_wait();
  } else {
    __syncthreads();
  }
  if (c != 0 || warp != 0) return;

  // ---- rank 0's first warp merges the S * W parts (the vector ranges of the
  // warps interleave, so equal values of different parts go by id)
  ls.mb = -INFINITY;
  ls.s = 0.f;
  int head[kMaxSplit * W / 32 > 0 ? kMaxSplit * W / 32 : 1];  // next entry of each of this lane's parts
#pragma unroll
  for (int j = 0; j < (int)(sizeof(head) / sizeof(int)); ++j) {
    head[j] = 0;
    const int p = lane + 32 * j;
    if (p < S * W) lse_merge(ls, part[p].mb, part[p].s);
  }
  float v0 = 0.f, v1 = 0.f;
  for (int k = 0; k < k_out; ++k) {
    uint32_t x = 0u;
    int ix = INT_MAX, from = -1;
#pragma unroll
    for (int j = 0; j < (int)(sizeof(head) / sizeof(int)); ++j) {
      const int p = lane + 32 * j;
      if (p < S * W && head[j] < KT) {
        const uint32_t y = part[p].key[head[j]];
        const int iy = part[p].id[head[j]];
        if (y > x || (y == x && iy < ix)) {
          x = y;
          ix = iy;
          from = j;
        }
      }
    }
    const uint32_t best = __reduce_max_sync(0xffffffffu, x);
    const int id = __reduce_min_sync(0xffffffffu, x == best ? ix : INT_MAX);
#pragma unroll
    for (int j = 0; j < (int)(sizeof(head) / sizeof(int)); ++j)
      if (from == j && x == best && ix == id) ++head[j];
    float v = key_value(best);
    if (v == 0.f) v = bf16_lo(rowp[id]);  // the key does not hold a zero's sign
    if (k == 0) v0 = v;
    if (k == 1) v1 = v;
    if (lane == 0) {
      top_ids[row * k_out + k] = id;
      top_vals[row * k_out + k] = v;
    }
  }
  warp_lse(ls);
  if (lane == 0) {
    if (margin) margin[row] = v0 - v1;
    // log p = (v0 log2(e) - mb - log2(s)) ln 2: the difference of the two large
    // exponents is taken first, in one rounding
    if (logp1) logp1[row] = (fmaf(v0, kLog2e, -ls.mb) - log2f(ls.s)) * kLn2;
  }
}

// Launch shape of the register-streaming scan: as many warps per row as fit one
// wave of the grid (at 70-80 registers an SM holds 28 warps as 4-warp CTAs and
// 24 as 8-warp ones), a power of two from 4 to 64, since a row's warps stream
// its parts side by side: with few rows the bytes in flight are what is short.
// 8-warp CTAs keep the cluster (<= 8 CTAs) within the portable size from 32
// warps a row on.  Graph-replayed, us per call, against the rule of at most
// 8 x 4 warps a row that this one replaced (same kernel, top-3):
//   16 x 128256   8 CTAs x 8 warps  5.3     (8 x 4: 6.2)
//   64 x 152000   4 x 8            10.8     (8 x 4: 12.2; 8 x 8, two waves: 13.8)
//   256 x 151937  4 x 4            18.2     (2 x 8: 26.6; 2 x 4: 22.2)
//   512 x 151936  2 x 4            30.4     (4 x 4: 34.0; 1 x 4: 37.8)
//   1024 x 128256 1 x 4            43.2     (2 x 4: 47.7; 1 x 8: 46.0)
// Each CTA keeps at least one vector per thread.
struct ScanShape {
  int split, threads;
};
ScanShape pick_scan(int64_t rows, int vocab) {
  const int nvec = vocab / 8;
  const int64_t slots256 = 24LL * num_sms(), slots128 = 28LL * num_sms();  // warps in one wave
  int t = 128, warps = 4;
  if (rows * 32 <= slots256) {
    t = 256;
    warps = rows * 64 <= slots256 ? 64 : 32;
  } else if (rows * 16 <= slots128) {
    warps = 16;
  } else if (rows * 8 <= slots128) {
    warps = 8;
  }
  int s = warps * 32 / t;
  while (s > 1 && nvec / s < t) --s;
  return {s, t};
}

// The grid is kept to one wave of at most six CTAs per SM (the occupancy the
// kernel is built for): one CTA per row when the rows alone reach that,
// else rows split over a cluster of up to 8 CTAs, each keeping at least two
// vectors per consumer thread.  Bytes in flight come from each CTA's ring, so
// a CTA that streams a whole row keeps the SM as busy as several would.
int pick_split_ring(int64_t rows, int vocab, int per_sm) {
  const int nvec = vocab / 8;
  const int64_t slots = (int64_t)per_sm * num_sms();
  if (rows >= slots) return 1;
  int s = (int)(slots / rows);
  s = max(1, min(s, 8));
  while (s > 1 && nvec / s < 2 * kThreads) --s;
  return s;
}

// Launch attributes shared by both scans: a cluster of S CTAs per row, and a
// programmatic dependent launch (see pdl_begin()).
struct ScanLaunch {
  cudaLaunchAttribute attr[2];
  cudaLaunchConfig_t cfg = {};
  ScanLaunch(int S, int64_t rows, int threads, cudaStream_t s) {
    cfg.gridDim = dim3(S, (unsigned)rows, 1);
    cfg.blockDim = dim3(threads, 1, 1);
    cfg.stream = s;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = S;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
  }
};

template <int KT>
cudaError_t launch_scan(const uint16_t* logits, int64_t rows, int vocab, int k_out, int32_t* top_ids,
                        float* top_vals, float* margin, float* logp1, cudaStream_t s) {
  const ScanShape sh = pick_scan(rows, vocab);
  ScanLaunch l(sh.split, rows, sh.threads, s);
  switch (sh.threads) {
    case 256:
      return cudaLaunchKernelEx(&l.cfg, vocab_scan_kernel<KT, 256>, logits, vocab, k_out, top_ids, top_vals, margin, logp1);
    default:
      return cudaLaunchKernelEx(&l.cfg, vocab_scan_kernel<KT, 128>, logits, vocab, k_out, top_ids, top_vals, margin, logp1);
  }
}

}  // namespace

cudaError_t launch_score(const uint16_t* logits, int64_t rows, int vocab, int topk,
                         int32_t* top_ids, float* top_vals, float* margin, float* logp1,
                         cudaStream_t s) {
  if (rows == 0) return cudaSuccess;
  switch (topk) {
    case 2: return launch_scan<2>(logits, rows, vocab, topk, top_ids, top_vals, margin, logp1, s);
    case 3: return launch_scan<3>(logits, rows, vocab, topk, top_ids, top_vals, margin, logp1, s);
    case 4: return launch_scan<4>(logits, rows, vocab, topk, top_ids, top_vals, margin, logp1, s);
    case 5:
    case 6: return launch_scan<6>(logits, rows, vocab, topk, top_ids, top_vals, margin, logp1, s);
    default: return launch_scan<8>(logits, rows, vocab, topk, top_ids, top_vals, margin, logp1, s);
  }
}

cudaError_t launch_target_argmax(const uint16_t* logits, int batch, int n_max, int vocab,
                                 const int32_t* n_nodes, int32_t* targ, cudaStream_t s) {
  const int64_t rows = (int64_t)batch * n_max;
  if (rows == 0) return cudaSuccess;
  ScanLaunch l(pick_split_ring(rows, vocab, 6), rows, kCtaThreads, s);
  return cudaLaunchKernelEx(&l.cfg, vocab_ring_kernel, logits, vocab, n_max, n_nodes, targ, device_error_word());
}

}  // namespace cure
