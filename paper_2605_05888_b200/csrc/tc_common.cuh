// PTX wrappers and constants shared by the tcgen05 expert-FFN kernels (one-CTA and CTA-pair forms).
#pragma once
#include <cuda.h>

#include "common.cuh"

namespace moehub {

constexpr int kTcThreads = 192;
constexpr int kStages = 4;
constexpr int kBK = 64;                       // k elements per stage (128 bytes of bf16)
constexpr int kUmmaN = 256;
constexpr int kABytes = kTileRows * kBK * 2;  // 16 KB
constexpr int kBBytes = kUmmaN * kBK * 2;     // 32 KB
constexpr int kStageBytes = kABytes + kBBytes;
constexpr int kTcSmem = kStages * kStageBytes + 1024 /*alignment slack*/ + 512 /*barriers, item ring*/;
constexpr unsigned long long kDefaultWaitNs = 2000000000ull;  // default bound on any single wait: 2 s

// ---- PTX wrappers ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned long long globaltimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_inval(uint32_t bar) { asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(bar) : "memory"); }
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// The hardware suspends the thread until the phase completes or the time hint (nanoseconds) has passed.
constexpr uint32_t kTryHintNs = 20000;
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity), "r"(kTryHintNs) : "memory");
  return ok != 0;
}
// Whether the phase has completed, without waiting.
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
// Bounded wait.  Returns false when the time limit ran out or another role already gave up.
// sleep_ns > 0 backs off between polls: for waits that are long by design (an epilogue warp waiting
// for a whole main loop) polling at full rate only burns power the tensor pipe could use.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                          unsigned long long limit_ns, unsigned sleep_ns = 0) {
  if (mbar_try(bar, parity)) return true;
  const unsigned long long t0 = globaltimer();
  for (unsigned it = 1;; ++it) {
    if (sleep_ns) __nanosleep(sleep_ns);
    if (mbar_try(bar, parity)) return true;
    if ((it & 31u) == 0u) {
      if (*abort_flag) return false;
      if (globaltimer() - t0 > limit_ns) return false;
    }
  }
}
// What a whole warp waited for: every lane looks at the clock for itself, so near the limit some may give up and others not.
// All of them go the way of the one that gave up: what follows (votes, barriers, tensor-memory loads) wants them together.
__device__ __forceinline__ bool warp_agrees(bool ok) { return __all_sync(0xffffffffu, ok); }
// One lane of the warp, the same every time (all 32 call).  The compiler takes what stands behind it as issued once and
// keeps the operands in uniform registers.
__device__ __forceinline__ bool elect_one() {
  uint32_t one;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(one));
  return one != 0;
}
// A value that is the same in all lanes, so that the compiler knows it is (MMA operands live in uniform registers).
template <typename T> __device__ __forceinline__ T uniform(T v) { return __shfl_sync(0xffffffffu, v, 0); }
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1) : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1,
                                            int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2) : "memory");
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, int c2,
                                            int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}
__device__ __forceinline__ void tma_load_4d_hint(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1,
                                                 int c2, int c3, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4, %5, %6}], [%2], %7;"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "l"(policy) : "memory");
}
// The same load with an L2 eviction-priority hint (a policy made by l2_policy_evict_first/_last).
__device__ __forceinline__ void tma_load_3d_hint(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1,
                                                 int c2, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4, %5}], [%2], %6;"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "l"(policy) : "memory");
}
__device__ __forceinline__ uint64_t l2_policy_evict_first() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                       uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void tc_ld16(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// One 32-byte store (a whole L2 sector) per lane.  The epilogues write a row per lane, so a 16-byte
// store covers half a sector and the L2 has to merge the halves; whole sectors need no merge.
__device__ __forceinline__ void st_global_32B(void* p, const uint4& lo, const uint4& hi) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(lo.x), "r"(lo.y), "r"(lo.z),
               "r"(lo.w), "r"(hi.x), "r"(hi.y), "r"(hi.z), "r"(hi.w) : "memory");
}

// silu(g) * u in fp32.  The quotient is the approximate divide (2 ulp, far inside the bf16 rounding that
// follows): the IEEE divide leaves its fast path for NaN, infinite and very large operands, and the
// padding rows of a partly filled tile hold whatever the pool held before, so a single such lane
// sends its whole warp through the slow subroutine (measured: 21 us instead of 2 us per 128 x 128 block
// when three quarters of a tile's rows are padding).
__device__ __forceinline__ float silu_mul(float g, float u) { return __fdividef(g, 1.0f + __expf(-g)) * u; }

// Shared-memory matrix descriptor of a K-major tile whose rows are 128 bytes (64 bf16) in the
// 128-byte swizzle: 8-row groups are 1024 bytes apart.
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr >> 4) & 0x3fff);   // start address, 16-byte units
  d |= (uint64_t)1 << 16;                  // leading byte offset (unused with swizzle, K-major)
  d |= (uint64_t)(1024 >> 4) << 32;        // stride byte offset between 8-row groups
  d |= (uint64_t)1 << 46;                  // descriptor version of this architecture
  d |= (uint64_t)2 << 61;                  // 128-byte swizzle
  return d;
}
// Instruction descriptor: bf16 x bf16 -> fp32, A and B K-major, M = 128, N = 256.
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kUmmaN >> 3) << 17) |
                            ((uint32_t)(kTileRows >> 4) << 24);

// Thin tiles (at most kThinRows rows): the MMA is M = 128 weight rows x N = 16*n16 tile rows.
constexpr int kThinRows = 64;
constexpr int kThinShift = 24;  // an item-ring entry is item | n16 << kThinShift
__host__ __device__ constexpr uint32_t thin_idesc(int n16) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n16 * 16 >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}

// Short last tile of an expert with several tiles: M = 64 MMAs on the tile's first 64 rows.
constexpr int kHalfForm = 8;  // value of the n16 field for this form (thin tiles use 1..4)
constexpr uint32_t kIdescHalf = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kUmmaN >> 3) << 17) | ((uint32_t)(64 >> 4) << 24);

constexpr int kMaxExperts = 256;

struct Item {
  int type;   // 0: GEMM1 (+SwiGLU), 1: GEMM2
  int e, nb, tile;
  int m;      // tiles of expert e
  bool cold;  // item of the weight-streaming-bound run (interleaved work list)
};

// The work list, built by every CTA for itself in shared memory from tile_expert[P] (the same
// deterministic result in every CTA, so no launch and no global round trip is spent on it).
//   tiles[estart[e] .. estart[e+1])  the used tiles of expert e, in ascending tile order;
//   the item sequence is at most 2E segments, segment = all GEMM1 items or all GEMM2 items of one
//   expert: seg_start[i] first item of segment i (seg_start[2E] = number of items), seg_info[i] =
//   expert | type << 16 (type 0: GEMM1, 1: GEMM2); n1 = items before the first GEMM2 item when the
//   two GEMMs are separate launches.
//   With hot_min > 0 (separate launches only) each GEMM's segments are ordered "hot" experts first
//   (at least hot_min tiles: their items are bound by the tensor pipe, the weights come out of L2),
//   then "cold" ones (fewer tiles: bound by streaming the expert's weights from HBM once), both in
//   ascending expert order, and n_hot[g] counts the hot items of GEMM g: the kernel walks the two
//   runs interleaved, so that at any moment some SMs pull weights from HBM while the others run MMAs.
constexpr int kMaxListTiles = 4608;
struct WorkList {
  int estart[kMaxExperts + 1];
  int seg_start[2 * kMaxExperts + 1];
  int seg_info[2 * kMaxExperts];
  int n1;
  int n_hot[2];
  uint16_t tiles[kMaxListTiles];
};
// What only the building needs (it lies in the operand stages, which are not in use yet).
struct WorkScratch {
  int cursor[kMaxExperts];
  int order[kMaxExperts];      // the experts in the order their segments are placed
  int units[kMaxExperts + 1];  // units (tiles, or pairs of them) of the experts placed before position i
  int after[kMaxExperts];      // the position whose GEMM1 segment the GEMM2 segment of position q follows
  int n_hot_experts;
  uint16_t owner[kMaxListTiles];  // tile_expert, 0xffff: unused
};

// All threads of the CTA call this (it synchronises the CTA).  pair = 2 counts one item per PAIR of
// tiles.  fused: the GEMM2 segment of an expert follows the first later GEMM1 segment that ends at least `lag` GEMM1
// items behind its own, as long as `lag` GEMM2 items stay in reserve for the end of the list; otherwise all
// GEMM1 segments come first.
// hist != nullptr: the list is built from the experts' row counts instead of tile_expert - expert e then
// owns the consecutive tiles [estart[e], estart[e + 1]) (the layout of the ordered dispatch), which is known
// before a single row has been dispatched.  hot_first: experts are placed by descending row count (the
// experts whose first tiles fill earliest come first) instead of by index.
// count: [kMaxExperts] rows per expert, filled in when the list is built from them (else -1), or nullptr.
//
// Every step but the scatter of the tiles is a prefix sum or a binary search per expert, because this stands in front
// of every expert launch: a serial walk over the experts with dependent shared-memory reads, and tile owners fetched
// from global memory 32 at a time, took 12-14 us with 60 experts (expert launch of one Qwen-like token 53.7 -> 45.4 us,
// of 512 tokens 190.8 -> 178.7; both launches of the 128-token DeepSeek-like layer 2382 -> 2319).
__device__ __forceinline__ void build_worklist(WorkList& wl, WorkScratch& ws, const int* __restrict__ tile_expert, int P, int E,
                                               int NB1, int NB2, int lag, int fused, int pair, int hot_min = 0,
                                               const int* __restrict__ hist = nullptr, int hot_first = 0, int* count = nullptr) {
  const int tid = threadIdx.x, nthr = blockDim.x, lane = tid % 32;
  constexpr int kPer = kMaxExperts / 32;  // experts per lane in the scans
  constexpr int kAhead = 4;               // tile owners fetched at once
  for (int e = tid; e < kMaxExperts; e += nthr) {
    ws.cursor[e] = (hist != nullptr && e < E) ? (hist[e] + kTileRows - 1) / kTileRows : 0;
    if (count != nullptr) count[e] = (hist != nullptr && e < E) ? hist[e] : -1;
    ws.order[e] = e;
  }
  __syncthreads();
  if (hist == nullptr) {
    for (int p0 = tid; p0 < P; p0 += kAhead * nthr) {
      int e[kAhead];
#pragma unroll
      for (int i = 0; i < kAhead; ++i) e[i] = p0 + i * nthr < P ? tile_expert[p0 + i * nthr] : -1;
#pragma unroll
      for (int i = 0; i < kAhead; ++i) {
        const int p = p0 + i * nthr;
        const bool used = e[i] >= 0 && e[i] < E;
        if (p < P) ws.owner[p] = used ? (uint16_t)e[i] : (uint16_t)0xffff;
        if (used) atomicAdd(&ws.cursor[e[i]], 1);
      }
    }
  } else if (hot_first) {
    // position of expert e = experts with more rows, or as many and a lower index
    for (int e = tid; e < E; e += nthr) {
      const int c = count[e];
      int rank = 0;
      for (int o = 0; o < E; ++o) {
        const int co = count[o];
        rank += (co > c || (co == c && o < e)) ? 1 : 0;
      }
      ws.order[rank] = e;
    }
  }
  __syncthreads();
  if (hot_min > 0 && !fused) {  // order: the hot experts, then the cold ones, each in index order
    if (tid < 32) {
      int hot[kPer], sum = 0;
#pragma unroll
      for (int i = 0; i < kPer; ++i) {
        const int e = lane * kPer + i;
        hot[i] = e < E && ws.cursor[e] >= hot_min ? 1 : 0;
        sum += hot[i];
      }
      int incl = sum;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const int n = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += n;
      }
      const int total = __shfl_sync(0xffffffffu, incl, 31);
      int run = incl - sum;
#pragma unroll
      for (int i = 0; i < kPer; ++i) {
        const int e = lane * kPer + i;
        if (e < E) ws.order[hot[i] ? run : total + e - run] = e;
        run += hot[i];
      }
      if (lane == 0) ws.n_hot_experts = total;
    }
    __syncthreads();
  }
  if (tid < 64) {  // warp 0: tiles of the experts before expert e; warp 1: units of the experts placed before position e
    const bool units = tid >= 32;
    int c[kPer], sum = 0;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int e = lane * kPer + i;
      c[i] = e < E ? ws.cursor[units ? ws.order[e] : e] : 0;
      if (units) c[i] = (c[i] + pair - 1) / pair;
      sum += c[i];
    }
    int incl = sum;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int n = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += n;
    }
    int run = incl - sum;
    int* dst = units ? ws.units : wl.estart;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int e = lane * kPer + i;
      if (e < E) dst[e] = run;
      run += c[i];
    }
    if (lane == 31) dst[E] = incl;
  }
  __syncthreads();
  if (tid < 32) {
    if (hist != nullptr) {
      const int total = min(wl.estart[E], kMaxListTiles);
      for (int t = lane; t < total; t += 32) wl.tiles[t] = (uint16_t)t;  // regions are consecutive tiles
    } else {
      for (int e = lane; e < E; e += 32) ws.cursor[e] = wl.estart[e];
      __syncwarp();
      // stable scatter, 32 tiles at a time: the same list in every CTA
      for (int p0 = 0; p0 < P; p0 += 32) {
        const int p = p0 + lane;
        const unsigned e = p < P ? ws.owner[p] : 0xffffu;
        const unsigned peers = __match_any_sync(0xffffffffu, e);
        if (e != 0xffffu) wl.tiles[ws.cursor[e] + __popc(peers & ((1u << lane) - 1u))] = (uint16_t)p;
        __syncwarp();
        if (e != 0xffffu && lane == __ffs(peers) - 1) ws.cursor[e] += __popc(peers);
        __syncwarp();
      }
    }
  } else if (tid < 64) {
    const int* units = ws.units;
    const int total = units[E];
    // Position q's GEMM2 segment goes behind position after[q]'s GEMM1 segment: the first one at least `lag` GEMM1
    // items on.  The last positions keep their GEMM2 segments for the end of the list, so that they too have `lag`
    // items between the two (without that their GEMM2 items waited up to half an item for the intermediate).
    for (int q = lane; q < E; q += 32) {
      int after = E - 1;
      if (fused && (long long)NB2 * (units[max(E - 1, q + 1)] - units[q + 1]) >= lag) {
        int lo = q, hi = E - 1;  // first i > q with NB1 * (units up to i - units up to q) >= lag; none: the last position
        while (hi - lo > 1) {
          const int mid = (lo + hi) / 2;
          if ((long long)NB1 * (units[mid + 1] - units[q + 1]) >= lag) hi = mid; else lo = mid;
        }
        after = hi;
      }
      ws.after[q] = after;
    }
    __syncwarp();
    for (int i = lane; i < E; i += 32) {
      int before = 0, hi = E;  // GEMM2 segments in front of position i's GEMM1 segment: those with after[q] < i
      while (before < hi) {
        const int mid = (before + hi) / 2;
        if (ws.after[mid] < i) before = mid + 1; else hi = mid;
      }
      wl.seg_start[i + before] = NB1 * units[i] + NB2 * units[before];
      wl.seg_info[i + before] = ws.order[i];
      const int seg2 = ws.after[i] + 1 + i;
      wl.seg_start[seg2] = NB1 * units[ws.after[i] + 1] + NB2 * units[i];
      wl.seg_info[seg2] = ws.order[i] | (1 << 16);
    }
    if (lane == 0) {
      const bool split = !fused && hot_min > 0;
      wl.n_hot[0] = split ? NB1 * units[ws.n_hot_experts] : -1;  // -1: no interleaving
      wl.n_hot[1] = split ? NB2 * units[ws.n_hot_experts] : -1;
      wl.n1 = fused ? 0 : NB1 * total;
      wl.seg_start[2 * E] = (NB1 + NB2) * total;
    }
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the scratch becomes the target of TMA loads
  __syncthreads();
}

// Everything the expert-FFN kernels take.
struct FfnParams {
  const int* tile_expert;  // [P]
  int P, lag, fused;
  int hot_min;  // > 0: interleave tensor-bound and weight-streaming-bound items (see WorkList)
  const int* push_src;  // push-style combine: the source info t*K+k of every pool row - the GEMM2 epilogue stores row r
                        // of the pool at row push_src[r] of `out` (the token's own position) and skips rows whose
                        // source is negative (empty slots); nullptr: rows stay where they are
  const int* hist;  // rows per expert (the ordered dispatch's counts): the work list is built from them, or nullptr
  int hot_first;    // with hist: experts are walked by descending row count
  int band;         // > 0 (the launch that carries the dispatch): an expert's items go band by band of this many tiles
                    // (column-block-major inside a band), so the first items need only the expert's first tiles,
                    // which the token-ordered dispatch completes first; 0: column-block-major over all its tiles
  int thin;         // the narrow (transposed) form for single tiles of at most 64 rows is in use
  int cold_below;   // experts with fewer tiles than this stream their weights once: their loads are evict-first
  int phase, E, F, H;
  int tp;  // TP shards per expert: expert index e of the work list is shard e % tp of expert e / tp (the down matrix's map is 4-D)
  __nv_bfloat16* inter;
  __nv_bfloat16* out;
  int* gemm1_done;
  int* work_counter;  // [4] items handed out beyond the first one per CTA: [0] phases 0 and 1, [1] phase 2 (zero at launch; the
                      // last CTA to leave zeroes it again); [2], [3]: CTAs that left
  const int* tile_count;
  const int* rows_done;
  int total_rows;
  unsigned long long wait_ns;  // bound on every wait inside the kernel
  int* status;
  unsigned long long* clock_probe;  // [2]: SM cycles and nanoseconds CTA 0 spent in the kernel (accumulated)
  unsigned long long* item_ns;      // work-item timeline (measurement; nullptr: off): 4 words per position of the item list
};

// Effective SM clock while a kernel runs: CTA 0 adds its elapsed %clock64 and %globaltimer.
struct ClockProbe {
  unsigned long long* out;
  long long c0;
  unsigned long long t0;
  __device__ explicit ClockProbe(unsigned long long* o) : out(o), c0(0), t0(0) {
    if (out != nullptr && blockIdx.x == 0 && threadIdx.x == 0) {
      c0 = clock64();
      t0 = globaltimer();
    }
  }
  __device__ void finish() {
    if (out != nullptr && blockIdx.x == 0 && threadIdx.x == 0) {
      atomicAdd(out, (unsigned long long)(clock64() - c0));
      atomicAdd(out + 1, globaltimer() - t0);
    }
  }
};

// The CTA-pair (cta_group::2) kernel lives in ffn_tc2.cu.
int launch_ffn_pair(moe_plan* p, const void* recv, const void* wg, const void* wu, const void* wd, FfnParams prm,
                    cudaStream_t st);

// A handful of tokens: plain FMAs, every SM streams weights (ffn_few.cu).
constexpr int kFewMaxTokens = 32;  // (beyond five: small layers only)
bool few_applies(const moe_plan* p);
int launch_ffn_few(moe_plan* p, const void* recv, const void* wg, const void* wu, const void* wd, const FfnParams& prm,
                   const int* push_src, cudaStream_t st, bool own);

// ---- tensor maps (host side) ---------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline int get_encoder(moe_plan* p, EncodeTiledFn* fn) {
  if (!p->encode_tiled) {
    void* sym = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &sym, cudaEnableDefault, &q) != cudaSuccess || !sym ||
        q != cudaDriverEntryPointSuccess)
      return MOE_ERR_CUDA;
    p->encode_tiled = sym;
  }
  *fn = (EncodeTiledFn)p->encode_tiled;
  return MOE_OK;
}

// bf16 matrix [rows, cols] (row-major, cols contiguous), box [box_rows, 64 cols], 128-byte swizzle.
inline int make_map_2d(EncodeTiledFn enc, CUtensorMap* m, const void* base, uint64_t rows, uint64_t cols,
                       uint32_t box_rows) {
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {cols * 2};
  cuuint32_t box[2] = {(cuuint32_t)kBK, box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? MOE_OK : MOE_ERR_CUDA;
}
// bf16 tensor [E, rows, cols], box [1, box_rows, 64].
inline int make_map_3d(EncodeTiledFn enc, CUtensorMap* m, const void* base, uint64_t E, uint64_t rows, uint64_t cols,
                       uint32_t box_rows) {
  cuuint64_t dims[3] = {cols, rows, E};
  cuuint64_t strides[2] = {cols * 2, rows * cols * 2};
  cuuint32_t box[3] = {(cuuint32_t)kBK, box_rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? MOE_OK : MOE_ERR_CUDA;
}
// The down matrices [E, H, F*tp] seen as [E, tp, H, F]: shard s of an expert is the column slice [s*F, (s+1)*F).
// Box [1, 1, box_rows, 64].
inline int make_map_wd(EncodeTiledFn enc, CUtensorMap* m, const void* base, uint64_t experts, uint64_t tp, uint64_t rows,
                       uint64_t cols, uint32_t box_rows) {
  cuuint64_t dims[4] = {cols, rows, tp, experts};
  cuuint64_t strides[3] = {cols * tp * 2, cols * 2, rows * cols * tp * 2};
  cuuint32_t box[4] = {(cuuint32_t)kBK, box_rows, 1, 1};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? MOE_OK : MOE_ERR_CUDA;
}

}  // namespace moehub
