// Expert FFN of dtype fp32 on the 5th-generation tensor cores (paper Section II-A, expert computation; per-tile
// availability of the intermediate as in Section IV-D): both GEMMs in one persistent launch.
//
// An fp32 number is the exact sum of three bf16 numbers (8 + 8 + 8 significand bits: x = hi + mid + lo, each the rounded
// rest of what the ones before it left), a product of two such numbers is six bf16 products, and the three left out
// (mid*lo, lo*mid, lo*lo) are below 2^-25 of it.  Products of bf16 numbers are exact in the tensor cores; what they would
// lose is in the additions, which truncate: one accumulator over the whole sum is further from the sum in 64 bits than a
// chain of fp32 FMAs.  So hi*hi goes to an accumulator that is drained every 32 k (sums of fewer than 256 terms) or 64 k into fp32
// registers (two or four MMAs, then an addition that rounds to nearest), and the other five, 2^-8 of it, to one of their own
// that is read once.
//
//   an item: 128 weight rows (the M side) x the rows of one 128-row tile (the N side, rounded up to 16)
//   GEMM1: 64 gate and the same 64 up rows, 16 and 16 in every quarter of the accumulator's lanes, so that a lane finds
//          its partner 16 lanes on; S = silu(g) * u is written as three bf16 planes, which GEMM2 loads as they are
//   GEMM2: 128 rows of Wd, results in fp32
//
// The weights arrive as fp32 (TMA, 32 k of every row per stage) and are split by eight warps on their way into tensor
// memory, where the MMA takes its A operand: through shared memory they would cost its bandwidth 52 KB per 16 k and item
// of 128 rows instead of 40 (six MMAs read A and B, 48 KB; split, 12 KB written), and that is the bound.  The rows are
// split once, by split_rows_kernel in front.
//
// What infinities and NaN in the operands make of a sum, the hi*hi products say: hi of an infinity is one, hi of a number is zero
// only if the number is (or, in a group of large rows, below 2^-118), and their signs are the numbers' own.  The other five (inf * mid
// has any sign, inf * 0 none) are clamped to finite numbers before they are added, which changes nothing where hi*hi is infinite or
// NaN.  Where a value that is not finite has no infinity or NaN behind it, or also large numbers (an overflow, an hi that rounded up
// to infinity), the lane that holds it recomputes it as a chain of fp32 FMAs (unexplained, below).
//
// Roles (864 threads): warp 0 claims and publishes the items and loads weights, warp 1 MMA issuer and TMEM owner, warps 2-9
// split weights (two sets of four, two A stages each), warps 10-25 drain accumulators and write results, warp 26 loads the
// rows' planes (apart from the weights, which need not wait for a GEMM2 item's intermediate).  Every wait is bounded in time.
#include <float.h>

#include "tc_common.cuh"

namespace moehub {

constexpr int kSpDrainWarps = 16;
constexpr int kSpThreads = 32 * (2 + 8 + kSpDrainWarps + 1);
constexpr int kSpWStages = 7, kSpBStages = 2;
constexpr int kSpWBytes = 128 * 32 * 4;             // 128 weight rows x 32 k, fp32
constexpr int kSpBBytes = 3 * kTileRows * kBK * 2;  // three planes of up to 128 rows x 64 k, bf16
constexpr int kSpRing = 16;  // the weights' producer is at most 7 items (W stages) ahead of the splitters, those 2 of the MMAs, those 2 of the drain
constexpr int kSpSmem = kSpBStages * kSpBBytes + kSpWStages * kSpWBytes + 1024 /*alignment*/ + 576 /*barriers*/;
constexpr uint32_t kSpRest = 256, kSpA = 384;       // tensor-memory columns: hi*hi at 0 and 128, the rest, four A stages of 3 x 8

struct SplitMaps {
  CUtensorMap wg, wu, wd;
  CUtensorMap rows[2][4];  // planes of recv, of the intermediate: boxes of 128, 64, 32 and 16 rows x 64 k x 3 planes
};
struct SplitParams {
  const int* tile_expert;  // [P]
  const int* tile_count;   // [P] rows per tile, or nullptr: every tile is computed whole
  const int* rows_done;
  int total_rows;
  int P, E, F, H, tp, lag;
  const float *recv, *wg, *wu, *wd;
  const __nv_bfloat16* recv_planes;  // [3][P * 128][recv_pitch]
  const uint2* group_large;          // [P] a byte for each of a tile's eight groups of 16 rows
  __nv_bfloat16* inter;              // [3][P * 128][inter_pitch]
  int recv_pitch, inter_pitch;
  float* out;              // [P * 128, H]
  int* gemm1_done;
  int* work_counter;
  unsigned long long wait_ns;
  int* status;
};
struct SplitShared {
  unsigned long long w_full[kSpWStages], w_empty[kSpWStages];
  unsigned long long b_full[kSpBStages], b_empty[kSpBStages];
  unsigned long long a_full[4], a_empty[4];
  unsigned long long hh_full[2], hh_empty[2];
  unsigned long long rest_full, rest_empty;
  unsigned long long item_bar[kSpRing];
  unsigned long long drain;
  int item_large[kSpRing];  // bit i: group i of the item's tile holds large numbers
  int item_ring[kSpRing];  // item | (rows of its tile / 16, rounded up) << kSpRowShift, or -1
  int w_fills;
  uint32_t b_fills[2];     // of each B stage
  uint32_t tmem_base;
  int abort_flag;
  int last_cta;
};
static_assert(sizeof(SplitShared) <= 576, "barriers behind the stages");
constexpr int kSpRowShift = 23;
constexpr int kSpDrain64 = 256;  // from sums of this length on, hi*hi is drained every 64 k instead of 32
template <uint32_t V> struct Const { static constexpr uint32_t value = V; };

// bf16 has fp32's exponents, so the last of three parts of a number below 2^-109 would have none left.  Weights are split times 2^16
// (down to fp32's smallest that keeps every bit), and so are the rows and the intermediate of a group of 16 rows, or, where one of
// its x is 2^32 and more, times 2^-16, so that their sums keep their range: the products come out times 2^32 or as they are.
// Without the scales, off by (relative, H 512, F 1024; fp32 FMAs 5.9e-7, with them 2.4e-7): Wd of size 2^-115 1.1e-6, of 2^-120 3.5e-5, of 2^-125
// 1.1e-3.  They take 1 to 2 % (T 1000, H 1024, 16 experts, F 2048 233.5 -> 236.7 us, T 300, H 400, F 500 49.4 -> 50.5).
constexpr float kUp = 65536.0f, kDown = 1.0f / 65536.0f, kLargeRow = 4294967296.0f;
constexpr int kSplitRows = 16;  // rows of a group
__device__ __forceinline__ float group_scale(int large) { return large ? kDown : kUp; }
__device__ __forceinline__ float group_result(int large) { return large ? 1.0f : kDown * kDown; }  // what a sum of a group's products is to be multiplied by

// Three bf16 numbers whose sum is x, if hi is finite.  A finite element of the intermediate for which it would not be has kBits, a NaN
// that no conversion gives, in its place and its own bits in the other two (store_top).
constexpr unsigned short kBits = 0x7fc1;
__device__ __forceinline__ void split3(float x, __nv_bfloat16& hi, __nv_bfloat16& mid, __nv_bfloat16& lo) {
  hi = __float2bfloat16_rn(x);
  const float r = x - __bfloat162float(hi);
  mid = __float2bfloat16_rn(r);
  lo = __float2bfloat16_rn(r - __bfloat162float(mid));
}
__device__ __forceinline__ uint32_t pack2(float a, float b) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&h);
}
// x minus the bf16 number in the lower half of w (exact product, one rounding: the same as widening it first).
__device__ __forceinline__ float minus_low(float x, uint32_t w) {
  asm("fma.rn.f32.bf16 %0, %1, %2, %0;" : "+f"(x) : "h"((unsigned short)w), "h"((unsigned short)0xbf80));
  return x;
}
// Two numbers at once, without the care for the largest ones (their results are recomputed anyway).
__device__ __forceinline__ void split_pair(float a, float b, uint32_t& hi, uint32_t& mid, uint32_t& lo) {
  hi = pack2(a, b);
  a = minus_low(a, hi);
  b -= __uint_as_float(hi & 0xffff0000u);
  mid = pack2(a, b);
  lo = pack2(minus_low(a, mid), b - __uint_as_float(mid & 0xffff0000u));
}

__device__ __forceinline__ unsigned long long mul_x2(unsigned long long v, float by) {
  unsigned long long d;
  asm("{\n\t.reg .b64 t;\n\tmov.b64 t, {%2, %2};\n\tmul.rn.f32x2 %0, %1, t;\n\t}" : "=l"(d) : "l"(v), "f"(by));
  return d;
}
// The same of two weights' bits, times kUp.
__device__ __forceinline__ void split_pair_up(uint32_t a, uint32_t b, uint32_t& hi, uint32_t& mid, uint32_t& lo) {
  const unsigned long long v = mul_x2((unsigned long long)b << 32 | a, kUp);
  split_pair(__uint_as_float((uint32_t)v), __uint_as_float((uint32_t)(v >> 32)), hi, mid, lo);
}

// A operand in tensor memory: D[128, N] (+)= A[128, 16] * B[N, 16]^T.
__device__ __forceinline__ void tc_mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void tc_st8(uint32_t taddr, const uint32_t* r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr), "r"(r[0]), "r"(r[1]),
               "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]) : "memory");
}
__device__ __forceinline__ void add_x2(unsigned long long& acc, uint32_t lo, uint32_t hi) {
  asm("{\n\t.reg .b64 t;\n\tmov.b64 t, {%1, %2};\n\tadd.rn.f32x2 %0, %0, t;\n\t}" : "+l"(acc) : "r"(lo), "r"(hi));
}
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Rows of the pool to planes [3][rows][pitch].  A CTA takes rows of one tile; rows nobody wrote to are left out.
__global__ void __launch_bounds__(256) split_rows_kernel(const float* __restrict__ x, const int* __restrict__ tile_expert,
                                                         const int* __restrict__ tile_count, const int* __restrict__ rows_done,
                                                         int total_rows, int E, int H, int pitch, size_t plane,
                                                         __nv_bfloat16* __restrict__ out, unsigned char* __restrict__ group_large) {
  pdl_wait();
  pdl_trigger();
  const int tile = blockIdx.x / (kTileRows / kSplitRows), r0 = blockIdx.x % (kTileRows / kSplitRows) * kSplitRows;
  const int e = tile_expert[tile];
  if (e < 0 || e >= E) return;
  int rows = kTileRows;
  if (tile_count != nullptr && *rows_done >= total_rows) rows = min(kTileRows, tile_count[tile]);
  rows = min(rows - r0, kSplitRows);
  const int quads = H / 4;
  auto split = [&](float scale) {  // whether one of them is large
    bool large = false;
    for (int i = threadIdx.x; i < rows * quads; i += 256) {
      const int r = i / quads, c = (i - r * quads) * 4;
      const size_t row = (size_t)tile * kTileRows + r0 + r;
      const float4 v = *reinterpret_cast<const float4*>(x + row * H + c);
      const float f[4] = {v.x, v.y, v.z, v.w};
      __align__(8) __nv_bfloat16 s[3][4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        split3(f[j] * scale, s[0][j], s[1][j], s[2][j]);
        large |= fabsf(f[j]) >= kLargeRow;
      }
#pragma unroll
      for (int q = 0; q < 3; ++q) *reinterpret_cast<uint2*>(out + q * plane + row * pitch + c) = *reinterpret_cast<const uint2*>(s[q]);
    }
    return large;
  };
  const int large = __syncthreads_or(split(kUp));
  if (large) split(kDown);
  if (threadIdx.x == 0) group_large[blockIdx.x] = large ? 1 : 0;
}

// Which of a warp's values that are not finite (bits of todo: rows h * 16 + 0...15 of the tile, and from bit 16 on the sixteen
// that lie 64 rows on) are what their operands' infinities and NaN make of them: the row's, and those of this lane's weight row and,
// in GEMM1, of the one 16 lanes on.  Returns the others.  All 32 lanes.  Large numbers are those whose products may add up to an overflow.
// Measured, layer, T 1000, H 1024, 16 experts, top-2, F 2048 (215 us as a rule), us, FMAs / every such value recomputed / this: one
// row with a NaN 737 / 465 / 217, one infinity in one Wg 741 / 24589 / 362, in every Wg 737 / 48854 / 571, every row NaN 698 / 66874 / 305,
// infinite 698 / - / 549, every Wg NaN 743 / - / 643.
struct Explain {
  const __nv_bfloat16* rows;    // hi plane
  const float* w;
  int pitch, K;
  bool paired;                  // GEMM1
};
constexpr float kLarge = 1.0e15f, kLargePart = 1.0e13f;  // (of a weight; of a row's hi, which may stand for 2^16 times as much: half a million products)
__device__ __noinline__ uint32_t unexplained(const Explain& q, uint32_t todo) {
  const int lane = threadIdx.x % 32;
  constexpr uint32_t all = 0xffffffffu;
  uint32_t row_inf = 0, row_large = 0;
  for (uint32_t m = __reduce_or_sync(all, todo); m != 0; m &= m - 1) {
    const uint32_t bit = m & (0u - m);
    const int b = __ffs(m) - 1;
    const uint2* at = reinterpret_cast<const uint2*>(q.rows + (size_t)((b >> 4) * 64 + (b & 15)) * q.pitch);
    for (int k0 = 0; k0 < q.K; k0 += 512) {
      bool nan = false;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int k = k0 + i * 128 + lane * 4;
        const uint2 v = k < q.K ? at[k / 4] : make_uint2(0u, 0u);
        const uint32_t f[4] = {v.x << 16 & 0x7fff0000u, v.x & 0x7fff0000u, v.y << 16 & 0x7fff0000u, v.y & 0x7fff0000u};  // magnitudes' bits
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          nan |= f[j] > 0x7f800000u && f[j] != (uint32_t)kBits << 16;
          if (f[j] == 0x7f800000u) row_inf |= bit;
          else if (f[j] > __float_as_uint(kLargePart)) row_large |= bit;
        }
      }
      if (__any_sync(all, nan)) {
        todo &= ~bit;
        break;
      }
    }
  }
  row_inf = __reduce_or_sync(all, row_inf);
  row_large = __reduce_or_sync(all, row_large);
  const uint32_t here = todo;
  if (q.paired) todo |= __shfl_xor_sync(all, todo, 16);
  uint32_t flags = 0;  // of this lane's weight row: 1 NaN (then looked at no further), 2 an infinity, 4 a large number
  for (uint32_t m = __ballot_sync(all, todo != 0); m != 0; m &= m - 1) {
    const int from = __ffs(m) - 1;
    const float* w = reinterpret_cast<const float*>(__shfl_sync(all, reinterpret_cast<unsigned long long>(q.w), from));
    uint32_t seen = 0;
    for (int k0 = 0; k0 < q.K; k0 += 512) {
      uint32_t now = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int k = k0 + i * 128 + lane * 4;
        const float4 v = k < q.K ? *reinterpret_cast<const float4*>(w + k) : make_float4(0.f, 0.f, 0.f, 0.f);
        const float f[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (!(fabsf(f[j]) <= kLarge)) now |= isnan(f[j]) ? 1u : isinf(f[j]) ? 2u : 4u;
      }
      seen |= __reduce_or_sync(all, now);
      if (seen & 1u) break;
    }
    if (lane == from) flags = seen;
  }
  const uint32_t others = __shfl_xor_sync(all, flags, 16);
  if (q.paired) flags |= others;
  if (flags & 1u) return 0u;
  if (!(flags & 4u)) todo &= ~((flags & 2u ? all : row_inf) & ~row_large);
  return todo & here;
}
// The recomputation of a value that is not finite.
__device__ __noinline__ float fp32_chain(const float* __restrict__ a, const float* __restrict__ b, int n) {
  float s = 0.0f;
  for (int k = 0; k < n; ++k) s = __fmaf_rn(a[k], b[k], s);
  return s;
}
// (a: written by other CTAs of this launch, so neither const __restrict__ nor any other way to the non-coherent loads)
__device__ __noinline__ float fp32_chain_planes(const __nv_bfloat16* a, size_t plane, float unscale, const float* b, int n) {
  float s = 0.0f;
  for (int k = 0; k < n; ++k) {
    const float hi = __bfloat162float(a[k]), mid = __bfloat162float(a[plane + k]), lo = __bfloat162float(a[2 * plane + k]);
    float v = (hi + (mid + lo)) * unscale;
    if (!(fabsf(hi) <= FLT_MAX)) v = __float_as_uint(hi) >> 16 == kBits ? __uint_as_float(__float_as_uint(mid) | __float_as_uint(lo) >> 16) : hi;
    s = __fmaf_rn(v, b[k], s);
  }
  return s;
}
constexpr float kNearTop = 3.38e38f;  // (bf16's largest finite number is 3.39e38: beyond that a number may round to infinity)
// The parts of s, an element of the intermediate, in a group of this scale.
__device__ __forceinline__ void store_top(float s, float scale, __nv_bfloat16* to, size_t plane) {
  split3(s * scale, to[0], to[plane], to[2 * plane]);
  if (fabsf(s) <= FLT_MAX && !(fabsf(s * scale) <= kNearTop)) {
    to[0] = __ushort_as_bfloat16(kBits);
    to[plane] = __ushort_as_bfloat16((unsigned short)(__float_as_uint(s) >> 16));
    to[2 * plane] = __ushort_as_bfloat16((unsigned short)__float_as_uint(s));
  }
}
__device__ __forceinline__ bool is_finite(float v) { return fabsf(v) < FLT_MAX; }  // (or the largest, which a clamped number leaves)

__global__ void __launch_bounds__(kSpThreads, 1)
ffn_split_kernel(const __grid_constant__ SplitMaps maps, const SplitParams prm) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t* w_base = base + kSpBStages * kSpBBytes;
  SplitShared* sh = reinterpret_cast<SplitShared*>(w_base + kSpWStages * kSpWBytes);
  __shared__ WorkList wl;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int E = prm.E, F = prm.F, H = prm.H, nseg = 2 * E;
  const int NB1 = (F + 63) / 64, NB2 = (H + 127) / 128;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kSpWStages; ++s) { mbar_init(smem_u32(&sh->w_full[s]), 1); mbar_init(smem_u32(&sh->w_empty[s]), 4); }
    for (int s = 0; s < kSpBStages; ++s) { mbar_init(smem_u32(&sh->b_full[s]), 1); mbar_init(smem_u32(&sh->b_empty[s]), 1); }
    for (int s = 0; s < 4; ++s) { mbar_init(smem_u32(&sh->a_full[s]), 4); mbar_init(smem_u32(&sh->a_empty[s]), 1); }
    for (int s = 0; s < 2; ++s) {
      mbar_init(smem_u32(&sh->hh_full[s]), 1);
      mbar_init(smem_u32(&sh->hh_empty[s]), kSpDrainWarps);
    }
    mbar_init(smem_u32(&sh->rest_full), 1);
    mbar_init(smem_u32(&sh->rest_empty), kSpDrainWarps);
    for (int i = 0; i < kSpRing; ++i) mbar_init(smem_u32(&sh->item_bar[i]), 1);
    mbar_init(smem_u32(&sh->drain), 1);
    sh->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sh->tmem_base)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  pdl_wait();
  int first_claim = 0;
  if (threadIdx.x == 0) first_claim = atomicAdd(prm.work_counter, 1);  // in flight while the work list is built
  build_worklist(wl, *reinterpret_cast<WorkScratch*>(base), prm.tile_expert, prm.P, E, NB1, NB2, prm.lag, 1, 1);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = uniform(sh->tmem_base);
  volatile int* abort_flag = &sh->abort_flag;
  const unsigned long long wait_ns = prm.wait_ns;
  const int item_end = wl.seg_start[nseg];

  int seg_cursor = -1;
  auto decode = [&](int item) {  // (a role's items only move forward: only its first lookup is a search)
    int lo = seg_cursor;
    if (lo < 0) {
      int hi = nseg;
      lo = 0;
      while (hi - lo > 1) {
        const int mid = (lo + hi) / 2;
        if (wl.seg_start[mid] <= item) lo = mid; else hi = mid;
      }
    } else {
      while (wl.seg_start[lo + 1] <= item) ++lo;
    }
    seg_cursor = lo;
    Item it;
    it.type = wl.seg_info[lo] >> 16;
    it.e = wl.seg_info[lo] & 0xffff;
    it.m = wl.estart[it.e + 1] - wl.estart[it.e];
    it.cold = it.m == 1;
    const int local = item - wl.seg_start[lo];
    it.nb = local / it.m;
    it.tile = wl.tiles[wl.estart[it.e] + local % it.m];
    return it;
  };
  volatile int* item_ring = sh->item_ring;
  // the item published in this slot, -1: no more
  auto entry_of = [&](int local_item) { return item_ring[local_item & (kSpRing - 1)]; };
  auto item_wait = [&](int local_item) {
    return mbar_wait(smem_u32(&sh->item_bar[local_item & (kSpRing - 1)]), (uint32_t)(local_item / kSpRing) & 1u, abort_flag, wait_ns);
  };
  // the smallest of the row boxes (128, 64, 32, 16 rows) that holds this many times 16 rows
  auto box_of = [](int n16) { return n16 > 4 ? 0 : n16 > 2 ? 1 : n16 > 1 ? 2 : 3; };

  int fail_site = 0;
  if (warp == 0) {
    // ===================== items and weights =====================
    if (lane == 0) {
      const bool counted = prm.tile_count != nullptr && ld_acquire(prm.rows_done) >= prm.total_rows;
      const uint64_t pol_once = l2_policy_evict_first();
      int ws = 0, fills = 0;
      uint32_t w_ph = 0;
      int item = first_claim;
      for (int local_item = 0; !fail_site; ++local_item) {
        const int slot = local_item & (kSpRing - 1);
        if (item >= item_end) {
          item_ring[slot] = -1;
          mbar_arrive(smem_u32(&sh->item_bar[slot]));
          break;
        }
        const int next_item = atomicAdd(prm.work_counter, 1);  // used after this item's loads
        const Item it = decode(item);
        if (it.tile < 0 || it.tile >= prm.P || it.e < 0 || it.e >= E) {  // own index check on what the work list gave
          set_status(prm.status, MOE_ERR_INTERNAL, 221);
          fail_site = kWaitItem;
          break;
        }
        const int rows = counted ? min(kTileRows, prm.tile_count[it.tile]) : kTileRows;
        item_ring[slot] = item | (max(1, (rows + 15) / 16) << kSpRowShift);
        {
          const uint2 g = prm.group_large[it.tile];
          auto bits = [](uint32_t w) { return (w & 1u) | (w >> 7 & 2u) | (w >> 14 & 4u) | (w >> 21 & 8u); };
          *(volatile int*)&sh->item_large[slot] = (int)(bits(g.x) | bits(g.y) << 4);
        }
        mbar_arrive(smem_u32(&sh->item_bar[slot]));
        const int KW = ((it.type == 0 ? H : F) + 31) / 32;
        for (int kw = 0; kw < KW; ++kw) {
          if (!mbar_wait(smem_u32(&sh->w_empty[ws]), w_ph ^ 1u, abort_flag, wait_ns)) { fail_site = kWaitMbarTma; break; }
          const uint32_t full = smem_u32(&sh->w_full[ws]), dst = smem_u32(w_base + ws * kSpWBytes);
          mbar_expect_tx(full, (uint32_t)kSpWBytes);
          if (it.type == 0) {
            if (it.cold) {
              tma_load_3d_hint(dst, &maps.wg, full, kw * 32, it.nb * 64, it.e, pol_once);
              tma_load_3d_hint(dst + kSpWBytes / 2, &maps.wu, full, kw * 32, it.nb * 64, it.e, pol_once);
            } else {
              tma_load_3d(dst, &maps.wg, full, kw * 32, it.nb * 64, it.e);
              tma_load_3d(dst + kSpWBytes / 2, &maps.wu, full, kw * 32, it.nb * 64, it.e);
            }
          } else if (it.cold) {
            tma_load_4d_hint(dst, &maps.wd, full, kw * 32, it.nb * 128, it.e % prm.tp, it.e / prm.tp, pol_once);
          } else {
            tma_load_4d(dst, &maps.wd, full, kw * 32, it.nb * 128, it.e % prm.tp, it.e / prm.tp);
          }
          ++fills;
          if (++ws == kSpWStages) { ws = 0; w_ph ^= 1u; }
        }
        item = next_item;
      }
      if (fail_site) sh->abort_flag = 1;
      sh->w_fills = fills;
    }
  } else if (warp == 2 + 8 + kSpDrainWarps) {
    // ===================== the rows' planes =====================
    if (lane == 0) {
      uint32_t b_ph = 0;  // bit s: parity of the uses of stage s
      uint32_t b_uses[2] = {0, 0};
      for (int local_item = 0; !fail_site; ++local_item) {
        if (!item_wait(local_item)) { fail_site = kWaitItem; break; }
        const int entry = entry_of(local_item);
        if (entry < 0) break;
        const int q = box_of(entry >> kSpRowShift);
        const Item it = decode(entry & ((1 << kSpRowShift) - 1));
        if (it.type == 1) {  // every drain warp of every GEMM1 block has bumped the tile's counter
          const int need = kSpDrainWarps * NB1;
          if (ld_acquire(&prm.gemm1_done[it.tile]) < need) {
            const unsigned long long t0 = globaltimer();
            while (ld_acquire(&prm.gemm1_done[it.tile]) < need) {
              if (*abort_flag || globaltimer() - t0 > wait_ns) { fail_site = kWaitTileReady; break; }
              __nanosleep(64);
            }
            if (fail_site) break;
          }
          asm volatile("fence.proxy.async.global;" ::: "memory");
        }
        const int KB = ((it.type == 0 ? H : F) + kBK - 1) / kBK;
        for (int kb = 0; kb < KB; ++kb) {
          const int bs = kb & 1;
          if (!mbar_wait(smem_u32(&sh->b_empty[bs]), ((b_ph >> bs) & 1u) ^ 1u, abort_flag, wait_ns)) { fail_site = kWaitMbarTma; break; }
          const uint32_t full = smem_u32(&sh->b_full[bs]);
          mbar_expect_tx(full, (uint32_t)(3 * (kTileRows >> q) * kBK * 2));
          tma_load_3d(smem_u32(base + bs * kSpBBytes), &maps.rows[it.type][q], full, kb * kBK, it.tile * kTileRows, 0);
          b_ph ^= 1u << bs;
          if (bs == 0) ++b_uses[0]; else ++b_uses[1];
        }
      }
      if (fail_site) sh->abort_flag = 1;
      sh->b_fills[0] = b_uses[0];
      sh->b_fills[1] = b_uses[1];
    }
  } else if (warp == 1) {
    // ===================== MMA issuer =====================
    // One elected lane, and operands that are a base and a constant: an item starts at B stage 0 and hi*hi accumulator 0, and
    // its 32-k blocks take the A stages 0, 1 and 2, 3 in turn.  Behind `lane == 0`, or with stages counted through,
    // moving each MMA's operands to uniform registers takes 45 clocks and more (N 128 takes 64, N 16 9).
    if (elect_one()) {
      const uint64_t b_base = smem_desc_sw128(smem_u32(base));
      uint32_t a_ph = 0, h_ph = 0, b_ph = 0;  // bit i: parity of the uses of A stages 2 i and 2 i + 1, of hi*hi accumulator i, of B stage i
      for (int local_item = 0; !fail_site; ++local_item) {
        if (!item_wait(local_item)) { fail_site = kWaitItem; break; }
        const int entry = entry_of(local_item);
        if (entry < 0) break;
        const int n16 = entry >> kSpRowShift;
        const int K = decode(entry & ((1 << kSpRowShift) - 1)).type == 0 ? H : F, KW = (K + 31) / 32;
        const uint32_t idesc = thin_idesc(n16);
        const uint64_t plane = (uint64_t)((kTileRows >> box_of(n16)) * kBK * 2) >> 4;  // descriptor units
        if (!mbar_wait(smem_u32(&sh->rest_empty), ((uint32_t)local_item & 1u) ^ 1u, abort_flag, wait_ns)) { fail_site = kWaitMbarTmemFree; break; }
        uint32_t first = 0;
        // Half HALF (32 k) of B stage BS, into hi*hi accumulator HH from its start or on top of the first half.  A look at a
        // barrier takes some hundred clocks even when it has long completed, so the next one is looked at before the MMAs in
        // front of it are issued.
        auto block = [&](auto bs_c, auto half_c, auto hh_c, auto start_c, bool end) {
          constexpr uint32_t BS = decltype(bs_c)::value, HALF = decltype(half_c)::value, HH = decltype(hh_c)::value, START = decltype(start_c)::value;
          const uint32_t ap = (a_ph >> HALF) & 1u, hp = ((h_ph >> HH) & 1u) ^ 1u, rest = tmem + kSpRest, hh = tmem + HH * 128u;
          const uint64_t b = b_base + BS * (kSpBBytes >> 4) + 4 * HALF;
          const uint32_t a0 = smem_u32(&sh->a_full[2 * HALF]), a1 = a0 + 8, hb = smem_u32(&sh->hh_empty[HH]), bb = smem_u32(&sh->b_full[BS]);
          const bool b_ok = HALF != 0 || mbar_test(bb, (b_ph >> BS) & 1u), hh_ok = START == 0 || mbar_test(hb, hp), a0_ok = mbar_test(a0, ap);
          if (!b_ok && !mbar_wait(bb, (b_ph >> BS) & 1u, abort_flag, wait_ns)) { fail_site = kWaitMbarMma; return; }
          if (!hh_ok && !mbar_wait(hb, hp, abort_flag, wait_ns)) { fail_site = kWaitMbarTmemFree; return; }
          if (!a0_ok && !mbar_wait(a0, ap, abort_flag, wait_ns)) { fail_site = kWaitMbarMma; return; }
          auto mmas = [&](auto k_c) {
            constexpr uint32_t k = decltype(k_c)::value;
            const uint32_t a = tmem + kSpA + (2 * HALF + k) * 24u;
            const uint64_t bk = b + 2 * k;
            tc_fence_after();
            tc_mma_ts(hh, a, bk, idesc, START != 0 && k == 0 ? 0u : 1u);
            if (k == 1 && end) tc_commit(smem_u32(&sh->hh_full[HH]));
            tc_mma_ts(rest, a + 16, bk, idesc, first);         // lo * hi
            tc_mma_ts(rest, a, bk + 2 * plane, idesc, 1u);     // hi * lo
            tc_mma_ts(rest, a + 8, bk + plane, idesc, 1u);     // mid * mid
            tc_mma_ts(rest, a + 8, bk, idesc, 1u);             // mid * hi
            tc_mma_ts(rest, a, bk + plane, idesc, 1u);         // hi * mid
            tc_commit(smem_u32(&sh->a_empty[2 * HALF + k]));
            first = 1;
          };
          const bool a1_ok = mbar_test(a1, ap);
          mmas(Const<0>());
          if (!a1_ok && !mbar_wait(a1, ap, abort_flag, wait_ns)) { fail_site = kWaitMbarMma; return; }
          mmas(Const<1>());
          a_ph ^= 1u << HALF;
          if (end) h_ph ^= 1u << HH;
        };
        const bool drain64 = K >= kSpDrain64;
        auto step = [&](auto bs_c, int kw) {  // 64 k
          const bool both = kw + 1 < KW;
          if (drain64) {
            block(bs_c, Const<0>(), bs_c, Const<1>(), !both);
            if (!fail_site && both) block(bs_c, Const<1>(), bs_c, Const<0>(), true);
          } else {
            block(bs_c, Const<0>(), Const<0>(), Const<1>(), true);
            if (!fail_site && both) block(bs_c, Const<1>(), Const<1>(), Const<1>(), true);
          }
          if (fail_site) return;
          tc_commit(smem_u32(&sh->b_empty[decltype(bs_c)::value]));
          b_ph ^= 1u << decltype(bs_c)::value;
        };
        for (int kw = 0; kw < KW && !fail_site; kw += 4) {
          step(Const<0>(), kw);
          if (!fail_site && kw + 2 < KW) step(Const<1>(), kw + 2);
        }
        if (fail_site) break;
        tc_commit(smem_u32(&sh->rest_full));
      }
      if (fail_site) sh->abort_flag = 1;
    }
    __syncwarp();
  } else if (warp < 10) {
    // ===================== weight splitters =====================
    // Four warps take every second 32-k block: lane l of the warp of quarter q reads the 128 bytes of one weight row and
    // writes its three bf16 rows to tensor-memory lane 32 q + l.  (128-byte swizzle: 16-byte unit u of row r is at u ^ r % 8.)
    const int q = warp & 3, set = (warp - 2) / 4;
    const uint32_t a = tmem + ((uint32_t)(q * 32) << 16) + kSpA + (uint32_t)set * 48u;  // two A stages of 16 k
    uint32_t mine = 0, ws = 0, w_ph = 0;  // blocks of this set so far; the next block's W stage
    for (int local_item = 0; !fail_site; ++local_item) {
      if (!warp_agrees(item_wait(local_item))) { fail_site = kWaitItem; break; }
      const int entry = entry_of(local_item);
      if (entry < 0) break;
      const Item it = decode(entry & ((1 << kSpRowShift) - 1));
      const int KW = ((it.type == 0 ? H : F) + 31) / 32;
      const int row = it.type == 1 ? q * 32 + lane : lane < 16 ? q * 16 + lane : 64 + q * 16 + lane - 16;
      const uint32_t r_off = (uint32_t)row * 128u, sw = (uint32_t)(row & 7) << 4;
      for (int kw = 0; kw < KW; ++kw) {
        const uint32_t s = ws, ph = w_ph;
        if (++ws == kSpWStages) { ws = 0; w_ph ^= 1u; }
        if ((kw & 1) != set) continue;
        if (!warp_agrees(mbar_wait(smem_u32(&sh->w_full[s]), ph, abort_flag, wait_ns))) { fail_site = kWaitMbarTma; break; }
        const uint32_t src = smem_u32(w_base) + s * (uint32_t)kSpWBytes + r_off;
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          uint32_t hi[8], mid[8], lo[8];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const uint4 v = lds128(src + (((uint32_t)(half * 4 + u) << 4) ^ sw));
            split_pair_up(v.x, v.y, hi[2 * u], mid[2 * u], lo[2 * u]);
            split_pair_up(v.z, v.w, hi[2 * u + 1], mid[2 * u + 1], lo[2 * u + 1]);
          }
          // (the split is done by the time the stage is free: the stages are two rounds of a splitter ahead of the MMAs)
          if (!warp_agrees(mbar_wait(smem_u32(&sh->a_empty[2 * set + half]), (mine & 1u) ^ 1u, abort_flag, wait_ns))) { fail_site = kWaitMbarMma; break; }
          tc_fence_after();
          tc_st8(a + half * 24, hi);
          tc_st8(a + half * 24 + 8, mid);
          tc_st8(a + half * 24 + 16, lo);
          tc_wait_st();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(smem_u32(&sh->a_full[2 * set + half]));
          if (half == 1 && lane == 0) mbar_arrive(smem_u32(&sh->w_empty[s]));
        }
        if (fail_site) break;
        ++mine;
      }
    }
    if (fail_site) sh->abort_flag = 1;
  } else {
    // ===================== drain and epilogue =====================
    // Accumulator lanes are weight rows, its columns the tile's rows: this warp adds up the units of 16 rows h and h + 4
    // of its quarter of the lanes.
    const int q = warp & 3, h = (warp - 10) / 4;
    const uint32_t lanes = tmem + ((uint32_t)(q * 32) << 16);
    uint32_t h_ph = 0;  // bit i: parity of the uses of hi*hi accumulator i
    const size_t plane = (size_t)prm.P * kTileRows * prm.inter_pitch;
    const bool counted = prm.tile_count != nullptr && ld_acquire(prm.rows_done) >= prm.total_rows;
    for (int local_item = 0; !fail_site; ++local_item) {
      if (!warp_agrees(item_wait(local_item))) { fail_site = kWaitItem; break; }
      const int entry = entry_of(local_item);
      if (entry < 0) break;
      const int n16 = entry >> kSpRowShift;
      const Item it = decode(entry & ((1 << kSpRowShift) - 1));
      const int rows = counted ? min(kTileRows, prm.tile_count[it.tile]) : kTileRows;
      const int K = it.type == 0 ? H : F, chunks = K >= kSpDrain64 ? (K + 63) / 64 : (K + 31) / 32;
      unsigned long long sum[2][8];  // (pairs of fp32 sums)
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) sum[i][j] = 0ull;
      auto add = [&](uint32_t from, auto rest) {
        if (h >= n16) return;
        uint32_t r[2][16];  // (the second unit whether or not it has rows: a condition on one load has the compiler spill; the
        tc_ld16(lanes + from + (uint32_t)h * 16u, r[0]);        // columns exist, and the sums are not used)
        tc_ld16(lanes + from + (uint32_t)(h + 4) * 16u, r[1]);
        tc_wait_ld();
        if (decltype(rest)::value != 0)
#pragma unroll
          for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 16; ++j) r[i][j] = __float_as_uint(fminf(fmaxf(__uint_as_float(r[i][j]), -FLT_MAX), FLT_MAX));
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int j = 0; j < 8; ++j) add_x2(sum[i][j], r[i][2 * j], r[i][2 * j + 1]);
      };
      for (int c = 0; c < chunks; ++c) {
        const uint32_t half = (uint32_t)c & 1u;
        if (!warp_agrees(mbar_wait(smem_u32(&sh->hh_full[half]), (h_ph >> half) & 1u, abort_flag, wait_ns))) { fail_site = kWaitMbarEpi; break; }
        h_ph ^= 1u << half;
        tc_fence_after();
        add(half * 128u, Const<0>());
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&sh->hh_empty[half]));
      }
      if (fail_site) break;
      if (!warp_agrees(mbar_wait(smem_u32(&sh->rest_full), (uint32_t)local_item & 1u, abort_flag, wait_ns))) { fail_site = kWaitMbarEpi; break; }
      tc_fence_after();
      add(kSpRest, Const<1>());
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&sh->rest_empty));
      const int large = *(volatile int*)&sh->item_large[local_item & (kSpRing - 1)] >> h;  // bits 0 and 4: of this warp's two groups
      const size_t row0 = (size_t)it.tile * kTileRows;
      const float unscale[2] = {group_result(large & 1), group_result(large >> 4 & 1)};
      auto acc = [&](int i, int j) { return __uint_as_float((uint32_t)(sum[i][j >> 1] >> (32 * (j & 1)))) * unscale[i]; };
      uint32_t bad = 0;  // results that are not finite
      auto exist = [&]() { return ((1u << min(max(rows - h * 16, 0), 16)) - 1u) | ((1u << min(max(rows - (h + 4) * 16, 0), 16)) - 1u) << 16; };
      if (it.type == 0) {
        const bool up = lane >= 16, odd = (lane & 1) != 0;
        const int f = it.nb * 64 + q * 16 + (lane & 15);
        const size_t pitch = (size_t)prm.inter_pitch;
        __nv_bfloat16* const dst = prm.inter + row0 * pitch + f;
        // Two rows at a time: the lanes of columns f and f + 1 (F is even) swap one, so that each stores two columns of one row.
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          if ((4 * i + h) * 16 >= rows) continue;
          __nv_bfloat16* to = dst + (size_t)((4 * i + h) * 16 + (up ? 8 : 0) + (odd ? 1 : 0)) * pitch - (odd ? 1 : 0);
#pragma unroll
          for (int j = 0; j < 8; j += 2, to += 2 * pitch) {  // a lane that holds gates takes rows 0-7 of the unit, one that holds ups 8-15
            float v[2];
#pragma unroll
            for (int n = 0; n < 2; ++n) {
              const float got = __shfl_xor_sync(0xffffffffu, up ? acc(i, j + n) : acc(i, j + n + 8), 16);
              const float g = up ? got : acc(i, j + n), u = up ? acc(i, j + n + 8) : got;
              const float s = g / (1.0f + expf(-g)) * u;
              v[n] = s * group_scale(large >> (4 * i) & 1);
              if (!(fabsf(v[n]) <= kNearTop))  // (g or u not finite: v is not either; finite both, and their product: too large for the parts)
                if (!is_finite(g) || !is_finite(u) || is_finite(s)) bad |= 1u << (16 * i + j + n);
            }
            uint32_t part[3];
            split_pair(v[0], v[1], part[0], part[1], part[2]);
            const int r = (4 * i + h) * 16 + j + (up ? 8 : 0) + (odd ? 1 : 0);
#pragma unroll
            for (int n = 0; n < 3; ++n) {
              const uint32_t other = __shfl_xor_sync(0xffffffffu, part[n], 1);
              if (f < F && r < rows) *reinterpret_cast<uint32_t*>(to + n * plane) = __byte_perm(part[n], other, odd ? 0x3276u : 0x5410u);
            }
          }
        }
        __syncwarp();
        if (__any_sync(0xffffffffu, bad != 0)) {
          const float* w = (up ? prm.wu : prm.wg) + ((size_t)it.e * F + min(f, F - 1)) * H;
          bad = f < F ? (up ? bad << 8 : bad) & exist() : 0u;
          bad = unexplained(Explain{prm.recv_planes + (row0 + h * 16) * prm.recv_pitch, w, prm.recv_pitch, H, true}, bad);
        }
        for (; bad != 0; bad &= bad - 1) {
          const int at = __ffs(bad) - 1, r = (4 * (at >> 4) + h) * 16 + (at & 15);
          const float* a = prm.recv + (row0 + r) * H;
          const size_t w = ((size_t)it.e * F + f) * H;
          const float g = fp32_chain(a, prm.wg + w, H), u = fp32_chain(a, prm.wu + w, H);
          store_top(g / (1.0f + expf(-g)) * u, group_scale(large >> (4 * (at >> 4)) & 1), dst + r * pitch, plane);
        }
        __syncwarp();
        // This warp's part of the block is written: make it visible (also to the async proxy, which is how the GEMM2
        // producer will read it) and bump the tile's status counter.
        asm volatile("fence.proxy.async.global;" ::: "memory");
        __threadfence();
        __syncwarp();
        if (lane == 0) asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(prm.gemm1_done + it.tile) : "memory");
      } else {
        const int hc = it.nb * 128 + q * 32 + lane;
        float* const dst = prm.out + row0 * H + hc;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const int r = (4 * i + h) * 16 + j;
            if (r < rows && hc < H) {
              dst[(size_t)r * H] = acc(i, j);
              if (!is_finite(acc(i, j))) bad |= 1u << (16 * i + j);
            }
          }
        }
        if (__any_sync(0xffffffffu, bad != 0)) {
          ld_acquire(&prm.gemm1_done[it.tile]);  // (complete, or the MMAs would not have had it: these loads come behind it too)
          const float* w = prm.wd + ((size_t)(it.e / prm.tp) * H + min(hc, H - 1)) * F * prm.tp + (size_t)(it.e % prm.tp) * F;
          bad = unexplained(Explain{prm.inter + (row0 + h * 16) * prm.inter_pitch, w, prm.inter_pitch, F, false}, bad);
        }
        for (; bad != 0; bad &= bad - 1) {
          const int at = __ffs(bad) - 1, r = (4 * (at >> 4) + h) * 16 + (at & 15);
          dst[(size_t)r * H] = fp32_chain_planes(prm.inter + (row0 + r) * prm.inter_pitch, plane, 1.0f / group_scale(large >> (4 * (at >> 4)) & 1),
                                                 prm.wd + ((size_t)(it.e / prm.tp) * H + hc) * F * prm.tp + (size_t)(it.e % prm.tp) * F, F);
        }
        __syncwarp();
      }
    }
    if (fail_site) sh->abort_flag = 1;
  }
  if (fail_site) set_status(prm.status, MOE_ERR_TIMEOUT, fail_site);

  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (sh->abort_flag) {
    // Whichever role gave up, copies and MMAs that others had issued may still be in flight: all of them end (bounded waits)
    // before the CTA gives up shared and tensor memory.
    auto settle = [&](unsigned long long* bar, uint32_t parity) {
      const unsigned long long t0 = globaltimer();
      while (!mbar_try(smem_u32(bar), parity))
        if (globaltimer() - t0 > wait_ns + 1000000ull) break;
    };
    if (warp == 1) {
      if (elect_one()) {
        tc_commit(smem_u32(&sh->drain));  // (the elected lane is the same every time: it is the one whose MMAs this follows)
        settle(&sh->drain, 0u);
      }
      __syncwarp();
    }
    if (threadIdx.x == 0) {
      for (int g = max(0, sh->w_fills - kSpWStages); g < sh->w_fills; ++g) settle(&sh->w_full[g % kSpWStages], (uint32_t)(g / kSpWStages) & 1u);
      for (int s = 0; s < kSpBStages; ++s)
        if (sh->b_fills[s] > 0) settle(&sh->b_full[s], (sh->b_fills[s] - 1) & 1u);
    }
    __syncthreads();
  }
  pdl_trigger();
  if (threadIdx.x == 0) {  // the last CTA to leave puts the counters back to zero (see ffn_tc_kernel)
    int* exit_counter = prm.work_counter + 2;
    const bool last = atomicAdd(exit_counter, 1) == (int)gridDim.x - 1;
    if (last) {
      *prm.work_counter = 0;
      *exit_counter = 0;
    }
    sh->last_cta = last ? 1 : 0;
  }
  __syncthreads();
  if (sh->last_cta)
    for (int pt = threadIdx.x; pt < prm.P; pt += kSpThreads) prm.gemm1_done[pt] = 0;
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

// ---- host side ------------------------------------------------------------------------------
static int make_map(EncodeTiledFn enc, CUtensorMap* m, CUtensorMapDataType type, const void* base, int rank, const cuuint64_t* dims,
                    const cuuint64_t* strides, const cuuint32_t* box) {
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  return enc(m, type, (cuuint32_t)rank, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
             CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS
             ? MOE_OK : MOE_ERR_CUDA;
}

int split_pitch(int n) { return (n + 7) / 8 * 8; }  // of a plane's rows: 16 bytes

// Where the plain FMAs of ffn_fp32_kernel are the slower ones: experts of some rows, and either a fair amount of work (below,
// both are a chain of launches and this one has one more to start up) or sums so long that the FMAs have too few CTAs for
// their GEMM2.  Measured, whole layer, this / FMAs, work = rows x H x F: up to 16 experts, H from 384, 24 to 40 M 0.79-0.97 (H 912 with
// 4 experts 1.00-1.04), 40 to 50 M 0.80-0.86; H 128 to 256 24 to 34 M 0.96-1.21, 39 to 51 M 0.88-1.01; 32 experts 51 M (256 x 200)
// 1.15, 80 M (448 x 400) 1.05, 92 M 0.88.  us, FMAs / this: 375 M (412 x 508, 32 experts) 117 / 69, 1677 M (444 x 1568) 425 / 136, 4194 M (T
// 1000, 1024 x 2048, 16 experts) 737 / 217.  Long sums: 22 M (92 x 1216) 88 / 50, 8 M (148 x 1432) 62 / 50.  Few rows per expert, where both stream weights and this splits all of them, the more experts the
// worse.  This over FMAs at 8 / 12 / 16 / 24 rows per expert, six shapes each (512 x 1024, 1024 x 2048, 448 x 400, 928 x 556, 1024 x
// 512; last 256 x 2048, whose short sums have the most items for their work): 8 and 16 experts 0.65-0.92 / 0.67-0.91 / 0.60-0.85 / 0.59-0.93;
// 32 experts 0.92-1.11 / 0.86-1.12 / 0.68-0.88, 0.74; 64 1.09-1.28 / 0.83-1.15 / 0.75-0.92, 0.85; 128 1.17-1.42 / 0.95-1.18 / 0.79-0.99, 1.12
// / 0.62-0.86, 0.96; 256 1.26-1.58 / 0.97-1.19 / 0.83-1.04, 1.58 / 0.60-0.77, 1.17, at 32 rows 0.49-0.63, 0.93.
// The planes take 6 bytes per element of the pool and of the intermediate, which alone takes 4 with the FMAs: T 8192, H 4096, 8 experts,
// top-2, F 14336 3.0 GB of workspace instead of 2.1.  Static regions, whose pool is not bounded by the rows, keep the FMAs (T 4096, H
// 4096, 64 experts, top-2, F 2048 would hold 18.5 GB instead of 11.0).
// (Calls with and without row counts go the same way, so their rows are the same bytes.)
bool ffn_split_applies(const moe_config_t& c, int64_t P) {
  const long long rows = (long long)c.T * c.K, items = (long long)P * ((c.F + 63) / 64 + (c.H + 127) / 128);
  if (c.dtype != MOE_DTYPE_FP32 || c.identity_experts || c.ffn_kernel == 1) return false;
  if (P > kMaxListTiles || items >= (1ll << kSpRowShift)) return false;  // the work list, the item ring's fields
  if (P > rows / kTileRows + c.E) return false;  // static regions of more tiles than the batch's rows fill: planes of all of them
  const int few = c.E <= 16 ? 8 : c.E > 64 && c.H < 384 ? 32 : 16;  // rows per expert from which on the tensor cores are the faster ones
  const long long work = c.E > 16 ? 90000000ll : c.H >= 384 ? 24000000ll : 40000000ll;
  return rows >= (long long)few * c.E && (rows * c.H * c.F >= work || c.F >= 900);
}

int launch_ffn_split(moe_plan* p, const void* recv, const int* tile_expert, const void* wg, const void* wu, const void* wd,
                     void* out_rows, const int* tile_count, const int* rows_done, cudaStream_t st) {
  const moe_config_t& c = p->cfg;
  EncodeTiledFn enc;
  int rc = get_encoder(p, &enc);
  if (rc != MOE_OK) return rc;
  const cuuint64_t pool = (cuuint64_t)p->P * kTileRows, E = (cuuint64_t)c.E, F = (cuuint64_t)c.F, H = (cuuint64_t)c.H, tp = (cuuint64_t)p->tp;
  SplitMaps maps;
  {
    const cuuint64_t dims[3] = {H, F, E}, str[2] = {H * 4, F * H * 4};  // a TP shard's gate / up rows are contiguous
    const cuuint32_t box[3] = {32, 64, 1};
    if ((rc = make_map(enc, &maps.wg, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, wg, 3, dims, str, box)) != MOE_OK) return rc;
    if ((rc = make_map(enc, &maps.wu, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, wu, 3, dims, str, box)) != MOE_OK) return rc;
    const cuuint64_t ddims[4] = {F, H, tp, E / tp}, dstr[3] = {F * tp * 4, F * 4, H * F * tp * 4};
    const cuuint32_t dbox[4] = {32, 128, 1, 1};
    if ((rc = make_map(enc, &maps.wd, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, wd, 4, ddims, dstr, dbox)) != MOE_OK) return rc;
  }
  const cuuint64_t hp = (cuuint64_t)split_pitch(c.H), fp = (cuuint64_t)split_pitch(c.F);
  for (int q = 0; q < 4; ++q) {
    const cuuint32_t box[3] = {(cuuint32_t)kBK, (cuuint32_t)(kTileRows >> q), 3};
    const cuuint64_t d1[3] = {H, pool, 3}, s1[2] = {hp * 2, pool * hp * 2}, d2[3] = {F, pool, 3}, s2[2] = {fp * 2, pool * fp * 2};
    if ((rc = make_map(enc, &maps.rows[0][q], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, p->s.recv_planes, 3, d1, s1, box)) != MOE_OK) return rc;
    if ((rc = make_map(enc, &maps.rows[1][q], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, p->s.inter, 3, d2, s2, box)) != MOE_OK) return rc;
  }
  SplitParams q;
  q.tile_expert = tile_expert;
  q.tile_count = tile_count;
  q.rows_done = rows_done;
  q.total_rows = c.T * c.K;
  q.P = (int)p->P;
  q.E = c.E;
  q.F = c.F;
  q.H = c.H;
  q.tp = p->tp;
  q.recv = (const float*)recv;
  q.recv_planes = (const __nv_bfloat16*)p->s.recv_planes;
  q.recv_pitch = (int)hp;
  q.group_large = (const uint2*)p->s.group_large;
  q.wg = (const float*)wg;
  q.wu = (const float*)wu;
  q.wd = (const float*)wd;
  q.inter = (__nv_bfloat16*)p->s.inter;
  q.inter_pitch = (int)fp;
  q.out = (float*)out_rows;
  q.gemm1_done = p->s.gemm1_done;
  q.work_counter = p->s.gemm1_done + p->P;
  q.wait_ns = c.wait_limit_ns ? c.wait_limit_ns : kDefaultWaitNs;
  q.status = p->s.status;
  const int grid = p->sm_count;
  q.lag = grid;
  mark(p, 3, st);
  if (launch_pdl(split_rows_kernel, dim3((unsigned)(p->P * (kTileRows / kSplitRows))), dim3(256), 0, st, (const float*)recv, tile_expert,
                 tile_count, rows_done, q.total_rows, c.E, c.H, (int)hp, (size_t)pool * hp, (__nv_bfloat16*)p->s.recv_planes, p->s.group_large) != cudaSuccess)
    return MOE_ERR_CUDA;
  static SmemAttrOnce once;
  if (ensure_dynamic_smem(ffn_split_kernel, kSpSmem, p->device, once) != cudaSuccess) return MOE_ERR_CUDA;
  p->launches += 2;
  if (launch_pdl(ffn_split_kernel, dim3(grid), dim3(kSpThreads), kSpSmem, st, maps, q) != cudaSuccess) return MOE_ERR_CUDA;
  mark(p, 4, st);
  return cudaGetLastError() == cudaSuccess ? 0 : MOE_ERR_CUDA;
}

}  // namespace moehub
