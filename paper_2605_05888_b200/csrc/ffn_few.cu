// Step 3 of the MoE layer (paper Section II-A, expert computation) for a handful of tokens in bf16: decoding.
//
// Bound by reading the picked experts' weights once.  The tensor-core kernels hand out blocks of 128 or 256 weight rows
// per CTA, which leaves most SMs without work when few experts have rows (one Qwen-like token: 44 blocks for 148 SMs,
// each streamed by one CTA at the latency of its own four stages).  Here a warp owns one column of the result (gate and
// up row of it, or a row of the down matrix), reads it in 16-byte vectors, eight loads in flight per lane, and forms the
// dot products with all of the expert's rows (at most R, which come from L1) on plain fp32 FMAs; CTAs walk the columns
// of one tile with a stride, so the work spreads over all SMs whatever the number of experts.
// Measured, layer time, us, before / now: one Qwen-like token 57.7 / 41.3, one Mixtral-like 209.6 / 140 (705 MB of weights:
// 109 at the copy rate), one DeepSeek-like 187 / 152; the rule in launch_ffn_tc has more.
#include "tc_common.cuh"
#include "route_common.cuh"

namespace moehub {

constexpr int kFewThreads = 256;
constexpr int kFewWarps = kFewThreads / 32;
constexpr int kFewUnroll = 4;  // 16-byte vectors per lane, matrix and pass

struct FewParams {
  const __nv_bfloat16* A;  // [P * 128, Kd]
  const __nv_bfloat16* b1;
  const __nv_bfloat16* b2;
  size_t expert_stride, shard_offset;  // elements between experts, between an expert's TP shards
  int tp, ldb, N, Kd;
  __nv_bfloat16* C;        // [P * 128, N], or the staging rows of the push-style combine
  const int* push_src;
  const int* tile_expert;
  int P, E;
  const int* tile_count;
  const int* rows_done;
  int total_rows;
  unsigned long long wait_ns;
  int* status;
};

// The columns of one tile, for at most R of its rows: those past `rows` are multiplied too (they are in the pool) and
// not stored.
template <int R, bool SWIGLU>
__device__ __forceinline__ void few_columns(const FewParams& p, const __nv_bfloat16* __restrict__ a, size_t base, int tile, int rows) {
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  for (int n = blockIdx.x * kFewWarps + warp; n < p.N; n += gridDim.x * kFewWarps) {
    const __nv_bfloat16* w1 = p.b1 + base + (size_t)n * p.ldb;
    const __nv_bfloat16* w2 = SWIGLU ? p.b2 + base + (size_t)n * p.ldb : nullptr;
    float acc1[R], acc2[SWIGLU ? R : 1];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      acc1[r] = 0.0f;
      if (SWIGLU) acc2[r] = 0.0f;
    }
    for (int k0 = lane * 8; k0 < p.Kd; k0 += 256 * kFewUnroll) {
      uint4 v1[kFewUnroll], v2[SWIGLU ? kFewUnroll : 1];
#pragma unroll
      for (int i = 0; i < kFewUnroll; ++i) {
        const int k = k0 + 256 * i;
        v1[i] = make_uint4(0, 0, 0, 0);
        if (k < p.Kd) v1[i] = __ldcs(reinterpret_cast<const uint4*>(w1 + k));
        if (SWIGLU) {
          v2[i] = make_uint4(0, 0, 0, 0);
          if (k < p.Kd) v2[i] = __ldcs(reinterpret_cast<const uint4*>(w2 + k));
        }
      }
#pragma unroll
      for (int i = 0; i < kFewUnroll; ++i) {
        const int k = k0 + 256 * i;
        if (k >= p.Kd) break;
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const uint4 x = *reinterpret_cast<const uint4*>(a + (size_t)r * p.Kd + k);
          const uint32_t xw[4] = {x.x, x.y, x.z, x.w};
          const uint32_t g[4] = {v1[i].x, v1[i].y, v1[i].z, v1[i].w};
#pragma unroll
          for (int q = 0; q < 4; ++q) acc1[r] = fma_bf16_hi(xw[q], g[q], fma_bf16_lo(xw[q], g[q], acc1[r]));
          if (SWIGLU) {
            const uint32_t u[4] = {v2[i].x, v2[i].y, v2[i].z, v2[i].w};
#pragma unroll
            for (int q = 0; q < 4; ++q) acc2[r] = fma_bf16_hi(xw[q], u[q], fma_bf16_lo(xw[q], u[q], acc2[r]));
          }
        }
      }
    }
    float mine = 0.0f;  // lane r: row r
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const float s1 = group_sum<32>(acc1[r]);
      const float s2 = SWIGLU ? group_sum<32>(acc2[r]) : 0.0f;
      if (lane == r) mine = SWIGLU ? silu_mul(s1, s2) : s1;
    }
    if (lane < rows) {
      long long row = (long long)tile * kTileRows + lane;
      if (!SWIGLU && p.push_src != nullptr) {  // push-style combine: to the token's own position
        row = __ldcg(p.push_src + row);
        if (row >= p.total_rows) row = -1;
      }
      if (row >= 0) p.C[(size_t)row * p.N + n] = __float2bfloat16_rn(mine);
    }
  }
}

template <int R, bool SWIGLU>
__global__ void __launch_bounds__(kFewThreads)
ffn_few_kernel(const FewParams p) {
  __shared__ int s_used[kFewWarps];
  __shared__ int s_tile, s_rows;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  if (threadIdx.x == 0) s_tile = -1;
  __syncthreads();
  pdl_wait();
  pdl_trigger();
  // this CTA's tile: number blockIdx.y among the used ones
  const int ordinal = blockIdx.y;
  for (int base = 0, seen = 0; base < p.P && seen <= ordinal; base += kFewThreads) {
    const int t = base + threadIdx.x;
    const int e = t < p.P ? p.tile_expert[t] : -1;
    const unsigned used = __ballot_sync(0xffffffffu, e >= 0 && e < p.E);
    if (lane == 0) s_used[warp] = __popc(used);
    __syncthreads();
    int before = seen;
    for (int w = 0; w < kFewWarps; ++w) {
      if (w < warp) before += s_used[w];
      seen += s_used[w];
    }
    if (((used >> lane) & 1u) && before + __popc(used & ((1u << lane) - 1u)) == ordinal) s_tile = t;
    __syncthreads();
  }
  const int tile = s_tile;
  if (tile < 0) return;
  if (threadIdx.x == 0) {  // availability of the tile's rows (Section IV-D): as in the tensor-core kernels, bounded
    const unsigned long long t0 = globaltimer();
    bool ready = true;
    while (ld_acquire(&p.tile_count[tile]) < kTileRows && ld_acquire(p.rows_done) < p.total_rows) {
      if (globaltimer() - t0 > p.wait_ns) {
        set_status(p.status, MOE_ERR_TIMEOUT, kWaitTileReady);
        ready = false;
        break;
      }
      __nanosleep(64);
    }
    s_rows = ready ? min(R, p.tile_count[tile]) : 0;
  }
  __syncthreads();
  const int rows = s_rows;
  if (rows <= 0) return;
  const int e = p.tile_expert[tile];
  const size_t base = (size_t)(e / p.tp) * p.expert_stride + (size_t)(e % p.tp) * p.shard_offset;
  const __nv_bfloat16* a = p.A + (size_t)tile * kTileRows * p.Kd;
  if (rows == 1) few_columns<1, SWIGLU>(p, a, base, tile, rows);
  else if (R >= 2 && rows == 2) few_columns<(R < 2 ? R : 2), SWIGLU>(p, a, base, tile, rows);
  else if (R >= 4 && rows <= 4) few_columns<(R < 4 ? R : 4), SWIGLU>(p, a, base, tile, rows);
  else few_columns<R, SWIGLU>(p, a, base, tile, rows);
}

template <int R>
static int launch_few(moe_plan* p, FewParams q, const void* recv, const void* wg, const void* wu, const void* wd, void* out,
                      const int* push_src, cudaStream_t st) {
  const moe_config_t& c = p->cfg;
  const int tiles = (int)min((long long)c.T * c.K, (long long)p->P);  // at most this many are used
  const int sms = p->sm_count > 0 ? p->sm_count : 148;
  const int per_tile = max(1, (8 * sms + tiles - 1) / tiles);          // CTAs per tile: up to eight per SM in all
  q.expert_stride = (size_t)c.F * p->tp * c.H;
  q.A = (const __nv_bfloat16*)recv;
  q.b1 = (const __nv_bfloat16*)wg;
  q.b2 = (const __nv_bfloat16*)wu;
  q.shard_offset = (size_t)c.F * c.H;
  q.ldb = c.H;
  q.N = c.F;
  q.Kd = c.H;
  q.C = (__nv_bfloat16*)p->s.inter;
  q.push_src = nullptr;
  const int g1 = min(per_tile, (c.F + kFewWarps - 1) / kFewWarps), g2 = min(per_tile, (c.H + kFewWarps - 1) / kFewWarps);
  if (launch_pdl(ffn_few_kernel<R, true>, dim3(g1, tiles), dim3(kFewThreads), 0, st, q) != cudaSuccess) return MOE_ERR_CUDA;
  mark(p, 4, st);
  q.A = (const __nv_bfloat16*)p->s.inter;
  q.b1 = (const __nv_bfloat16*)wd;
  q.b2 = nullptr;
  q.shard_offset = (size_t)c.F;
  q.ldb = c.F * p->tp;
  q.N = c.H;
  q.Kd = c.F;
  q.C = (__nv_bfloat16*)out;
  q.push_src = push_src;
  if (launch_pdl(ffn_few_kernel<R, false>, dim3(g2, tiles), dim3(kFewThreads), 0, st, q) != cudaSuccess) return MOE_ERR_CUDA;
  p->launches += 2;
  return 0;
}

int launch_ffn_few(moe_plan* p, const void* recv, const void* wg, const void* wu, const void* wd, const FfnParams& prm,
                   const int* push_src, cudaStream_t st) {
  FewParams q = {};
  q.tp = p->tp;
  q.tile_expert = prm.tile_expert;
  q.P = prm.P;
  q.E = prm.E;
  q.tile_count = prm.tile_count;
  q.rows_done = prm.rows_done;
  q.total_rows = prm.total_rows;
  q.wait_ns = prm.wait_ns;
  q.status = prm.status;
  const int T = p->cfg.T;
  if (T <= 1) return launch_few<1>(p, q, recv, wg, wu, wd, prm.out, push_src, st);
  if (T <= 2) return launch_few<2>(p, q, recv, wg, wu, wd, prm.out, push_src, st);
  if (T <= 4) return launch_few<4>(p, q, recv, wg, wu, wd, prm.out, push_src, st);
  return launch_few<8>(p, q, recv, wg, wu, wd, prm.out, push_src, st);
}

}  // namespace moehub
