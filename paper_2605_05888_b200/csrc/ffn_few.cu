// Step 3 of the MoE layer (paper Section II-A, expert computation) for a handful of tokens in bf16 (decoding), and for
// small layers of some tens of tokens.
//
// Bound by reading the picked experts' weights once.  The tensor-core kernels hand out blocks of 128 or 256 weight rows
// per CTA, which leaves most SMs without work when few experts have rows (one Qwen-like token: 44 blocks for 148 SMs,
// each streamed by one CTA at the latency of its own four stages).  Here a warp owns one column of the result (gate and
// up row of it, or a row of the down matrix), reads it in 16-byte vectors, eight loads in flight per lane, and forms the
// dot products with all of the expert's rows (at most R, which come from L1) on plain fp32 FMAs; CTAs walk the columns
// of one tile with a stride, so the work spreads over all SMs whatever the number of experts.
// Measured, layer time, us, tensor-core kernels / this / with dispatch and combine taken in (second half of the file): one
// Qwen-like token 57.7 / 41.3 / 31, one Mixtral-like 209.6 / 140 / 125 (705 MB of weights: 109 at the copy rate), one
// DeepSeek-like 187 / 152 / 147; the rule at few_applies has more.
#include "tc_common.cuh"
#include "route_common.cuh"

namespace moehub {

constexpr int kFewThreads = 256;
constexpr int kFewWarps = kFewThreads / 32;
constexpr int kFewAssign = 256;  // most assignments (token, k): a thread per assignment
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

// One column of the result for R rows, a + off[r]: lane r returns row r's value (gate and up rows w1, w2: the activated
// product).
template <int R, bool SWIGLU>
__device__ __forceinline__ float few_dots(const __nv_bfloat16* __restrict__ w1, const __nv_bfloat16* __restrict__ w2,
                                          const __nv_bfloat16* a, const int (&off)[R], int Kd) {
  const int lane = threadIdx.x % 32;
  float acc1[R], acc2[SWIGLU ? R : 1];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    acc1[r] = 0.0f;
    if (SWIGLU) acc2[r] = 0.0f;
  }
  for (int k0 = lane * 8; k0 < Kd; k0 += 256 * kFewUnroll) {
    uint4 v1[kFewUnroll], v2[SWIGLU ? kFewUnroll : 1];
#pragma unroll
    for (int i = 0; i < kFewUnroll; ++i) {
      const int k = k0 + 256 * i;
      v1[i] = make_uint4(0, 0, 0, 0);
      if (k < Kd) v1[i] = __ldcs(reinterpret_cast<const uint4*>(w1 + k));
      if (SWIGLU) {
        v2[i] = make_uint4(0, 0, 0, 0);
        if (k < Kd) v2[i] = __ldcs(reinterpret_cast<const uint4*>(w2 + k));
      }
    }
#pragma unroll
    for (int i = 0; i < kFewUnroll; ++i) {
      const int k = k0 + 256 * i;
      if (k >= Kd) break;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const uint4 x = *reinterpret_cast<const uint4*>(a + off[r] + k);
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
  float mine = 0.0f;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const float s1 = group_sum<32>(acc1[r]);
    const float s2 = SWIGLU ? group_sum<32>(acc2[r]) : 0.0f;
    if (lane == r) mine = SWIGLU ? silu_mul(s1, s2) : s1;
  }
  return mine;
}

// The columns of one tile, for `rows` (at most R) of its rows from r0 on: those past them are multiplied too (the tile
// has them) and not stored.
template <int R, bool SWIGLU>
__device__ __forceinline__ void few_columns(const FewParams& p, size_t base, int tile, int r0, int rows) {
  const __nv_bfloat16* a = p.A + ((size_t)tile * kTileRows + r0) * p.Kd;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  int off[R];
#pragma unroll
  for (int r = 0; r < R; ++r) off[r] = r * p.Kd;
  for (int n = blockIdx.x * kFewWarps + warp; n < p.N; n += gridDim.x * kFewWarps) {
    const float mine = few_dots<R, SWIGLU>(p.b1 + base + (size_t)n * p.ldb, SWIGLU ? p.b2 + base + (size_t)n * p.ldb : nullptr, a, off, p.Kd);
    if (lane < rows) {
      long long row = (long long)tile * kTileRows + r0 + lane;
      if (!SWIGLU && p.push_src != nullptr) {  // push-style combine: to the token's own position
        row = __ldcg(p.push_src + row);
        if (row >= p.total_rows) row = -1;
      }
      if (row >= 0) p.C[(size_t)row * p.N + n] = __float2bfloat16_rn(mine);
    }
  }
}

struct FewTile {  // shared memory
  int used[kFewWarps];
  int tile, rows, owned;
};

// The tile that is number `ordinal` among the owned ones (-1: there are not so many).  The whole CTA calls.
__device__ __forceinline__ int few_find_tile(const FewParams& p, FewTile& s, int ordinal) {
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  int seen = 0;
  for (int base = 0; base < p.P; base += kFewThreads) {
    const int t = base + threadIdx.x;
    const int e = t < p.P ? p.tile_expert[t] : -1;
    const unsigned used = __ballot_sync(0xffffffffu, e >= 0 && e < p.E);
    if (lane == 0) s.used[warp] = __popc(used);
    __syncthreads();
    int before = seen;
    for (int w = 0; w < kFewWarps; ++w) {
      if (w < warp) before += s.used[w];
      seen += s.used[w];
    }
    if (((used >> lane) & 1u) && before + __popc(used & ((1u << lane) - 1u)) == ordinal) s.tile = t;
    __syncthreads();
  }
  if (threadIdx.x == 0) s.owned = seen;
  return s.tile;
}

// How many rows the tile holds, once they are available (Section IV-D; as in the tensor-core kernels, bounded: -1 when the
// wait ran out).  The whole CTA calls.
__device__ __forceinline__ int few_tile_rows(const FewParams& p, FewTile& s, int tile) {
  if (threadIdx.x == 0) {
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
    s.rows = ready ? min(kTileRows, p.tile_count[tile]) : -1;
  }
  __syncthreads();
  return s.rows;
}

__device__ __forceinline__ size_t few_weights(const FewParams& p, int tile) {
  const int e = p.tile_expert[tile];
  return (size_t)(e / p.tp) * p.expert_stride + (size_t)(e % p.tp) * p.shard_offset;
}

// The owned tiles beyond the first gridDim.y: what a dispatch leaves owns at most T * K tiles, one per blockIdx.y, but a
// caller's own table may name an owner for every tile of its regions.  Row by row and not inlined, so that the kernel's body
// keeps its registers.  Measured on moe_expert_ffn, one to five tokens, four shapes, against the kernel that looks at the first
// gridDim.y only: 0.90 to 1.07 of its time, mean 1.01; moe_layer, whose table is a dispatch's, has that kernel.
template <bool SWIGLU>
__device__ __noinline__ void few_more_tiles(const FewParams& p, FewTile& s) {
  for (int ordinal = blockIdx.y + gridDim.y;; ordinal += gridDim.y) {
    __syncthreads();
    if (threadIdx.x == 0) s.tile = -1;
    __syncthreads();
    const int tile = few_find_tile(p, s, ordinal);
    if (tile < 0) return;
    const int rows = few_tile_rows(p, s, tile);
    if (rows < 0) return;
    const size_t base = few_weights(p, tile);
    for (int r0 = 0; r0 < rows; ++r0) few_columns<1, SWIGLU>(p, base, tile, r0, 1);
  }
}

// ANY: the table may be any caller's (false: a dispatch's).
template <int R, bool SWIGLU, bool ANY>
__device__ __forceinline__ void few_tiles(const FewParams& p) {
  __shared__ FewTile s;
  if (threadIdx.x == 0) s.tile = -1;
  __syncthreads();
  pdl_wait();
  pdl_trigger();
  const int tile = few_find_tile(p, s, blockIdx.y);
  if (tile < 0) return;
  const int rows = few_tile_rows(p, s, tile);
  if (rows < 0 || (!ANY && rows == 0)) return;
  if (!ANY || rows > 0) {
    const size_t base = few_weights(p, tile);
    if (rows == 1) few_columns<1, SWIGLU>(p, base, tile, 0, rows);
    else if (R >= 2 && rows == 2) few_columns<(R < 2 ? R : 2), SWIGLU>(p, base, tile, 0, rows);
    else if (R >= 4 && rows <= 4) few_columns<(R < 4 ? R : 4), SWIGLU>(p, base, tile, 0, rows);
    else few_columns<R, SWIGLU>(p, base, tile, 0, min(rows, R));
    for (int r0 = R; r0 < rows;) {  // more rows than tokens: a caller's routing that names an expert twice for a token
      const int n = R < 8 || rows - r0 < 8 ? 1 : 8;  // (or more than 8 tokens)
      if (n == 1) few_columns<1, SWIGLU>(p, base, tile, r0, 1);
      else few_columns<(R < 8 ? 1 : 8), SWIGLU>(p, base, tile, r0, 8);
      r0 += n;
    }
  }
  if (ANY && (int)(blockIdx.y + gridDim.y) < s.owned) few_more_tiles<SWIGLU>(p, s);
}

template <int R, bool SWIGLU>
__global__ void __launch_bounds__(kFewThreads)
ffn_few_kernel(const FewParams p) {
  few_tiles<R, SWIGLU, false>(p);
}
template <int R, bool SWIGLU>
__global__ void __launch_bounds__(kFewThreads)
ffn_few_any_kernel(const __grid_constant__ FewParams p) {
  few_tiles<R, SWIGLU, true>(p);
}

static dim3 few_grid(const moe_plan* p, int tiles, int columns) {  // CTAs per tile: up to eight per SM in all
  const int sms = p->sm_count > 0 ? p->sm_count : 148;
  return dim3(max(1, min((8 * sms + tiles - 1) / tiles, (columns + kFewWarps - 1) / kFewWarps)), tiles);
}

// Up to five tokens: measured, layer time tensor cores / plain FMAs (four and five launches, without what the second half
// of the file saves): one token 1.23 (256 experts of 88 MB) to 1.81 (32 of 6 MB), five 1.03-1.21, six 0.93-1.22, eight
// 0.92-1.11 (an expert's rows share a weight's load but not its FMAs).
// More tokens while the layer is so small that launches and latencies are what it costs, by the number of dot products;
// measured, layer time, us, tensor cores / plain FMAs with three launches: H 256, F 256, K 2: T 8 28.8 / 13.3, T 32 28.8 /
// 16.8 (49 thousand); H 512, F 512, K 2: T 16 32.9 / 23.6 (49), T 32 32.9 / 30.0 (98); H 1024, F 512, K 2: T 16 39.1 / 29.6
// (66), T 32 39.1 / 39.3 (131); H 512, F 512, K 4, 32 experts: T 8 35.0 / 30.0 (49), T 12 35.5 / 36.3 (74); H 512, F 256, K 8,
// 64 experts: T 8 41.2 / 37.1 (66), T 12 40.8 / 46.5 (98).
constexpr long long kFewDots = 65536;
bool few_applies(const moe_plan* p) {
  const moe_config_t& c = p->cfg;
  const long long dots = (long long)c.T * c.K * (c.H + 2ll * c.F);
  return c.ffn_kernel == 0 && (c.T <= 5 || (c.T <= kFewMaxTokens && c.T * c.K <= kFewAssign && dots <= kFewDots)) && c.H >= 256 && c.F >= 256 && c.ffn_hot_min_tiles <= 0 && c.ffn_thin_tiles >= 0 &&
         c.ffn_split == 0 && !p->trace;
}

template <int R, bool ANY>
static int launch_few_gate_up(moe_plan* p, FewParams q, const void* recv, const void* wg, const void* wu, cudaStream_t st) {
  const moe_config_t& c = p->cfg;
  q.expert_stride = (size_t)c.F * p->tp * c.H;
  q.A = (const __nv_bfloat16*)recv;
  q.b1 = (const __nv_bfloat16*)wg;
  q.b2 = (const __nv_bfloat16*)wu;
  q.shard_offset = (size_t)c.F * c.H;
  q.ldb = c.H;
  q.N = c.F;
  q.Kd = c.H;
  q.C = (__nv_bfloat16*)p->s.inter;
  p->launches += 1;
  return launch_pdl(ANY ? ffn_few_any_kernel<R, true> : ffn_few_kernel<R, true>, few_grid(p, (int)min((long long)c.T * c.K, (long long)p->P), c.F), dim3(kFewThreads), 0, st, q) == cudaSuccess ? 0 : MOE_ERR_CUDA;
}

template <int R, bool ANY>
static int launch_few_down(moe_plan* p, FewParams q, const void* wd, void* out, const int* push_src, cudaStream_t st) {
  const moe_config_t& c = p->cfg;
  q.expert_stride = (size_t)c.F * p->tp * c.H;
  q.A = (const __nv_bfloat16*)p->s.inter;
  q.b1 = (const __nv_bfloat16*)wd;
  q.shard_offset = (size_t)c.F;
  q.ldb = c.F * p->tp;
  q.N = c.H;
  q.Kd = c.F;
  q.C = (__nv_bfloat16*)out;
  q.push_src = push_src;
  p->launches += 1;
  return launch_pdl(ANY ? ffn_few_any_kernel<R, false> : ffn_few_kernel<R, false>, few_grid(p, (int)min((long long)c.T * c.K, (long long)p->P), c.H), dim3(kFewThreads), 0, st, q) == cudaSuccess ? 0 : MOE_ERR_CUDA;
}

template <int R, bool ANY>
static int launch_few(moe_plan* p, const FewParams& q, const void* recv, const void* wg, const void* wu, const void* wd, void* out,
                      const int* push_src, cudaStream_t st) {
  int rc = launch_few_gate_up<R, ANY>(p, q, recv, wg, wu, st);
  if (rc != 0) return rc;
  mark(p, 4, st);
  return launch_few_down<R, ANY>(p, q, wd, out, push_src, st);
}

int launch_ffn_few(moe_plan* p, const void* recv, const void* wg, const void* wu, const void* wd, const FfnParams& prm,
                   const int* push_src, cudaStream_t st, bool own) {
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
#define MOEHUB_FEW(R) (own ? launch_few<R, false>(p, q, recv, wg, wu, wd, prm.out, push_src, st) : launch_few<R, true>(p, q, recv, wg, wu, wd, prm.out, push_src, st))
  if (T <= 1) return MOEHUB_FEW(1);
  if (T <= 2) return MOEHUB_FEW(2);
  if (T <= 4) return MOEHUB_FEW(4);
  if (T <= 5) return MOEHUB_FEW(5);
  return MOEHUB_FEW(8);
#undef MOEHUB_FEW
}

// ---- the whole layer behind the router ----------------------------------------------------------------
// With so few tokens every CTA can resolve all addresses for itself from the picks: used experts in
// ascending order, each with one tile, rows in (token, k) order.  So the dispatch has no launch of its own: the gate/up
// kernel reads the token's row where it is, and one CTA per tile leaves the rows and the tables where a dispatch would
// have put them.  The down kernel's CTAs hold a column for every used tile, so they also form the combined output.
// Each kernel costs about 4 us of launch, ramp and drain whatever it does: three instead of five.
// Measured, layer time, us, five launches / this: H 512, F 512, 32 experts, K 4: one token 20.8 / 14.0, five 29.8 / 23.0;
// H 1024, F 1024, 64 experts, K 8: 36.1 / 24.9, 65.5 / 59.7; Qwen-like: 42.5 / 30.9, 84.2 / 73.1; H 256, F 256: 19.8 / 14.0.
constexpr long long kFewDownBytes = 64ll << 20;

struct FewLayerParams {
  const __nv_bfloat16* x;  // [T, H]
  const __nv_bfloat16* w1; // gate rows, or the down matrix
  const __nv_bfloat16* w2; // up rows
  size_t expert_stride, shard_offset;
  int tp, ldb;
  int T, H, K, E, F;
  int tile_step;           // tiles per expert of the static regions; 0: the used experts' tiles follow one another
  const int* topk_idx;     // [T, K]
  const float* topk_w;     // [T, K]
  __nv_bfloat16* inter;    // [P * 128, F]
  __nv_bfloat16* out;      // [P * 128, H], or the staging rows of the push-style combine
  int push;
  __nv_bfloat16* y;        // [T, H]
  __nv_bfloat16* recv;     // what a dispatch leaves behind
  int *expert_count, *tile_expert, *src_info, *slot_of, *tile_count, *rows_done;
  int* status;
};

struct FewPicks {
  int idx[kFewAssign];     // the picked expert per assignment, -1: none
  int used[kMaxExperts];   // the used experts, ascending
  int mark[kMaxExperts];
  int warp_used[kFewWarps];
};

// Every thread of the CTA calls; returns the number of used experts.
__device__ __forceinline__ int few_picks(const FewLayerParams& p, FewPicks& s) {
  static_assert(kMaxExperts == kFewThreads && kFewAssign <= kFewThreads, "a thread per expert, a thread per assignment");
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
  s.mark[tid] = 0;
  __syncthreads();
  if (tid < p.T * p.K) {
    int e = __ldcg(p.topk_idx + tid);  // (may run before the wait on the previous kernel: from L2)
    if (e < 0 || e >= p.E) e = -1;
    s.idx[tid] = e;
    if (e >= 0) s.mark[e] = 1;
  }
  __syncthreads();
  const bool mine = s.mark[tid] != 0;
  const unsigned b = __ballot_sync(0xffffffffu, mine);
  if (lane == 0) s.warp_used[warp] = __popc(b);
  __syncthreads();
  int before = 0, n = 0;
#pragma unroll
  for (int w = 0; w < kFewWarps; ++w) {
    if (w < warp) before += s.warp_used[w];
    n += s.warp_used[w];
  }
  if (mine) s.used[before + __popc(b & ((1u << lane) - 1u))] = tid;
  __syncthreads();
  return n;
}

// A warp lists the assignments of expert e in ascending order, at most kFewMaxTokens of them (an expert is picked at
// most once per token); returns how many.
__device__ __forceinline__ int few_rows(const FewLayerParams& p, const FewPicks& s, int e, int* list) {
  const int lane = threadIdx.x % 32;
  int n = 0;
  __syncwarp();
  for (int base = 0; base < p.T * p.K; base += 32) {
    const bool hit = base + lane < p.T * p.K && s.idx[base + lane] == e;
    const unsigned b = __ballot_sync(0xffffffffu, hit);
    const int at = n + __popc(b & ((1u << lane) - 1u));
    if (hit && at < kFewMaxTokens) list[at] = base + lane;
    n += __popc(b);
  }
  __syncwarp();
  return min(n, kFewMaxTokens);
}

// The columns of one tile, for the `rows` (at most R) assignments listed, its rows from r0 on.
template <int R>
__device__ __forceinline__ void few_gate_up(const FewLayerParams& p, size_t base, int tile, int r0, const int* list, int rows) {
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  int off[R];
#pragma unroll
  for (int r = 0; r < R; ++r) off[r] = list[r < rows ? r : 0] / p.K * p.H;
  for (int n = blockIdx.x * kFewWarps + warp; n < p.F; n += gridDim.x * kFewWarps) {
    const size_t at = base + (size_t)n * p.ldb;
    const float mine = few_dots<R, true>(p.w1 + at, p.w2 + at, p.x, off, p.H);
    if (lane < rows) p.inter[((size_t)tile * kTileRows + r0 + lane) * p.F + n] = __float2bfloat16_rn(mine);
  }
}

// Grid: (CTAs per tile, T * K): blockIdx.y is the used expert's number.
template <int R>
__global__ void __launch_bounds__(kFewThreads)
few_gate_up_kernel(const FewLayerParams p) {
  __shared__ FewPicks s;
  __shared__ int s_list[kFewWarps][kFewMaxTokens];
  pdl_wait();
  pdl_trigger();
  const int n_used = few_picks(p, s);
  const int u = blockIdx.y;
  if (u >= n_used) return;
  const int warp = threadIdx.x / 32;
  const int e = s.used[u], tile = p.tile_step > 0 ? e * p.tile_step : u;
  const int* list = s_list[warp];
  const int rows = few_rows(p, s, e, s_list[warp]);
  if (blockIdx.x == gridDim.x - 1) {  // this tile's rows and table entries, for whoever looks at them after the layer
    const int vec = p.H / 8;
    for (int i = threadIdx.x; i < rows * vec; i += kFewThreads) {
      const int r = i / vec, v = i - r * vec;
      reinterpret_cast<uint4*>(p.recv + ((size_t)tile * kTileRows + r) * p.H)[v] =
          reinterpret_cast<const uint4*>(p.x + (size_t)(list[r] / p.K) * p.H)[v];
    }
    if ((int)threadIdx.x < rows) {
      const int slot = tile * kTileRows + threadIdx.x;
      p.src_info[slot] = list[threadIdx.x];
      p.slot_of[list[threadIdx.x]] = slot;
    }
    if (threadIdx.x == 0) {
      p.expert_count[e] = rows;
      p.tile_expert[tile] = e;
      p.tile_count[tile] = rows;
    }
    if (u == 0)
      for (int a = threadIdx.x; a < p.T * p.K; a += kFewThreads) {
        if (a == 0) *p.rows_done = p.T * p.K;
        if (s.idx[a] < 0) {  // not an expert: reported, adds nothing
          set_status(p.status, MOE_ERR_ARG, a / p.K);
          p.slot_of[a] = -1;
        }
      }
  }
  const size_t base = (size_t)(e / p.tp) * p.expert_stride + (size_t)(e % p.tp) * p.shard_offset;
  for (int r0 = 0; r0 < rows; r0 += R) {
    const int n = min(R, rows - r0);
    if (n == 1) few_gate_up<1>(p, base, tile, r0, list + r0, n);
    else if (R >= 2 && n == 2) few_gate_up<(R < 2 ? R : 2)>(p, base, tile, r0, list + r0, n);
    else if (R >= 4 && n <= 4) few_gate_up<(R < 4 ? R : 4)>(p, base, tile, r0, list + r0, n);
    else few_gate_up<R>(p, base, tile, r0, list + r0, n);
    if (R < 8) break;  // as many rows as tokens at most
  }
}

// The first 4 KB of a weight row on their way into L2.
__device__ __forceinline__ void few_prefetch(const __nv_bfloat16* w, int Kd) {
  const int k = (threadIdx.x % 32) * 64;
  if (k < Kd) asm volatile("prefetch.global.L2 [%0];" ::"l"(w + k));
}

template <int R>
__device__ __forceinline__ float few_down(const FewLayerParams& p, const __nv_bfloat16* w, int row0, int rows) {
  int off[R];
#pragma unroll
  for (int r = 0; r < R; ++r) off[r] = (r < rows ? r : 0) * p.F;
  return few_dots<R, false>(w, nullptr, p.inter + (size_t)row0 * p.F, off, p.F);
}

// A CTA holds kFewWarps / S columns, a column's used tiles being dealt to S warps; the CTA then adds up each token's K
// values in ascending k, rounded to the storage type as they are in `out`.
template <int R, int S>
__global__ void __launch_bounds__(kFewThreads, 3)
few_down_kernel(const FewLayerParams p) {
  constexpr int C = kFewWarps / S;
  __shared__ FewPicks s;
  __shared__ int s_list[kFewWarps][kFewMaxTokens];
  __shared__ float s_val[C][kFewAssign];
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, c = warp / S, part = warp % S;
  // The picks are the router's, complete before the gate/up kernel let this one start: they need no wait.
  const int n_used = few_picks(p, s);
  auto weights = [&](int e, int n) {
    return p.w1 + (size_t)(e / p.tp) * p.expert_stride + (size_t)(e % p.tp) * p.shard_offset + (size_t)n * p.ldb;
  };
  if (part < n_used && (int)blockIdx.x * C + c < p.H) few_prefetch(weights(s.used[part], blockIdx.x * C + c), p.F);
  pdl_wait();
  pdl_trigger();
  for (int n0 = blockIdx.x * C; n0 < p.H; n0 += gridDim.x * C) {
    const int n = n0 + c;
    for (int a = lane + 32 * part; a < p.T * p.K; a += 32 * S)
      if (s.idx[a] < 0) s_val[c][a] = 0.0f;
    for (int u = part; u < n_used && n < p.H; u += S) {
      const int e = s.used[u], tile = p.tile_step > 0 ? e * p.tile_step : u;
      const int rows = few_rows(p, s, e, s_list[warp]);
      if (u + S < n_used) few_prefetch(weights(s.used[u + S], n), p.F);
      else if (n + (int)gridDim.x * C < p.H) few_prefetch(weights(s.used[part], n + gridDim.x * C), p.F);
      const __nv_bfloat16* w = weights(e, n);
      for (int r0 = 0; r0 < rows; r0 += R) {
        const int m = min(R, rows - r0), row0 = tile * kTileRows + r0;
        float v;
        if (m == 1) v = few_down<1>(p, w, row0, m);
        else if (R >= 2 && m == 2) v = few_down<(R < 2 ? R : 2)>(p, w, row0, m);
        else if (R >= 4 && m <= 4) v = few_down<(R < 4 ? R : 4)>(p, w, row0, m);
        else v = few_down<R>(p, w, row0, m);
        if (lane < m) {
          const int a = s_list[warp][r0 + lane];
          const __nv_bfloat16 b = __float2bfloat16_rn(v);
          p.out[(size_t)(p.push ? a : row0 + lane) * p.H + n] = b;
          s_val[c][a] = __bfloat162float(b);
        }
        if (R < 8) break;
      }
    }
    __syncthreads();
    static_assert(kFewMaxTokens * C <= kFewThreads, "a thread per token and column");
    if ((int)threadIdx.x < p.T * C) {
      const int t = threadIdx.x / C, cc = threadIdx.x % C;
      if (n0 + cc < p.H) {
        float acc = 0.0f;
        for (int k = 0; k < p.K; ++k) acc = __fmaf_rn(p.topk_w[t * p.K + k], s_val[cc][t * p.K + k], acc);
        p.y[(size_t)t * p.H + n0 + cc] = __float2bfloat16_rn(acc);
      }
    }
    __syncthreads();
  }
}

// The rows are read again for every column and live in L1, so the gate/up kernel asks for most of it: launched behind the
// router while that still runs, it otherwise gets what its ring of shared memory left (Mixtral-like layer, one token:
// 139 us without this, 128 with it; two tokens 246 and 223).
template <typename Kern>
static void few_prefer_l1(Kern kern, int device, SmemAttrOnce& once) {
  if (device >= 0 && device < 64 && once.set[device]) return;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 8) != cudaSuccess) cudaGetLastError();  // a hint only
  if (device >= 0 && device < 64) once.set[device] = 1;
}

template <int R>
static int launch_few_layer(moe_plan* p, FewLayerParams q, const void* wd, cudaStream_t st) {
  const moe_config_t& c = p->cfg;
  static SmemAttrOnce once;
  const int tiles = min(c.T * c.K, c.E);  // at most this many are used
  few_prefer_l1(few_gate_up_kernel<R>, p->device, once);
  if (launch_pdl(few_gate_up_kernel<R>, few_grid(p, tiles, c.F), dim3(kFewThreads), 0, st, q) != cudaSuccess) return MOE_ERR_CUDA;
  p->launches += 1;
  mark(p, 4, st);
  // The combined form for one token, and for more while the down matrices are small: its warps wait for the slowest
  // tile of their column, which costs more than a launch when experts have unequal row counts and long columns.  Measured,
  // down (+ 5 us for the combine launch) / combined, us, by the down matrices' bytes: one token 23 MB 14.3 / 14.3, 235 MB
  // 45.1 / 45.1; two or more 46 MB 18.4 / 20.4, 84 MB 24.6 / 28.7, 115 MB 34.8 / 38.9, 940 MB 129 / 188.
  if (c.T > 1 && (long long)tiles * c.H * c.F * 2 > kFewDownBytes) {
    FewParams d = {};
    d.tp = p->tp;
    d.tile_expert = q.tile_expert;
    d.P = (int)p->P;
    d.E = c.E;
    d.tile_count = q.tile_count;
    d.rows_done = q.rows_done;
    d.total_rows = c.T * c.K;
    d.wait_ns = kDefaultWaitNs;
    d.status = q.status;
    int rc = launch_few_down<R, false>(p, d, wd, q.out, q.push ? q.src_info : nullptr, st);
    if (rc != 0) return rc;
    mark(p, 5, st);
    return launch_combine(p, q.out, q.slot_of, q.topk_w, q.y, st, q.push) ? MOE_ERR_CUDA : 0;
  }
  q.w1 = (const __nv_bfloat16*)wd;
  q.w2 = nullptr;
  q.shard_offset = (size_t)c.F;
  q.ldb = c.F * p->tp;
  const int sms = p->sm_count > 0 ? p->sm_count : 148;
  const int S = tiles >= 8 ? 8 : tiles >= 4 ? 4 : tiles >= 2 ? 2 : 1;  // warps per column: as many as there are tiles for
  const int grid = min(8 * sms, (c.H + kFewWarps / S - 1) / (kFewWarps / S));
  auto kern = S == 1 ? few_down_kernel<R, 1> : S == 2 ? few_down_kernel<R, 2> : S == 4 ? few_down_kernel<R, 4> : few_down_kernel<R, 8>;
  if (launch_pdl(kern, dim3(grid), dim3(kFewThreads), 0, st, q) != cudaSuccess) return MOE_ERR_CUDA;
  p->launches += 1;
  mark(p, 5, st);
  return 0;
}

// Four or five tokens with very long columns keep the separate dispatch: its launch saved is nothing there, and the rows
// taken from where the tokens are cost the gate/up kernel about 2 % (F 14336: 332 us with a dispatch, 339 without; F 6400
// and five tokens: 230 and 219).
bool few_layer_applies(const moe_plan* p) {
  const moe_config_t& c = p->cfg;
  return c.T > 0 && (c.T <= 3 || c.F <= 8192) && c.dtype == MOE_DTYPE_BF16 && !c.identity_experts && c.overlap == 0 &&
         p->P <= kMaxListTiles /* the expert call's limit, whatever the batch */ && few_applies(p);
}

int launch_few_layer(moe_plan* p, const void* x, const void* wg, const void* wu, const void* wd, void* y, cudaStream_t st) {
  const moe_config_t& c = p->cfg;
  Scratch& s = p->s;
  FewLayerParams q = {};
  q.x = (const __nv_bfloat16*)x;
  q.w1 = (const __nv_bfloat16*)wg;
  q.w2 = (const __nv_bfloat16*)wu;
  q.expert_stride = (size_t)c.F * p->tp * c.H;
  q.shard_offset = (size_t)c.F * c.H;
  q.tp = p->tp;
  q.ldb = c.H;
  q.T = c.T;
  q.H = c.H;
  q.K = c.K;
  q.E = c.E;
  q.F = c.F;
  q.tile_step = c.dispatch_mode == MOE_DISPATCH_ATOMIC_STATIC ? (int)(p->cap_rows / kTileRows) : 0;
  q.topk_idx = s.topk_idx;
  q.topk_w = s.topk_w;
  q.inter = (__nv_bfloat16*)s.inter;
  q.out = (__nv_bfloat16*)s.out_rows;
  q.push = c.combine_mode == 1;
  q.y = (__nv_bfloat16*)y;
  q.recv = (__nv_bfloat16*)s.recv;
  q.expert_count = s.expert_count;
  q.tile_expert = s.tile_expert;
  q.src_info = s.src_info;
  q.slot_of = s.slot_of;
  q.tile_count = s.tile_count;
  q.rows_done = s.rows_done;
  q.status = s.status;
  mark(p, 3, st);
  if (c.T <= 1) return launch_few_layer<1>(p, q, wd, st);
  if (c.T <= 2) return launch_few_layer<2>(p, q, wd, st);
  if (c.T <= 4) return launch_few_layer<4>(p, q, wd, st);
  if (c.T <= 5) return launch_few_layer<5>(p, q, wd, st);
  return launch_few_layer<8>(p, q, wd, st);
}

}  // namespace moehub
