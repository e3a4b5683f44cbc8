// Step 1 of the MoE layer (paper Section II-A, routing): every (token, expert) logit as ONE ascending fp32 FMA
// chain over h, then softmax weights and top-K.  Used for up to 64 experts, and for more while the batch is small
// (route_filter.cu takes over where running every chain costs more than finding out which ones matter).
//
// What bounds it: the chain itself (4.5 cycles per h with one chain per thread and one warp per SM scheduler) while
// an SM holds up to about 256 chains, and the issue slots beyond that (a thread with 2 chains: 16 FMAs, 12 unpacking,
// 3 address and 3 shared-load instructions per 8 h).  bf16 operands go into the FMA as they are (fma.rn.f32.bf16: the
// exact product of two bf16 numbers plus an fp32 sum, rounded once - the same bits as widening both first, with one
// instead of two extra instructions per pair of elements; the upper half of a word still has to be moved down).
//
// Layout.  A CTA owns a block of tokens and up to 64 experts (65-256 experts: 2 to 4 CTAs per block of tokens).  One thread streams the rows of x and Wr through a ring of shared-memory stages by TMA
// (128-byte boxes, 128-byte swizzle: rows that are read together lie on different banks); the compute warps wait per
// stage on its mbarrier, so no barrier holds the warps together.  The two lane grids (token by lane / 2, experts by
// lane % 2; or the other way round) are those whose 16-byte shared loads cost two pipe cycles instead of four.  With
// up to 64 experts the logits stay in the CTA's shared memory, where a warp (8 or 16 lanes for few experts) selects
// for a token; with more they go to a [T, 256] scratch and a second small launch selects.
//
// Measured (whole router call, us; before: operands converted to fp32 on their way into shared memory with one CTA
// barrier per 256 h, for more than 64 experts the tensor-core filter):
//   T 512, H 2048, 60 experts 18.6 -> 12.0; T 2777 65.7 -> 28.8; T 8192 170 -> 66; T 24, H 4096, 8 experts 30.9 -> 16.6;
//   T 4096 32.9 -> 20.7; T 1023, H 4096, 16 experts 41.9 -> 18.7; H 7168, 256 experts: T 64 151 -> 27, T 256 123 -> 43.
#include "route_common.cuh"
#include "route_shape.h"
#include "tc_common.cuh"

namespace moehub {

constexpr int kRcBox = 128;                 // bytes of a row per TMA box
constexpr int kRcMaxBoxes = 4;              // most boxes per stage
constexpr int kRcMaxStages = 8;
constexpr int kRcRingBytes = 160 * 1024;    // most shared memory for the ring
constexpr int kRcMaxWarps = 24;             // most compute warps per CTA (one CTA per SM, 80 registers a thread)

// One 16-byte unit of TM tokens' rows against one of TN experts' rows.
__device__ __forceinline__ uint32_t word_of(const uint4& v, int q) { return q == 0 ? v.x : q == 1 ? v.y : q == 2 ? v.z : v.w; }
template <int TM, int TN>
__device__ __forceinline__ void chain_unit(const uint4 (&x)[TM], const uint4 (&w)[TN], float (&acc)[TM][TN], float) {
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j)
        acc[i][j] = __fmaf_rn(__uint_as_float(word_of(x[i], q)), __uint_as_float(word_of(w[j], q)), acc[i][j]);
}
template <int TM, int TN>
__device__ __forceinline__ void chain_unit(const uint4 (&x)[TM], const uint4 (&w)[TN], float (&acc)[TM][TN], __nv_bfloat16) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) acc[i][j] = fma_bf16_lo(word_of(x[i], q), word_of(w[j], q), acc[i][j]);
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) acc[i][j] = fma_bf16_hi(word_of(x[i], q), word_of(w[j], q), acc[i][j]);
  }
}

struct ChainParams {
  const float* bias;  // [E] or nullptr
  int T, E, K, renorm, tp;
  int row_bytes;      // H * element size
  int tb;             // tokens per CTA
  int boxes, stages;  // boxes per stage, stages of the ring
  int split;          // CTAs that share a block of tokens
  float* logits;      // [T, 256], split > 1
  int* topk_idx;
  float* topk_w;
  unsigned long long wait_ns;
  int* status;
};

__host__ __device__ constexpr int rc_x_box_bytes(int tb) { return (tb * kRcBox + 1023) & ~1023; }  // boxes start on 1024 bytes
__host__ constexpr size_t rc_smem(int tb, int epc, int boxes, int stages, int split) {
  return 1024 + (size_t)stages * boxes * (rc_x_box_bytes(tb) + epc * kRcBox) + (split > 1 ? 0 : (size_t)tb * epc * 4);
}

// SWAP false: a warp is 16 TM tokens x 2 TN experts; true: 2 TM tokens x 16 TN experts.  EW warps side by side cover the
// CTA's experts, the rest of the compute warps its tokens; the last warp brings the operands in.
template <typename XT, bool SWAP, int TM, int TN, int EW>
__global__ void __launch_bounds__(32 * (kRcMaxWarps + 1), 1)
route_chains_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w, const ChainParams p,
                    const PrepArgs prep) {
  constexpr int GT = SWAP ? 2 : 16, GE = SWAP ? 16 : 2;  // token / expert groups of a warp
  constexpr int EPC = EW * GE * TN;                       // experts of the CTA
  constexpr int kWBox = EPC * kRcBox;
  __shared__ int s_hist[kRouteMaxExperts];
  __shared__ unsigned long long s_full[kRcMaxStages], s_empty[kRcMaxStages];
  __shared__ int s_abort;
  extern __shared__ uint8_t rc_dyn[];
  uint8_t* ring = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(rc_dyn) + 1023) & ~(uintptr_t)1023);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int cwarps = blockDim.x / 32 - 1;
  const int x_box = rc_x_box_bytes(p.tb), stage_bytes = p.boxes * (x_box + kWBox);
  float* ls = reinterpret_cast<float*>(ring + (size_t)p.stages * stage_bytes);  // [tb][EPC], split == 1
  const int t0 = (int)(blockIdx.x / p.split) * p.tb;
  const int e0 = (int)(blockIdx.x % p.split) * EPC;
  const bool split = p.split > 1;
  const int nbox = (p.row_bytes + kRcBox - 1) / kRcBox, nstage = (nbox + p.boxes - 1) / p.boxes;
  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(smem_u32(&s_full[s]), 1);
      mbar_init(smem_u32(&s_empty[s]), cwarps);
    }
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  pdl_wait();
  pdl_trigger();
  __syncthreads();
  volatile int* abort_flag = &s_abort;
  bool failed = false;
  int issued = 0;  // stages the producer has filled

  if (warp == cwarps) {
    if (lane == 0) {  // producer
      int b = 0;
      uint32_t phase = 1;
      for (int s = 0; s < nstage; ++s) {
        if (!mbar_wait(smem_u32(&s_empty[b]), phase, abort_flag, p.wait_ns)) {
          failed = true;
          s_abort = 1;
          break;
        }
        issued = s + 1;
        const int boxes = min(p.boxes, nbox - s * p.boxes);
        const uint32_t bar = smem_u32(&s_full[b]), dst = smem_u32(ring) + (uint32_t)(b * stage_bytes);
        mbar_expect_tx(bar, (uint32_t)boxes * (uint32_t)(p.tb * kRcBox + kWBox));
        for (int q = 0; q < boxes; ++q) {  // rows past T or E and columns past H arrive as zeros
          const int c = (s * p.boxes + q) * (kRcBox / (int)sizeof(XT));
          tma_load_2d(dst + (uint32_t)(q * x_box), &map_x, bar, c, t0);
          tma_load_2d(dst + (uint32_t)(p.boxes * x_box + q * kWBox), &map_w, bar, c, e0);
        }
        if (++b == p.stages) { b = 0; phase ^= 1u; }
      }
    }
    __syncwarp();
    route_prep_begin(prep, s_hist);
  } else {
    route_prep_begin(prep, s_hist);  // while the first stages are on their way
    const int tl = (warp / EW) * GT * TM + (SWAP ? lane % 2 : lane / 2);  // this lane's tokens of the block: tl + GT * i
    const int el = (warp % EW) * GE * TN + (SWAP ? lane / 2 : lane % 2);  // its experts: el + GE * j
    // byte offsets of the rows inside a box, the swizzle's row bits in place: unit u of a row is at (offset ^ u * 16)
    uint32_t xoff[TM], woff[TN];
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      const int r = tl + GT * i;
      xoff[i] = (uint32_t)r * kRcBox + ((uint32_t)(r & 7) << 4);
    }
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int r = el + GE * j;
      woff[j] = (uint32_t)(p.boxes * x_box) + (uint32_t)r * kRcBox + ((uint32_t)(r & 7) << 4);
    }
    float acc[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) acc[i][j] = 0.0f;
    const uint32_t ring0 = smem_u32(ring);
    // One unit of operands ahead: while unit u is computed, unit u + 1 is on its way from shared memory - across the
    // boxes of a stage too; only a new stage starts with a wait.
    auto fetch = [&](uint4 (&xv)[TM], uint4 (&wv)[TN], const uint32_t (&xa)[TM], const uint32_t (&wa)[TN], int u) {
#pragma unroll
      for (int i = 0; i < TM; ++i) xv[i] = lds128(xa[i] ^ (uint32_t)(u << 4));
#pragma unroll
      for (int j = 0; j < TN; ++j) wv[j] = lds128(wa[j] ^ (uint32_t)(u << 4));
    };
    int ring_stage = 0;
    uint32_t ring_phase = 0;
    for (int box0 = 0; box0 < nbox; box0 += p.boxes) {
      // A lane whose wait ran out stays with its warp (the others' may not have) and computes on whatever the stage holds.
      failed |= !mbar_wait(smem_u32(&s_full[ring_stage]), ring_phase, abort_flag, p.wait_ns);
      const int boxes = min(p.boxes, nbox - box0);
      const uint32_t base = ring0 + (uint32_t)(ring_stage * stage_bytes);
      uint32_t xa[TM], wa[TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) xa[i] = base + xoff[i];
#pragma unroll
      for (int j = 0; j < TN; ++j) wa[j] = base + woff[j];
      uint4 xv[TM], wv[TN];
      fetch(xv, wv, xa, wa, 0);
#pragma unroll 1
      for (int q = 0; q < boxes; ++q) {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          if (u == 7) {  // the next box's first unit (after the last box: operands nobody uses, from inside the ring)
#pragma unroll
            for (int i = 0; i < TM; ++i) xa[i] += q + 1 < boxes ? (uint32_t)x_box : 0u;
#pragma unroll
            for (int j = 0; j < TN; ++j) wa[j] += q + 1 < boxes ? (uint32_t)kWBox : 0u;
          }
          uint4 nx[TM], nw[TN];
          fetch(nx, nw, xa, wa, (u + 1) & 7);
          chain_unit(xv, wv, acc, XT());
#pragma unroll
          for (int i = 0; i < TM; ++i) xv[i] = nx[i];
#pragma unroll
          for (int j = 0; j < TN; ++j) wv[j] = nw[j];
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&s_empty[ring_stage]));
      if (++ring_stage == p.stages) { ring_stage = 0; ring_phase ^= 1u; }
    }
    if (failed) s_abort = 1;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      const int t = tl + GT * i;
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        const int ec = el + GE * j, e = e0 + ec;
        float l = acc[i][j];
        if (p.bias != nullptr && e < p.E) l = l + p.bias[e];
        if (!split) ls[t * EPC + ec] = l;
        else if (t0 + t < p.T) p.logits[(size_t)(t0 + t) * kRouteMaxExperts + e] = l;
      }
    }
  }
  __syncthreads();
  if (failed) set_status(p.status, MOE_ERR_TIMEOUT, kWaitMbarTma);
  if (s_abort) {  // (read after the barrier) no copy may still be landing when the CTA's shared memory goes away
    for (int g = max(0, issued - p.stages); g < issued; ++g) {  // only the producer has issued any
      const unsigned long long ts = globaltimer();
      while (!mbar_try(smem_u32(&s_full[g % p.stages]), (uint32_t)(g / p.stages) & 1u))
        if (globaltimer() - ts > p.wait_ns + 1000000ull) break;
    }
    __syncthreads();
  }
  if (split) return;
  constexpr int G = EPC < 32 ? EPC : 32;
  select_topk<G, EPC / G>(ls, EPC, min(p.tb, p.T - t0), t0, p.E, p.K, p.renorm, p.topk_idx, p.topk_w, prep.hist ? s_hist : nullptr,
                          p.tp);
  route_prep_end(prep, s_hist);
}

// Selection for more than 64 experts: a warp per token on the logits the chain kernel left in global memory.
constexpr int kRsTokens = 4;
__global__ void __launch_bounds__(32 * kRsTokens)
route_select_kernel(const ChainParams p, const PrepArgs prep) {
  __shared__ int s_hist[kRouteMaxExperts];
  if (prep.hist != nullptr)
    for (int e = threadIdx.x; e < kRouteMaxExperts; e += blockDim.x) s_hist[e] = 0;
  __syncthreads();
  pdl_wait();
  pdl_trigger();
  const int t0 = blockIdx.x * kRsTokens;
  const float* ls = p.logits + (size_t)t0 * kRouteMaxExperts;
  int* hist = prep.hist ? s_hist : nullptr;
  if (p.E <= 128) select_topk<32, 4>(ls, kRouteMaxExperts, min(kRsTokens, p.T - t0), t0, p.E, p.K, p.renorm, p.topk_idx, p.topk_w, hist, p.tp);
  else select_topk<32, 8>(ls, kRouteMaxExperts, min(kRsTokens, p.T - t0), t0, p.E, p.K, p.renorm, p.topk_idx, p.topk_w, hist, p.tp);
  route_prep_end(prep, s_hist);
}

// ---- host side ----------------------------------------------------------------------------------------
// Rows of 16-byte units by their bytes: [rows, row_bytes], box [box_rows, 128 bytes], 128-byte swizzle.
static int make_row_map(EncodeTiledFn enc, CUtensorMap* m, const void* base, int rows, int cols, int elem, int box_rows) {
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)cols * elem};
  cuuint32_t box[2] = {(cuuint32_t)(kRcBox / elem), (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(m, elem == 2 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(base),
                   dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? MOE_OK : MOE_ERR_CUDA;
}

template <typename XT, bool SWAP, int TM, int TN, int EW>
static int launch_chains(moe_plan* p, const void* x, const void* wr, const float* bias, int* topk_idx, float* topk_w,
                         const PrepArgs& prep, int split, cudaStream_t st) {
  constexpr int GT = (SWAP ? 2 : 16) * TM, EPC = EW * (SWAP ? 16 : 2) * TN;
  constexpr int kMaxTw = kRcMaxWarps / EW;
  const moe_config_t& c = p->cfg;
  const int sms = p->sm_count > 0 ? p->sm_count : 148;
  const int tw = route_token_warps(c.T, c.H, GT, split, EW, TM * TN, kMaxTw, sms);
  ChainParams q;
  q.bias = bias;
  q.T = c.T;
  q.E = p->route_E;
  q.K = p->route_K;
  q.renorm = c.renormalize;
  q.tp = p->tp;
  q.row_bytes = c.H * (int)sizeof(XT);
  q.tb = GT * tw;
  q.split = split;
  q.logits = p->s.route_logits;
  // Stages of up to 512 bytes of every row (a stage costs a wait and a hand-back, about 60 cycles), at least four of them.
  const int box_bytes = rc_x_box_bytes(q.tb) + EPC * kRcBox, nbox = (q.row_bytes + kRcBox - 1) / kRcBox;
  q.boxes = max(1, min(kRcMaxBoxes, kRcRingBytes / 4 / box_bytes));
  q.stages = max(1, min(min(kRcMaxStages, kRcRingBytes / (q.boxes * box_bytes)), (nbox + q.boxes - 1) / q.boxes));
  q.topk_idx = topk_idx;
  q.topk_w = topk_w;
  q.wait_ns = kDefaultWaitNs;  // the waits are on this CTA's own copies: nothing a caller's limit is meant for
  q.status = p->s.status;
  EncodeTiledFn enc;
  int rc = get_encoder(p, &enc);
  if (rc != MOE_OK) return rc;
  CUtensorMap mx, mw;
  if ((rc = make_row_map(enc, &mx, x, c.T, c.H, (int)sizeof(XT), q.tb)) != MOE_OK) return rc;
  if ((rc = make_row_map(enc, &mw, wr, p->route_E, c.H, (int)sizeof(XT), EPC)) != MOE_OK) return rc;
  auto kern = route_chains_kernel<XT, SWAP, TM, TN, EW>;
  const size_t smem = rc_smem(q.tb, EPC, q.boxes, q.stages, split);
  static SmemAttrOnce once;  // per instantiation
  if (cudaError_t e = ensure_dynamic_smem(kern, smem, p->device, once)) return (int)e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((c.T + q.tb - 1) / q.tb * split));
  cfg.blockDim = dim3((unsigned)(32 * (EW * tw + 1)));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  p->launches += 1;  // (the first kernel of the layer is launched plainly, see common.cuh)
  if (cudaError_t e = cudaLaunchKernelEx(&cfg, kern, mx, mw, q, prep)) return (int)e;
  if (split == 1) return 0;
  p->launches += 1;
  return (int)launch_pdl(route_select_kernel, dim3((c.T + kRsTokens - 1) / kRsTokens), dim3(32 * kRsTokens), 0, st, q, prep);
}

template <typename XT>
static int launch_chains_typed(moe_plan* p, const void* x, const void* wr, const float* bias, int* topk_idx, float* topk_w,
                               const PrepArgs& prep, cudaStream_t st) {
  const int E = p->route_E, T = p->cfg.T;  // the experts the router scores (the plan's E counts every TP shard of an expert)
  const int sms = p->sm_count > 0 ? p->sm_count : 148;
  const long long chains = (long long)T * (E <= 8 ? 8 : E <= 16 ? 16 : (E + 31) / 32 * 32);
  // Chains per thread.  One (4.5 cycles per h) while a scheduler then has one warp at most; two (6.2, 3.8 per warp from
  // four warps on); eight (12.5 per warp) where the SMs are full: a third fewer unpacking and load instructions per
  // chain (T 8192, H 2048, 60 experts: 81 -> 66 us; T 2777: 29 us with two, 35 with eight).
#define MOEHUB_CHAINS(SWAP, TM, TN, EW, CS) launch_chains<XT, SWAP, TM, TN, EW>(p, x, wr, bias, topk_idx, topk_w, prep, CS, st)
  if (chains <= 128ll * sms) {
    if (E <= 8) return MOEHUB_CHAINS(false, 1, 1, 4, 1);
    if (E <= 16) return MOEHUB_CHAINS(false, 1, 1, 8, 1);
    if (E <= 32) return MOEHUB_CHAINS(true, 1, 1, 2, 1);
    return MOEHUB_CHAINS(true, 1, 1, 4, (E + 63) / 64);
  }
  if (E <= 8) return MOEHUB_CHAINS(false, 1, 2, 2, 1);
  if (E <= 16) return MOEHUB_CHAINS(false, 1, 2, 4, 1);
  if (E <= 32) return MOEHUB_CHAINS(true, 1, 2, 1, 1);
  const long long slots = (long long)T * ((E + 63) / 64) * 64;  // (a CTA has 64 experts' chains whether or not they exist)
  if (slots <= 1536ll * sms) return MOEHUB_CHAINS(true, 1, 2, 2, (E + 63) / 64);
  return MOEHUB_CHAINS(true, 4, 2, 2, (E + 63) / 64);
#undef MOEHUB_CHAINS
}

int launch_route_chains(moe_plan* p, const void* x, const void* wr, const float* bias, int* topk_idx, float* topk_w,
                        const PrepArgs& prep, cudaStream_t st) {
  if (p->cfg.dtype == MOE_DTYPE_BF16)
    return launch_chains_typed<__nv_bfloat16>(p, x, wr, bias, topk_idx, topk_w, prep, st);
  return launch_chains_typed<float>(p, x, wr, bias, topk_idx, topk_w, prep, st);
}

}  // namespace moehub
