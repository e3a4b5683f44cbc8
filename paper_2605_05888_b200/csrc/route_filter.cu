// Step 1 of the MoE layer (paper Section II-A, routing) for many experts on bf16 data: a tensor-core filter
// in front of the exact chains.
//
// The pick of the K experts is defined on ONE ascending fp32 FMA chain per (token, expert), and it has to
// come out bit for bit.  Only a handful of the E chains of a token decide anything, though.  So:
//
//  (1) route_tc_logits_kernel: approximate logits l~ = x * Wr^T for every (token, expert) with tcgen05 MMAs
//      (128 tokens x 128 experts per CTA, operands by TMA, four fp32 accumulators in tensor memory that take the
//      64-column steps of h in turn and are summed at the end), written to a [T, 256] fp32 scratch.  Products of two bf16 numbers are exact in fp32; only the order and rounding
//      of the additions differ from the chain.  Its idle epilogue warps also compute |w_e|^2 per expert.
//  (2) route_refine_kernel: per token, the K-th largest approximate logit minus twice an error bound is a
//      threshold; every expert at or above it is a candidate and gets its exact chain; the exact values
//      replace the approximate ones and the usual selection runs on the row.
//
// Why the picks are the exact ones.  Error model: every fp32 addition, whether rounded to nearest or truncated, is
// off by at most 2^-23 of the sum of the magnitudes that have gone into it, which never exceeds S = sum_h |x_h * w_eh|.
// An MMA adds 16 products to an accumulator: 17 additions, in whatever order; an accumulator takes at most
// n = 4 * ceil(H / 256) MMAs, and the four meet in 3 more additions.  Over the accumulators' shares of S that is
// |l~ - exact sum| <= (17 n + 3) * 2^-23 * S, and the chain (rounded to nearest) is within H * 2^-24 * S of the exact
// sum: |l~ - l| <= eps = (H / 2 + 17 n + 3) * 2^-23 * S, with S <= |x_t| * max_e |w_e| (Cauchy-Schwarz) computed from
// the data of the call.  The K experts with the largest l~ have l >= kth~ - eps
// and every expert below the threshold kth~ - 2 eps has l < kth~ - eps, so none of those can be among the K
// largest l, ties included.  The kernel checks the model on every candidate (both values are at hand) and
// reports MOE_ERR_INTERNAL if |l~ - l| ever exceeded eps.  Largest |l~ - l| / eps over EVERY expert of 1100 tokens, H 64 to
// 7168: 0.16 on constant rows of one sign (where S is all of |x| |w| and every rounding goes the same way), 0.04 on rows
// that fall off over twenty binades, at most 0.03 on normal, parallel, one-sign, cancelling, spiked and wide-ranged ones.
//
// The softmax weights use the exact logits of the candidates and the approximate ones of the rest: the rest
// only enters the denominator.  What the accumulation's rounding adds up to grows with the number of additions
// in a row (measured), which is why the approximate logit is the sum of four accumulators.
#include "route_common.cuh"
#include "tc_common.cuh"

namespace moehub {

constexpr int kRfEP = 256;           // experts covered (the accumulator's columns)
constexpr float kRfUlp = 1.1920929e-7f;  // 2^-23
constexpr int kRfChunk = 64;         // h per staged chunk: 128 bytes of a row
constexpr int kRfBufs = 3;           // staged chunks in flight
constexpr int kRfAhead = 8;          // chunks of x asked for ahead of that, into L2
constexpr int kRfWBytes = kRfEP * kRfChunk * 2;  // one chunk of every expert's row: 32 KB
// shared memory of the refine kernel for tpc tokens per CTA (half a warp each): kRfBufs buffers of one chunk of Wr
// and of the tokens' rows of x (written by TMA, 128-byte swizzle), the tokens' logit rows, the list of chains
__host__ __device__ constexpr int rf_x_bytes(int tpc) { return (tpc * kRfChunk * 2 + 1023) & ~1023; }  // buffers start on 1024 bytes
constexpr size_t rf_smem(int tpc) {
  return 1024 + (size_t)kRfBufs * (kRfWBytes + rf_x_bytes(tpc)) + (size_t)tpc * kRfEP * 4 + (size_t)tpc * kRfEP * 2;
}

// M = 128 tokens, N = 128 experts per MMA
constexpr uint32_t kRfIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(128 >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);

struct RfShared {
  unsigned long long full[kStages];
  unsigned long long empty[kStages];
  unsigned long long acc_full;
  unsigned long long drain;
  int fills;  // stages that the producer has filled
  uint32_t tmem_base;
  int abort_flag;
};

__global__ void __launch_bounds__(kTcThreads, 1)
route_tc_logits_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w,
                       const __nv_bfloat16* __restrict__ wr, int T, int H, int E, float* __restrict__ logits,
                       float* __restrict__ wnorm2, unsigned long long wait_ns, int* __restrict__ status) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* stage_base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  RfShared* sh = reinterpret_cast<RfShared*>(stage_base + kStages * kStageBytes);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(smem_u32(&sh->full[s]), 1);
      mbar_init(smem_u32(&sh->empty[s]), 1);
    }
    mbar_init(smem_u32(&sh->acc_full), 1);
    mbar_init(smem_u32(&sh->drain), 1);
    sh->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sh->tmem_base)),
                 "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  pdl_wait();
  pdl_trigger();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = sh->tmem_base;
  volatile int* abort_flag = &sh->abort_flag;
  // this CTA's slice of h, in steps of 64 columns (gridDim.z slices: a scratch of their own each, summed by the reader)
  const int all = (H + kBK - 1) / kBK, per = (all + gridDim.z - 1) / gridDim.z;
  const int kb0 = blockIdx.z * per, KB = min(per, all - kb0);
  logits += (size_t)blockIdx.z * T * kRfEP;
  const int t0 = blockIdx.x * kTileRows;
  const int e0 = blockIdx.y * 128;  // this CTA's half of the experts
  int fail_site = 0;

  if (warp == 0) {
    if (lane == 0) {  // TMA producer: the tokens' x tile and all experts' Wr block, 64 columns of h per stage
      int stage = 0, fills = 0;
      uint32_t phase_bit = 0;
      for (int kb = 0; kb < KB; ++kb) {
        if (!mbar_wait(smem_u32(&sh->empty[stage]), phase_bit ^ 1u, abort_flag, wait_ns)) { fail_site = kWaitMbarTma; break; }
        const uint32_t full = smem_u32(&sh->full[stage]);
        const uint32_t a_dst = smem_u32(stage_base + stage * kStageBytes);
        mbar_expect_tx(full, (uint32_t)(kABytes + kBBytes / 2));
        tma_load_2d(a_dst, &map_x, full, (kb0 + kb) * kBK, t0);   // rows past T and columns past H arrive as zeros
        tma_load_2d(a_dst + kABytes, &map_w, full, (kb0 + kb) * kBK, e0);  // 128 experts' rows
        ++fills;
        if (++stage == kStages) { stage = 0; phase_bit ^= 1u; }
      }
      if (fail_site) sh->abort_flag = 1;
      sh->fills = fills;
    }
  } else if (warp == 1) {
    if (lane == 0) {  // MMA issuer: D[128 tokens, 256 experts] += x tile * Wr block^T
      int stage = 0;
      uint32_t phase_bit = 0;
      for (int kb = 0; kb < KB; ++kb) {
        if (!mbar_wait(smem_u32(&sh->full[stage]), phase_bit, abort_flag, wait_ns)) { fail_site = kWaitMbarMma; break; }
        tc_fence_after();
        const uint32_t a_addr = smem_u32(stage_base + stage * kStageBytes);
        const uint64_t adesc = smem_desc_sw128(a_addr), bdesc = smem_desc_sw128(a_addr + kABytes);
#pragma unroll
        // four accumulators that take the steps in turn: a quarter as many additions in a row for each logit
        // (they are summed in the epilogue), and so a quarter of what the accumulation's rounding adds up to
        for (int k = 0; k < kBK / 16; ++k)
          tc_mma(tmem_base + (uint32_t)(kb & 3) * 128u, adesc + 2 * k, bdesc + 2 * k, kRfIdesc, ((kb >> 2) | k) != 0 ? 1u : 0u);
        tc_commit(smem_u32(&sh->empty[stage]));
        if (++stage == kStages) { stage = 0; phase_bit ^= 1u; }
      }
      if (!fail_site) tc_commit(smem_u32(&sh->acc_full));
      if (fail_site) sh->abort_flag = 1;
    }
  } else {
    // While the main loop runs: |w_e|^2 for this CTA's share of the experts (the refine kernel's error bound).
    for (int e = ((blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x) * 4 + (warp - 2); e < E; e += gridDim.x * gridDim.y * gridDim.z * 4) {
      const uint4* row = reinterpret_cast<const uint4*>(wr + (size_t)e * H);
      float s = 0.0f;
      uint32_t bits = 0;
#pragma unroll 8
      for (int v = lane; v < H / 8; v += 32) {
        float f[8];
        const uint4 u = __ldg(row + v);
        bits |= u.x | u.y | u.z | u.w;
        Vec16<__nv_bfloat16>::unpack(u, f);
#pragma unroll
        for (int q = 0; q < 8; ++q) s = fmaf(f[q], f[q], s);
      }
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
      const bool zeros = __all_sync(0xffffffffu, (bits & 0x7fff7fffu) == 0u);
      if (lane == 0) wnorm2[e] = zeros ? 0.0f : fmaxf(s, FLT_MIN);  // (zero: a row of zeros; fmaxf keeps s unless it underflowed or is NaN)
    }
    // epilogue: the accumulator row of token t0 + 32 * (warp % 4) + lane, 16 experts at a time
    const int quarter = warp & 3;
    if (!warp_agrees(mbar_wait(smem_u32(&sh->acc_full), 0u, abort_flag, wait_ns, 200))) {
      fail_site = kWaitMbarEpi;
    } else {
      tc_fence_after();
      const int t = t0 + quarter * 32 + lane;
      const uint32_t t_row = tmem_base + ((uint32_t)(quarter * 32) << 16);
      float* dst = logits + (size_t)t * kRfEP + e0;
      const int nacc = min(KB, 4);  // accumulators that were written at all
#pragma unroll 1
      for (int c = 0; c < 128; c += 16) {
        float f[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) f[q] = 0.0f;
        for (int a = 0; a < nacc; ++a) {
          uint32_t v[16];
          tc_ld16(t_row + (uint32_t)a * 128u + c, v);
          tc_wait_ld();
#pragma unroll
          for (int q = 0; q < 16; ++q) f[q] += __uint_as_float(v[q]);
        }
        if (t < T) {
#pragma unroll
          for (int q = 0; q < 16; q += 4) *reinterpret_cast<float4*>(dst + c + q) = make_float4(f[q], f[q + 1], f[q + 2], f[q + 3]);
        }
        __syncwarp();  // (the last tokens' lanes stored, those past T did not; the next loads want the whole warp)
      }
    }
    if (fail_site) sh->abort_flag = 1;
  }
  if (fail_site) set_status(status, MOE_ERR_TIMEOUT, fail_site);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (sh->abort_flag) {  // whichever role gave up: MMAs and copies in flight end (bounded) before their memory is freed
    if (warp == 1 && lane == 0) {
      tc_commit(smem_u32(&sh->drain));
      const unsigned long long ts = globaltimer();
      while (!mbar_try(smem_u32(&sh->drain), 0u))
        if (globaltimer() - ts > wait_ns + 1000000ull) break;
    }
    if (threadIdx.x == 0) {
      for (int g = max(0, sh->fills - kStages); g < sh->fills; ++g) {
        const unsigned long long ts = globaltimer();
        while (!mbar_try(smem_u32(&sh->full[g % kStages]), (uint32_t)(g / kStages) & 1u))
          if (globaltimer() - ts > wait_ns + 1000000ull) break;
      }
    }
    __syncthreads();
  }
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
}


// ---- (2) candidates, exact chains, selection ----------------------------------------------------------
// A CTA takes tpc tokens, half a warp each (a warp runs two tokens in lockstep) for everything that is per
// token: the row of approximate logits (+ bias) into shared memory; |x_t| from the row of x; the K-th largest
// approximate logit by K rounds of a 16-lane arg-max; the threshold; the candidates.  The chains of all
// tokens of the CTA are then numbered through and thread s runs chain s (so no lane idles because its token
// has few candidates).  A chain reads its expert's row of Wr front to back; threads reading different rows
// straight from global memory would spend their time in the load unit and fetch a row once per (token,
// candidate) pair, so one thread brings in one chunk (64 h: 128 bytes) of EVERY expert's row and of every
// token's row of x per step with two TMA copies, kRfBufs - 1 chunks ahead, and each chain reads its rows from
// shared memory (128-byte swizzle: 16-byte unit u of row r sits at u ^ (r % 8)).  Exact values go back into
// the logit rows; then the common selection.
// What bounds it: shared memory (ncu, T 8192, H 7168, 256 experts: its pipe 65 % busy with 5.4 wavefronts per 16-byte load
// and another 11 % with the TMA writes; issue slots 48 %).  Whole router call, us, before / after the numbering by e % 8,
// CTAs of any even token count (T 8192: 147 CTAs of 56 tokens instead of 128 of 64) and x asked for ahead / with the
// error bound counted per MMA (before: H * 2^-23 * S for the approximate logit too, half a candidate more per token), all
// experts equally popular (with Zipf 1.2 at T 16384 the call takes 492 instead of 431: popular classes overflow): T 2048
// 113 / 108 / 107, T 4096 147 / 131 / 130, T 6000 262 / 176 / 169, T 8192 258 / 225 / 213, T 16384 508 / 438 / 414.
template <int MAXT>
__global__ void __launch_bounds__(MAXT * 16, 1)
route_refine_kernel(const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_x,
                    const __nv_bfloat16* __restrict__ x, const float* __restrict__ bias, const float* __restrict__ logits,
                    const float* __restrict__ wnorm2, int tpc, int T, int H, int E, int K, int renorm, int* __restrict__ topk_idx,
                    float* __restrict__ topk_w, const PrepArgs prep, int tp, unsigned long long wait_ns,
                    int* __restrict__ status) {
  const int NT = tpc * 16;
  const int kXBytes = rf_x_bytes(tpc);
  __shared__ int s_hist[kRouteMaxExperts];
  __shared__ unsigned char s_ncand[MAXT][8];  // a token's candidates per bucket (expert % 8)
  __shared__ int s_total[8];
  __shared__ float s_eps[MAXT];
  __shared__ unsigned long long s_full[kRfBufs];
  __shared__ unsigned long long s_empty[kRfBufs];  // a buffer may be refilled once every warp has left it
  __shared__ int s_abort;
  extern __shared__ uint8_t rf_dyn[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(rf_dyn) + 1023) & ~(uintptr_t)1023);
  uint8_t* w_stage = base;                                              // [kRfBufs][256 experts][128 bytes]
  uint8_t* x_stage = base + (size_t)kRfBufs * kRfWBytes;                // [kRfBufs][tpc tokens][128 bytes]
  float* ls = reinterpret_cast<float*>(x_stage + (size_t)kRfBufs * kXBytes);  // [tpc][256] logits: approximate, exact where a chain ran
  unsigned short* chains = reinterpret_cast<unsigned short*>(ls + (size_t)tpc * kRfEP);  // [tpc * 256]: token << 8 | expert; 0xffff: none
  const int t0 = blockIdx.x * tpc;
  const int tvalid = min(tpc, T - t0);
  const int lane = threadIdx.x % 32, l16 = threadIdx.x % 16, half = lane / 16;
  const int tl = threadIdx.x / 16;  // this half-warp's token inside the block
  const bool live = tl < tvalid;
  if (threadIdx.x == 0) {
    for (int b = 0; b < kRfBufs; ++b) {
      mbar_init(smem_u32(&s_full[b]), 1);
      mbar_init(smem_u32(&s_empty[b]), NT / 32);
    }
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  pdl_wait();
  pdl_trigger();
  route_prep_begin(prep, s_hist);
  volatile int* abort_flag = &s_abort;

  // the row of approximate logits (16 per lane: experts l16 + 16 j), bias added the way the chain's value gets it
  float v[16];
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const int e = l16 + 16 * j;
    float a = -FLT_MAX;
    if (live && e < E) {
      a = logits[(size_t)(t0 + tl) * kRfEP + e];
      if (bias != nullptr) a = a + bias[e];
    }
    v[j] = a;
    ls[tl * kRfEP + e] = a;
  }
  // |x_t|^2 and max_e |w_e|^2
  float xn2 = 0.0f, wm2 = 0.0f;
  if (live) {
    const uint4* xr = reinterpret_cast<const uint4*>(x + (size_t)(t0 + tl) * H);
#pragma unroll 8
    for (int q = l16; q < H / 8; q += 16) {
      float f[8];
      Vec16<__nv_bfloat16>::unpack(__ldg(xr + q), f);
#pragma unroll
      for (int i = 0; i < 8; ++i) xn2 = fmaf(f[i], f[i], xn2);
    }
  }
  for (int e = l16; e < E; e += 16) wm2 = fmaxf(wm2, wnorm2[e]);
#pragma unroll
  for (int off = 8; off > 0; off >>= 1) {
    xn2 += __shfl_xor_sync(0xffffffffu, xn2, off);
    wm2 = fmaxf(wm2, __shfl_xor_sync(0xffffffffu, wm2, off));
  }
  // K-th largest approximate logit: K rounds, each removes one maximum (lowest index among equals)
  unsigned taken = 0;
  float kth = -FLT_MAX;
  for (int k = 0; k < K; ++k) {
    float bv = -FLT_MAX;
    int be = 0x7fffffff;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const int e = l16 + 16 * j;
      const bool ok = (e < E) && !((taken >> j) & 1u);
      if (ok && (be == 0x7fffffff || v[j] > bv)) { bv = v[j]; be = e; }
    }
#pragma unroll
    for (int off = 8; off > 0; off >>= 1) {
      const float ov = __shfl_xor_sync(0xffffffffu, bv, off);
      const int oe = __shfl_xor_sync(0xffffffffu, be, off);
      const bool other = (oe != 0x7fffffff) && (be == 0x7fffffff || ov > bv || (ov == bv && oe < be));
      if (other) { bv = ov; be = oe; }
    }
    if (be != 0x7fffffff && (be & 15) == l16) taken |= 1u << (be >> 4);
    kth = bv;
  }
  // The error bound of this token (a little extra for the two roundings of "+ bias").  First threshold: one bound
  // (plus a sliver) below the K-th largest approximate logit - half the window the proof needs, so about ten
  // candidates instead of twelve and hardly ever more than sixteen.  The missing half is made up afterwards with
  // the exact values: see the end of the round.
  const float eps = kRfUlp * (0.5f * (float)H + 68.0f * (float)((H + 255) / 256) + 3.0f) * sqrtf(xn2 * wm2) * 1.0001f + 4.0e-7f * (1.0f + fabsf(kth));
  if (l16 == 0) s_eps[tl] = eps;
  float thr = kth - eps - 1.0e-3f * (1.0f + fabsf(kth));
  unsigned done = 0;  // bit j: the chain of expert l16 + 16 j has been run
  const int nchunk = (H + kRfChunk - 1) / kRfChunk;
  int issued = 0, consumed = 0;  // chunks over all passes: buffer = count % kRfBufs, phase = count / kRfBufs
  bool failed = false;
  // The copies are issued by one thread: the first lane of the last warp, which has chains to run only when the
  // CTA's list is full.  The warps are not held together by a barrier per step: each waits for the step's buffer,
  // runs its chains over it and reports that it has left it; the issuing thread refills a buffer when all have.
  const bool producer = threadIdx.x == NT - 32;
  auto issue = [&](int ch) {  // the producer only
    const int b = issued % kRfBufs;
    if (!mbar_wait(smem_u32(&s_empty[b]), ((uint32_t)(issued / kRfBufs) & 1u) ^ 1u, abort_flag, wait_ns)) {
      failed = true;
      s_abort = 1;
      return;
    }
    const uint32_t bar = smem_u32(&s_full[b]);
    mbar_expect_tx(bar, (uint32_t)(kRfWBytes + tpc * kRfChunk * 2));
    tma_load_2d(smem_u32(w_stage + (size_t)b * kRfWBytes), &map_w, bar, ch * kRfChunk, 0);   // rows past E, columns past H: zeros
    tma_load_2d(smem_u32(x_stage + (size_t)b * kXBytes), &map_x, bar, ch * kRfChunk, t0);    // rows past T: zeros
    if (ch + kRfAhead < nchunk)  // x comes from HBM (Wr stays in L2): ask for it well before its turn
      asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global [%0, {%1, %2}];" ::"l"(&map_x), "r"((ch + kRfAhead) * kRfChunk), "r"(t0) : "memory");
    ++issued;
  };
  // candidates of the first round, while the approximate logits are still in registers (later rounds, which are
  // rare, fetch them again: the chains' loop should not have to carry sixteen values it never uses)
  unsigned cand0 = 0;
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const int e = l16 + 16 * j;
    if (live && e < E && v[j] >= thr) cand0 |= 1u << j;
  }
  for (int round = 0; round < 3; ++round) {  // a second round is rare, a third cannot be needed
    // candidates of this round: at or above the threshold and not yet done; counted, then listed CTA-wide
    unsigned cand = cand0;
    if (round > 0) {
      cand = 0;
      if (live && thr < FLT_MAX) {
        for (int j = 0; j < 16; ++j) {
          const int e = l16 + 16 * j;
          if (e >= E || ((done >> j) & 1u)) continue;
          float a = logits[(size_t)(t0 + tl) * kRfEP + e];
          if (bias != nullptr) a = a + bias[e];
          if (a >= thr) cand |= 1u << j;
        }
      }
    }
    // The CTA's chains are numbered so that lane l of a warp gets an expert with e % 8 == l % 8: the eight lanes that
    // read shared memory together then read eight different 16-byte units whatever their rows are (numbered token by
    // token, their units met in a bank two and a half times on average).  Chain number i of bucket b is slot 8 i + b; a
    // bucket is in token order, so neighbouring lanes also read (nearly) the same token's row.  What a bucket has beyond
    // an eighth of the chains (popular experts) takes the slots that other buckets leave free.
    const int bucket = l16 & 7;  // of all of this lane's experts l16 + 16 j
    const int mine = __popc(cand), other = __shfl_xor_sync(0xffffffffu, mine, 8);  // lanes l16 and l16 ^ 8 share a bucket
    if (l16 < 8) s_ncand[tl][bucket] = (unsigned char)(mine + other);
    __syncthreads();
    int first = l16 < 8 ? 0 : other, in_bucket = 0;
    for (int i = 0; i < tpc; ++i) {
      const int n = s_ncand[i][bucket];
      if (i < tl) first += n;
      in_bucket += n;
    }
    if (tl == 0 && l16 < 8) s_total[bucket] = in_bucket;
    int total = 0;
#pragma unroll
    for (int b = 0; b < 8; ++b) total += __shfl_sync(0xffffffffu, in_bucket, b);
    if (total == 0) break;  // no token of the CTA asks for more (CTA-uniform)
    const int rows = (total + 7) / 8;
    total = 8 * rows;
    int over = 0;  // chains beyond `rows` in the buckets before this lane's
#pragma unroll
    for (int b = 0; b < 8; ++b) {
      const int n = __shfl_sync(0xffffffffu, in_bucket, b);
      if (b < bucket) over += max(0, n - rows);
    }
    for (int i = threadIdx.x; i < total; i += NT) chains[i] = 0xffff;
    __syncthreads();
    for (int j = 0, pos = first; j < 16; ++j) {
      if (!((cand >> j) & 1u)) continue;
      int slot = 8 * pos + bucket;
      if (pos >= rows) {
        int o = over + pos - rows;
        for (int b = 0; b < 8; ++b) {
          const int n = s_total[b], free = max(0, rows - n);
          if (o < free) { slot = 8 * (n + o) + b; break; }
          o -= free;
        }
      }
      ++pos;
      chains[slot] = (unsigned short)((tl << 8) | (l16 + 16 * j));
    }
    done |= cand;
    __syncthreads();
    const int passes = (total + NT - 1) / NT;
    for (int p = 0; p < passes; ++p) {
      const int sidx = p * NT + threadIdx.x;
      int e = -1, tk = 0;
      if (sidx < total && chains[sidx] != 0xffff) {
        e = chains[sidx] & 0xff;
        tk = chains[sidx] >> 8;
      }
      // shared-memory byte offsets of the eight 16-byte units of this chain's two rows inside a buffer (swizzled)
      uint32_t wo[8], xo[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        wo[q] = (uint32_t)(e >= 0 ? e : 0) * 128u + (((uint32_t)q ^ (uint32_t)(e & 7)) << 4);
        xo[q] = (uint32_t)tk * 128u + (((uint32_t)q ^ (uint32_t)(tk & 7)) << 4);
      }
      const uint32_t w_base = smem_u32(w_stage), x_base = smem_u32(x_stage);
      if (producer)  // (after a wait that ran out nothing more is issued: a buffer may still be in flight)
        for (int ch = 0; ch < kRfBufs - 1 && ch < nchunk && !failed; ++ch) issue(ch);
      float acc = 0.0f;
      for (int ch = 0; ch < nchunk; ++ch) {
        if (producer && !failed && ch + kRfBufs - 1 < nchunk) issue(ch + kRfBufs - 1);
        const int b = consumed % kRfBufs;
        // one lane per warp polls the barrier (a thousand pollers would keep the shared-memory pipe busy)
        if (lane == 0 && !failed && !mbar_wait(smem_u32(&s_full[b]), (uint32_t)(consumed / kRfBufs) & 1u, abort_flag, wait_ns)) {
          failed = true;
          s_abort = 1;
        }
        failed = __shfl_sync(0xffffffffu, (int)failed, 0) != 0;
        ++consumed;
        if (e >= 0 && !failed) {
          const uint32_t wb = w_base + (uint32_t)b * (uint32_t)kRfWBytes, xb = x_base + (uint32_t)b * (uint32_t)kXBytes;
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const uint4 xa = lds128(xb + xo[q]);
            const uint4 wa = lds128(wb + wo[q]);
            acc = fma_bf16_lo(xa.x, wa.x, acc);
            acc = fma_bf16_hi(xa.x, wa.x, acc);
            acc = fma_bf16_lo(xa.y, wa.y, acc);
            acc = fma_bf16_hi(xa.y, wa.y, acc);
            acc = fma_bf16_lo(xa.z, wa.z, acc);
            acc = fma_bf16_hi(xa.z, wa.z, acc);
            acc = fma_bf16_lo(xa.w, wa.w, acc);
            acc = fma_bf16_hi(xa.w, wa.w, acc);
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&s_empty[b]));  // this warp has left the buffer
      }
      if (e >= 0 && !failed) {
        const float exact = bias != nullptr ? acc + bias[e] : acc;
        // the error model, checked where both values are at hand: a miss is an error of this kernel, said aloud
        if (!(fabsf(exact - ls[tk * kRfEP + e]) <= s_eps[tk])) set_status(status, MOE_ERR_INTERNAL, 501);
        ls[tk * kRfEP + e] = exact;
      }
    }
    __syncthreads();
    if (s_abort) break;  // (CTA-uniform: read after the barrier)
    // The K-th largest EXACT logit among the experts done so far.  An expert that is not done has l~ below the
    // threshold, hence l < thr + eps; if that is at most the K-th exact value, none of them belongs to the K
    // largest and the token is finished.  Otherwise the threshold drops to (K-th exact - eps), which is final:
    // more exact values can only raise the K-th one.
    unsigned tkn = 0;
    float kx = -FLT_MAX;
    for (int k = 0; k < K; ++k) {
      float bv = -FLT_MAX;
      int be = 0x7fffffff;
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const int e = l16 + 16 * j;
        if (!((done >> j) & 1u) || ((tkn >> j) & 1u)) continue;
        const float xv = ls[tl * kRfEP + e];
        if (be == 0x7fffffff || xv > bv) { bv = xv; be = e; }
      }
#pragma unroll
      for (int off = 8; off > 0; off >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, bv, off);
        const int oe = __shfl_xor_sync(0xffffffffu, be, off);
        const bool other = (oe != 0x7fffffff) && (be == 0x7fffffff || ov > bv || (ov == bv && oe < be));
        if (other) { bv = ov; be = oe; }
      }
      if (be != 0x7fffffff && (be & 15) == l16) tkn |= 1u << (be >> 4);
      kx = bv;
    }
    thr = (live && thr + eps > kx) ? kx - eps : FLT_MAX;  // FLT_MAX: nothing more to do for this token
  }
  __syncthreads();
  if (s_abort) {
    // A copy that was waited for too long is still on its way: every issued copy has to land before the CTA's
    // shared memory goes away (bounded again; the copies depend on nobody).
    if (producer) {
      for (int g = 0; g < issued; ++g) {
        if (g + kRfBufs < issued) continue;  // an older fill of the same buffer: the later one's phase covers it
        const unsigned long long ts = globaltimer();
        while (!mbar_try(smem_u32(&s_full[g % kRfBufs]), (uint32_t)(g / kRfBufs) & 1u))
          if (globaltimer() - ts > wait_ns + 1000000ull) break;
      }
      set_status(status, MOE_ERR_TIMEOUT, kWaitMbarTma);
    }
    __syncthreads();
    return;
  }
  select_topk<32, kRfEP / 32>(ls, kRfEP, tvalid, t0, E, K, renorm, topk_idx, topk_w, prep.hist ? s_hist : nullptr, tp);
  route_prep_end(prep, s_hist);
}

// ---- (2') the same for batches of up to some thousand tokens ------------------------------------------
// The refine kernel above brings all of Wr to every CTA, which pays where a CTA has tens of tokens.  Here a CTA takes two
// tokens, keeps their rows of x in shared memory and fetches the rows of its candidates alone (about twenty), each lane of
// a producer warp the row of one chain, 1 KB at a time through two buffers (a bulk copy costs its issuer some fifty clocks:
// in pieces of 256 bytes they took longer than the chains, 60 us instead of 39).  One warp runs the chains, a lane each; rows
// lie 16 bytes off a multiple of 128 apart, so its 16-byte loads meet no bank twice.  What bounds it is the chain's own
// latency (4.5 cycles per h: 17 us at H 7168) where running all E chains is bound by their FMAs.  Whole router call, 256
// experts, H 7168, us, every chain / this: T 256 43 / 37, T 512 70 / 39, T 1024 99 / 70 (a second wave of CTAs).
// A CTA with more than two warps' worth of candidates (logits that differ by less than their bound, large numbers in x) brings 64
// columns of all of Wr at a time, and each of its threads runs the chains of two experts for both tokens.  The call at H 7168,
// 256 experts, us, candidates' passes alone / so / every chain in its kernel: one such CTA, T 256 and 512 183 / 83 / 48 and 75, T
// 1024 189 / 87 / 124; every CTA, T 512 324 / 107 / 75, T 1024 624 / 204 / 124.  A token of zeros, a router of zeros and a token
// with a NaN or an infinity have no need of chains: T 512 42 us (324 for zeros before), where every row is zero 22.
constexpr int kRdTokens = 2, kRdChains = 32, kRdThreads = 128, kRdBufs = 2;
constexpr int kRdMany = 2 * kRdChains;  // more candidates than this: all of Wr
constexpr int kRdWideBufs = 2, kRdWideChunk = kRfChunk, kRdWideBytes = kRfWBytes;  // boxes of 64 h of every expert's row
constexpr int kRdChunk = 512, kRdPitch = kRdChunk * 2 + 16;  // h per step; bytes from one chain's chunk to the next one's
__host__ __device__ constexpr int rd_x_pitch(int H) { return (H * 2 + 127) / 128 * 128 + 16; }
constexpr size_t rd_smem(int H) {
  return 16 + (size_t)kRdTokens * rd_x_pitch(H) + (size_t)kRdBufs * kRdChains * kRdPitch + (size_t)kRdTokens * kRfEP * (4 + 2);
}

__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}

// The K-th largest of a warp's keys (order_key; 0: none), eight per lane at experts lane + 32 j; FLT_MAX's negative if there are fewer.
__device__ __forceinline__ float rd_kth(int K, int lane, unsigned (&key)[8]) {
  unsigned bk = 0;
  for (int k = 0; k < K; ++k) {
    bk = key[0];
#pragma unroll
    for (int j = 1; j < 8; ++j) bk = max(bk, key[j]);
    bk = __reduce_max_sync(0xffffffffu, bk);
    unsigned be = 0xffffffffu;
#pragma unroll
    for (int j = 7; j >= 0; --j)
      if (key[j] == bk) be = (unsigned)(lane + 32 * j);
    be = __reduce_min_sync(0xffffffffu, be);  // one of several equal ones leaves
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (be == (unsigned)(lane + 32 * j)) key[j] = 0u;
  }
  return bk == 0u ? -FLT_MAX : __uint_as_float((bk & 0x80000000u) ? bk ^ 0x80000000u : ~bk);
}

// A token with a logit that is NaN or infinite, or without a bound, or with a bound of zero.  Three kinds need no chains (thr: FLT_MAX).
// x or Wr zero: every chain is zero, and what the tensor cores made of it.  A NaN in x makes one of every chain.  An infinity in x
// makes of every chain what the tensor cores made of the sum, unless large numbers beside it may overflow.  Of the others an
// expert whose logit or whose weights' norm is not finite is a candidate, whatever its logit, and so is every expert where that
// leaves no bound.  checked: infinity where chains are run whose values the bound says nothing of, else eps.  A warp.
struct RdUnusual { unsigned must; float eps, thr, checked; };
__device__ __noinline__ RdUnusual rd_unusual(float* l, uint32_t x, const float* wnorm2, int H, int E, float xn2, float kth, float slope, float floor) {
  constexpr uint32_t warp = 0xffffffffu;
  const int lane = threadIdx.x % 32;
  RdUnusual r = {0u, INFINITY, FLT_MAX, INFINITY};
  float wm2 = 0.0f;
  bool finite = false;  // a logit that is
  for (int e = lane, j = 0; e < E; e += 32, ++j) {
    const float n2 = wnorm2[e], v = l[e];
    if (!(n2 <= FLT_MAX) || !(v <= FLT_MAX)) r.must |= 1u << j;
    if (n2 <= FLT_MAX) wm2 = fmaxf(wm2, n2);
    finite = finite || fabsf(v) <= FLT_MAX;
  }
  for (int off = 16; off > 0; off >>= 1) wm2 = fmaxf(wm2, __shfl_xor_sync(warp, wm2, off));
  const bool any_must = __any_sync(warp, r.must != 0u);
  if (!any_must && xn2 <= FLT_MAX && (xn2 == 0.0f || wm2 == 0.0f)) return r;
  if (!(xn2 <= FLT_MAX)) {
    const bool nan = isnan(xn2);
    bool large = finite || !(wm2 <= 1.0e36f);
    for (int q = lane; q < H / 8; q += 32) {
      float f[8];
      Vec16<__nv_bfloat16>::unpack(lds128(x + (uint32_t)q * 16u), f);
#pragma unroll
      for (int i = 0; i < 8; ++i) large = large || (fabsf(f[i]) > 1.0e18f && !isinf(f[i]));
    }
    large = __any_sync(warp, large);
    if (nan || !large) {
      for (int e = lane; e < E; e += 32)
        if (nan || isnan(l[e])) l[e] = __int_as_float(0x7fffffff);
      r.must = 0u;
      return r;
    }
  }
  r.eps = slope * sqrtf(xn2 * wm2) + floor;
  r.thr = kth - r.eps - fminf(r.eps, 1.0e-3f * (1.0f + fabsf(kth)));
  if (!(r.eps <= FLT_MAX) || !(fabsf(r.thr) <= FLT_MAX)) {
    r.must = 0xffu;
    r.thr = -INFINITY;
  } else if (!any_must) {
    r.checked = r.eps;
  }
  return r;
}

// The chains of all experts for both tokens, by all threads: experts threadIdx.x and threadIdx.x + 128, 64 h of every expert's row at
// a time (62 us at H 7168 for one CTA, what an SM fetches in boxes of 128-byte rows; boxes of 128 experts or of 32 h take 85 to 108).
// Eight lanes' 16-byte loads meet different units of the swizzled rows, and the four chains of a thread take turns, FMA by FMA, or
// each would wait for itself.  Only candidates' values are used, so that what a token gets does not depend on the other.  false, for
// all threads: a wait ran out.  (Apart from the kernel, which is 3 us slower with this in it.)
struct RdEvery {
  const CUtensorMap* map_w;
  const float* bias;
  float* ls;
  uint32_t xrow, ring, bars;
  const uint32_t* cand;
  const float* eps;
  int* fills;
  volatile int* abort_flag;
  unsigned long long wait_ns;
  int* status;
  int x_pitch, H, tvalid, step;  // step: boxes so far: buffer = step % kRdWideBufs
};
__device__ __noinline__ bool rd_every_chain(const RdEvery& q) {
  const uint32_t wide = (q.ring + 1023u) & ~1023u, swizzle = (uint32_t)(threadIdx.x & 7) << 4;
  const int n = (q.H + kRdWideChunk - 1) / kRdWideChunk;
  auto fill = [&](int i) {  // (one thread; the buffer is free)
    const int b = (q.step + i) % kRdWideBufs;
    mbar_expect_tx(q.bars + 8 * b, kRdWideBytes);
    tma_load_2d(wide + b * kRdWideBytes, q.map_w, q.bars + 8 * b, i * kRdWideChunk, 0);
    *q.fills = q.step + i + 1;
  };
  if (threadIdx.x == 0)
    for (int i = 0; i < min(kRdWideBufs, n); ++i) fill(i);
  float acc[2][kRdTokens] = {};
  for (int ch = 0; ch < n; ++ch) {
    const int g = q.step + ch, b = g % kRdWideBufs;
    const bool late = !mbar_wait(q.bars + 8 * b, (uint32_t)(g / kRdWideBufs) & 1u, q.abort_flag, q.wait_ns);
    if (!late) {
      const uint32_t w0 = wide + b * kRdWideBytes + threadIdx.x * 128u, x0 = q.xrow + (uint32_t)(ch * kRdWideChunk) * 2u;
      auto eight = [&](int u) {
        uint32_t wv[2][4], xv[kRdTokens][4];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const uint4 w = lds128(w0 + i * (kRdWideBytes / 2) + ((uint32_t)(u << 4) ^ swizzle));
          wv[i][0] = w.x, wv[i][1] = w.y, wv[i][2] = w.z, wv[i][3] = w.w;
        }
#pragma unroll
        for (int t = 0; t < kRdTokens; ++t) {
          const uint4 x = lds128(x0 + (uint32_t)(t * q.x_pitch + u * 16));
          xv[t][0] = x.x, xv[t][1] = x.y, xv[t][2] = x.z, xv[t][3] = x.w;
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
#pragma unroll
          for (int c = 0; c < 2 * kRdTokens; ++c) acc[c & 1][c >> 1] = fma_bf16_lo(xv[c >> 1][j], wv[c & 1][j], acc[c & 1][c >> 1]);
#pragma unroll
          for (int c = 0; c < 2 * kRdTokens; ++c) acc[c & 1][c >> 1] = fma_bf16_hi(xv[c >> 1][j], wv[c & 1][j], acc[c & 1][c >> 1]);
        }
      };
      const int units = min(kRdWideChunk, q.H - ch * kRdWideChunk) / 8;
      if (units == kRdWideChunk / 8) {
#pragma unroll
        for (int u = 0; u < kRdWideChunk / 8; ++u) eight(u);
      } else {
        for (int u = 0; u < units; ++u) eight(u);
      }
    }
    if (__syncthreads_or(late)) return false;
    if (threadIdx.x == 0 && ch + kRdWideBufs < n) fill(ch + kRdWideBufs);
  }
#pragma unroll
  for (int t = 0; t < kRdTokens; ++t)
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int e = (int)threadIdx.x + 128 * i;
      if (t >= q.tvalid || !((q.cand[t * (kRfEP / 32) + e / 32] >> (e % 32)) & 1u)) continue;
      const float exact = q.bias != nullptr ? acc[i][t] + q.bias[e] : acc[i][t];
      float& l = q.ls[t * kRfEP + e];
      if (!(fabsf(exact - l) <= q.eps[t]) && q.eps[t] <= FLT_MAX) set_status(q.status, MOE_ERR_INTERNAL, 502);  // (the error model, as below)
      l = exact;
    }
  return true;
}

__global__ void __launch_bounds__(kRdThreads)
route_direct_kernel(const __grid_constant__ CUtensorMap map_w, const __nv_bfloat16* __restrict__ x, const __nv_bfloat16* __restrict__ wr, const float* __restrict__ bias,
                    const float* __restrict__ logits, int slices, const float* __restrict__ wnorm2, float additions, int sms, int T, int H,
                    int E, int K, int renorm, int* __restrict__ topk_idx, float* __restrict__ topk_w, const PrepArgs prep, int tp,
                    unsigned long long wait_ns, int* __restrict__ status) {
  __shared__ int s_hist[kRouteMaxExperts];
  __shared__ float s_xn2[kRdThreads / 32], s_eps[kRdTokens];
  __shared__ uint32_t s_cand[kRdTokens][kRfEP / 32];  // the tokens' candidates, where there are many
  __shared__ unsigned long long s_full[kRdBufs], s_empty[kRdBufs], s_wide[kRdWideBufs], s_x;
  __shared__ int s_total[3], s_fills, s_wide_fills, s_abort;  // chains per round; chunks and boxes whose copies have been issued
  extern __shared__ uint8_t rd_dyn[];
  uint8_t* xrow = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(rd_dyn) + 15) & ~(uintptr_t)15);
  const int x_pitch = rd_x_pitch(H);
  uint8_t* ring = xrow + kRdTokens * x_pitch;                                        // [kRdBufs][kRdChains][kRdPitch]
  static_assert(kRdBufs * kRdChains * kRdPitch >= kRdWideBufs * kRdWideBytes + 1008, "or, on 1024 bytes, [kRdWideBufs][256 experts][128 bytes]");
  float* ls = reinterpret_cast<float*>(ring + kRdBufs * kRdChains * kRdPitch);       // [kRdTokens][256]
  unsigned short* chains = reinterpret_cast<unsigned short*>(ls + kRdTokens * kRfEP);  // token << 8 | expert
  const int t0 = blockIdx.x * kRdTokens, tvalid = min(kRdTokens, T - t0);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, tl = warp;  // a warp per token for what is per token
  const bool live = tl < tvalid;
  // the CTAs of an SM run their chains on different schedulers
  const int chain_warp = (int)(blockIdx.x / (unsigned)sms) % 4, load_warp = (chain_warp + 1) % 4;
  if (threadIdx.x == 0) {
    for (int b = 0; b < kRdBufs; ++b) {
      mbar_init(smem_u32(&s_full[b]), 1);
      mbar_init(smem_u32(&s_empty[b]), 1);
    }
    for (int b = 0; b < kRdWideBufs; ++b) mbar_init(smem_u32(&s_wide[b]), 1);
    mbar_init(smem_u32(&s_x), 1);
    s_abort = s_fills = s_wide_fills = s_total[0] = s_total[1] = s_total[2] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    // (x and Wr were complete before the kernel in front of this one could start)
    mbar_expect_tx(smem_u32(&s_x), (uint32_t)(tvalid * H * 2));
    for (int i = 0; i < tvalid; ++i) bulk_load(smem_u32(xrow + i * x_pitch), x + (size_t)(t0 + i) * H, (uint32_t)(H * 2), smem_u32(&s_x));
  }
  __syncthreads();
  volatile int* abort_flag = &s_abort;
  bool failed = !mbar_wait(smem_u32(&s_x), 0u, abort_flag, wait_ns);
  if (failed) s_abort = 1;
  {  // |x_t|^2: two warps per token
    const int t = warp / 2;
    float s = 0.0f;
    uint32_t bits = 0;
    if (t < tvalid && !failed)
      for (int q = (warp % 2) * 32 + lane; q < H / 8; q += 64) {
        float f[8];
        const uint4 u = lds128(smem_u32(xrow + t * x_pitch) + (uint32_t)q * 16u);
        bits |= u.x | u.y | u.z | u.w;
        Vec16<__nv_bfloat16>::unpack(u, f);
#pragma unroll
        for (int i = 0; i < 8; ++i) s = fmaf(f[i], f[i], s);
      }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    const bool zeros = __all_sync(0xffffffffu, (bits & 0x7fff7fffu) == 0u);
    if (lane == 0) s_xn2[warp] = s == 0.0f && !zeros ? FLT_MIN : s;  // (zero: a row of zeros)
  }
  pdl_wait();
  pdl_trigger();
  route_prep_begin(prep, s_hist);
  // the slices of the approximate logits, four experts per thread, and the bias the way the chain's value gets it
  for (int i = threadIdx.x; i < tvalid * (kRfEP / 4); i += kRdThreads) {
    const int t = i / (kRfEP / 4), e = i % (kRfEP / 4) * 4;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    const float4* src = reinterpret_cast<const float4*>(logits + (size_t)(t0 + t) * kRfEP + e);
    if (e < E) {
#pragma unroll 16
      for (int z = 0; z < slices; ++z) {
        const float4 v = __ldcg(src + (size_t)z * T * (kRfEP / 4));
        a.x += v.x; a.y += v.y; a.z += v.z; a.w += v.w;
      }
    }
    const float f[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) ls[t * kRfEP + e + q] = e + q >= E ? -FLT_MAX : bias != nullptr ? f[q] + bias[e + q] : f[q];
  }
  __syncthreads();
  const float* row = ls + (live ? tl : 0) * kRfEP;
  unsigned must = 0;                   // bit j: expert lane + 32 j is a candidate whatever its logit
  float v[8], thr = 0.0f, eps = 0.0f;  // the approximate logits of experts lane + 32 j
  if (live) {
    float wm2 = 0.0f;
    unsigned key[8];
    bool unusual = false;  // a logit that is NaN or infinite.  (A bias of minus infinity makes none: such an expert's logit is that in any case.)
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int e = lane + 32 * j;
      v[j] = row[e];
      key[j] = e < E ? max(order_key(v[j]), 1u) : 0u;
      unusual = unusual || (e < E && !(v[j] <= FLT_MAX));
      if (e < E) wm2 = fmaxf(wm2, wnorm2[e]);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) wm2 = fmaxf(wm2, __shfl_xor_sync(0xffffffffu, wm2, off));
    const float kth = rd_kth(K, lane, key);
    // (the same first threshold and the same proof as in the refine kernel)
    const float xn2 = s_xn2[2 * tl] + s_xn2[2 * tl + 1], norms = xn2 * wm2;
    const float slope = kRfUlp * (0.5f * (float)H + additions) * 1.0001f, floor = 4.0e-7f * (1.0f + fabsf(kth));
    eps = slope * sqrtf(norms) + floor;
    float checked = eps;
    // (below the bound a sliver, so that the candidates' exact values settle the matter in one round; the bound itself is enough for that)
    thr = kth - eps - fminf(eps, 1.0e-3f * (1.0f + fabsf(kth)));
    unusual = __any_sync(0xffffffffu, unusual);
    if (unusual || !(eps <= FLT_MAX) || !(norms > 0.0f)) {  // (the same for all lanes)
      const RdUnusual u = rd_unusual(ls + tl * kRfEP, smem_u32(xrow) + (uint32_t)(tl * x_pitch), wnorm2, H, E, xn2, kth, slope, floor);
      must = u.must;
      eps = u.eps;
      thr = u.thr;
      checked = u.checked;
    }
    if (lane == 0) s_eps[tl] = checked;
  }
  unsigned done = 0;  // bit j: the chain of expert lane + 32 j has been run
  const int nchunk = (H + kRdChunk - 1) / kRdChunk;
  int step = 0, wide_step = 0;  // chunks, boxes so far over all passes: buffer = step % kRdBufs, wide_step % kRdWideBufs
  for (int round = 0; round < 3; ++round) {  // a second round is rare, a third cannot be needed
    unsigned cand = 0;
    if (live && thr < FLT_MAX) {
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (lane + 32 * j < E && (((must >> j) & 1u) || v[j] >= thr) && !((done >> j) & 1u)) cand |= 1u << j;
    }
    done |= cand;
    if (cand != 0) {
      int at = atomicAdd(&s_total[round], __popc(cand));
      for (unsigned c = cand; c != 0; c &= c - 1) chains[at++] = (unsigned short)((tl << 8) | (lane + 32 * (__ffs(c) - 1)));
    }
    __syncthreads();
    const int total = s_total[round];
    if (total == 0 || s_abort) break;  // no token of the CTA asks for more (CTA-uniform)
    if (total > kRdMany) {
      if (live)
        for (int j = 0; j < kRfEP / 32; ++j) {
          const uint32_t word = __ballot_sync(0xffffffffu, (cand >> j) & 1u);
          if (lane == 0) s_cand[tl][j] = word;
        }
      __syncthreads();
      failed = !rd_every_chain(RdEvery{&map_w, bias, ls, smem_u32(xrow), smem_u32(ring), smem_u32(s_wide), &s_cand[0][0], s_eps, &s_wide_fills, abort_flag,
                                       wait_ns, status, x_pitch, H, tvalid, wide_step});
      wide_step += (H + kRdWideChunk - 1) / kRdWideChunk;
      if (failed) s_abort = 1;
    } else
    for (int p = 0; p < total; p += kRdChains, step += nchunk) {
      const int n = min(kRdChains, total - p);
      const int mine = lane < n ? chains[p + lane] : -1, e = mine & 0xff, tk = (mine >> 8) & 0xff;
      if (warp == load_warp) {
        for (int ch = 0; ch < nchunk && !failed; ++ch) {
          const int g = step + ch, b = g % kRdBufs;
          if (!warp_agrees(mbar_wait(smem_u32(&s_empty[b]), ((uint32_t)(g / kRdBufs) & 1u) ^ 1u, abort_flag, wait_ns))) { failed = true; break; }
          const uint32_t bytes = (uint32_t)min(kRdChunk, H - ch * kRdChunk) * 2u;
          if (lane == 0) {
            mbar_expect_tx(smem_u32(&s_full[b]), bytes * (uint32_t)n);
            s_fills = g + 1;
          }
          __syncwarp();
          if (mine >= 0)
            bulk_load(smem_u32(ring + (b * kRdChains + lane) * kRdPitch), wr + (size_t)e * H + ch * kRdChunk, bytes, smem_u32(&s_full[b]));
        }
        if (failed) s_abort = 1;
      } else if (warp == chain_warp) {
        float acc = 0.0f;
        const uint32_t w0 = smem_u32(ring) + (uint32_t)lane * kRdPitch, x0 = smem_u32(xrow) + (uint32_t)(mine >= 0 ? tk : 0) * (uint32_t)x_pitch;
        auto eight = [&](const uint4& xa, const uint4& wa) {
          acc = fma_bf16_lo(xa.x, wa.x, acc);
          acc = fma_bf16_hi(xa.x, wa.x, acc);
          acc = fma_bf16_lo(xa.y, wa.y, acc);
          acc = fma_bf16_hi(xa.y, wa.y, acc);
          acc = fma_bf16_lo(xa.z, wa.z, acc);
          acc = fma_bf16_hi(xa.z, wa.z, acc);
          acc = fma_bf16_lo(xa.w, wa.w, acc);
          acc = fma_bf16_hi(xa.w, wa.w, acc);
        };
        for (int ch = 0; ch < nchunk && !failed; ++ch) {
          const int g = step + ch, b = g % kRdBufs;
          if (!warp_agrees(mbar_wait(smem_u32(&s_full[b]), (uint32_t)(g / kRdBufs) & 1u, abort_flag, wait_ns))) { failed = true; break; }
          const uint32_t wb = w0 + (uint32_t)(b * kRdChains * kRdPitch), xb = x0 + (uint32_t)(ch * kRdChunk * 2);
          const int units = min(kRdChunk, H - ch * kRdChunk) / 8;
          if (units == kRdChunk / 8) {
            uint4 xr[2][4], wv[2][4];  // the next four units' loads go out before this four's chain of 32 FMAs
#pragma unroll
            for (int i = 0; i < 4; ++i) { xr[0][i] = lds128(xb + 16u * i); wv[0][i] = lds128(wb + 16u * i); }
#pragma unroll 4
            for (int q = 0; q < kRdChunk / 32; ++q) {
              if (q + 1 < kRdChunk / 32)
#pragma unroll
                for (int i = 0; i < 4; ++i) { xr[(q + 1) & 1][i] = lds128(xb + 16u * (4 * q + 4 + i)); wv[(q + 1) & 1][i] = lds128(wb + 16u * (4 * q + 4 + i)); }
#pragma unroll
              for (int i = 0; i < 4; ++i) eight(xr[q & 1][i], wv[q & 1][i]);
            }
          } else {
            for (int q = 0; q < units; ++q) eight(lds128(xb + 16u * q), lds128(wb + 16u * q));
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(smem_u32(&s_empty[b]));
        }
        if (failed) s_abort = 1;
        if (mine >= 0 && !failed) {
          const float exact = bias != nullptr ? acc + bias[e] : acc;
          // the error model, checked where both values are at hand: a miss is an error of this kernel, said aloud
          if (!(fabsf(exact - ls[tk * kRfEP + e]) <= s_eps[tk]) && s_eps[tk] <= FLT_MAX) set_status(status, MOE_ERR_INTERNAL, 502);
          ls[tk * kRfEP + e] = exact;
        }
      }
    }
    __syncthreads();
    if (s_abort) break;  // (CTA-uniform: it is set in the passes alone)
    // The K-th largest EXACT logit so far decides whether more chains are wanted: see the refine kernel.
    if (live && thr < FLT_MAX) {
      unsigned key[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) key[j] = ((done >> j) & 1u) ? max(order_key(row[lane + 32 * j]), 1u) : 0u;
      const float kx = rd_kth(K, lane, key);
      thr = thr + eps > kx ? kx - eps : FLT_MAX;
    } else {
      thr = FLT_MAX;
    }
  }
  __syncthreads();
  if (s_abort) {
    // a copy that was waited for too long is still on its way: it has to land before the CTA's shared memory goes away
    if (threadIdx.x == 0) {
      auto settle = [&](unsigned long long* bar, uint32_t parity) {
        const unsigned long long ts = globaltimer();
        while (!mbar_try(smem_u32(bar), parity))
          if (globaltimer() - ts > wait_ns + 1000000ull) break;
      };
      settle(&s_x, 0u);
      for (int g = max(0, s_fills - kRdBufs); g < s_fills; ++g) settle(&s_full[g % kRdBufs], (uint32_t)(g / kRdBufs) & 1u);
      for (int g = max(0, s_wide_fills - kRdWideBufs); g < s_wide_fills; ++g) settle(&s_wide[g % kRdWideBufs], (uint32_t)(g / kRdWideBufs) & 1u);
    }
    if (threadIdx.x == 0) set_status(status, MOE_ERR_TIMEOUT, kWaitMbarTma);
    __syncthreads();
    return;
  }
  select_topk<32, kRfEP / 32>(ls, kRfEP, tvalid, t0, E, K, renorm, topk_idx, topk_w, prep.hist ? s_hist : nullptr, tp);
  route_prep_end(prep, s_hist);
}

// ---- host side ----------------------------------------------------------------------------------------
bool route_filter_applies(const moe_plan* p) {
  return p->cfg.dtype == MOE_DTYPE_BF16 && p->route_E > 64 && p->route_E <= kRfEP && p->cfg.route_filter >= 0 &&
         p->s.route_logits != nullptr;
}

// The slices of h that the approximate logits are computed in: as many CTAs as SMs, of four steps of 64 columns at least, and
// not more than sixteen (their reader sums them).
int route_direct_slices(int experts, int tokens, int H) {
  const int tiles = (tokens + kTileRows - 1) / kTileRows * ((experts + 127) / 128), steps = (H + kBK - 1) / kBK;
  const int per = (steps + max(1, min(min(148 / tiles, steps / 4), 16)) - 1) / max(1, min(min(148 / tiles, steps / 4), 16));
  return (steps + per - 1) / per;
}

int launch_route_direct(moe_plan* p, const void* x, const void* wr, const float* bias, int* topk_idx, float* topk_w,
                        const PrepArgs& prep, cudaStream_t st) {
  const moe_config_t& c = p->cfg;
  EncodeTiledFn enc;
  int rc = get_encoder(p, &enc);
  if (rc != MOE_OK) return rc;
  CUtensorMap mx, mwh, mwide;
  if ((rc = make_map_2d(enc, &mx, x, (uint64_t)c.T, (uint64_t)c.H, kTileRows)) != MOE_OK) return rc;
  if ((rc = make_map_2d(enc, &mwh, wr, (uint64_t)p->route_E, (uint64_t)c.H, 128)) != MOE_OK) return rc;
  if ((rc = make_map_2d(enc, &mwide, wr, (uint64_t)p->route_E, (uint64_t)c.H, kRfEP)) != MOE_OK) return rc;
  static SmemAttrOnce once, once_b;
  if (ensure_dynamic_smem(route_tc_logits_kernel, kTcSmem, p->device, once) != cudaSuccess) return MOE_ERR_CUDA;
  if (ensure_dynamic_smem(route_direct_kernel, rd_smem(c.H), p->device, once_b) != cudaSuccess) return MOE_ERR_CUDA;
  const unsigned long long wait_ns = c.wait_limit_ns ? c.wait_limit_ns : kDefaultWaitNs;
  const int slices = p->s.route_slices, steps = (c.H + kBK - 1) / kBK, per = (steps + slices - 1) / slices;
  if (launch_maybe_pdl(false, route_tc_logits_kernel, dim3((c.T + kTileRows - 1) / kTileRows, (p->route_E + 127) / 128, slices),
                       dim3(kTcThreads), kTcSmem, st, mx, mwh, (const __nv_bfloat16*)wr, c.T, c.H, p->route_E, p->s.route_logits,
                       p->s.route_wnorm2, wait_ns, p->s.status) != cudaSuccess)
    return MOE_ERR_CUDA;
  // the additions of the error model: 17 per MMA of an accumulator, the four accumulators' sum, the slices'
  const float additions = 68.0f * (float)((per + 3) / 4) + 3.0f + (float)(slices - 1);
  if (launch_pdl(route_direct_kernel, dim3((c.T + kRdTokens - 1) / kRdTokens), dim3(kRdThreads), rd_smem(c.H), st, mwide,
                 (const __nv_bfloat16*)x, (const __nv_bfloat16*)wr, bias, (const float*)p->s.route_logits, slices,
                 (const float*)p->s.route_wnorm2, additions, p->sm_count > 0 ? p->sm_count : 148, c.T, c.H, p->route_E, p->route_K,
                 c.renormalize, topk_idx, topk_w, prep, p->tp, wait_ns, p->s.status) != cudaSuccess)
    return MOE_ERR_CUDA;
  p->launches += 2;
  return 0;
}

int launch_route_filter(moe_plan* p, const void* x, const void* wr, const float* bias, int* topk_idx, float* topk_w,
                        const PrepArgs& prep, cudaStream_t st) {
  const moe_config_t& c = p->cfg;
  EncodeTiledFn enc;
  int rc = get_encoder(p, &enc);
  if (rc != MOE_OK) return rc;
  CUtensorMap mx, mw;
  if ((rc = make_map_2d(enc, &mx, x, (uint64_t)c.T, (uint64_t)c.H, kTileRows)) != MOE_OK) return rc;
  if ((rc = make_map_2d(enc, &mw, wr, (uint64_t)p->route_E, (uint64_t)c.H, kRfEP)) != MOE_OK) return rc;
  CUtensorMap mwh;  // half of the experts per box, for the filter's CTAs
  if ((rc = make_map_2d(enc, &mwh, wr, (uint64_t)p->route_E, (uint64_t)c.H, 128)) != MOE_OK) return rc;
  static SmemAttrOnce once;
  if (ensure_dynamic_smem(route_tc_logits_kernel, kTcSmem, p->device, once) != cudaSuccess) return MOE_ERR_CUDA;
  const unsigned long long wait_ns = c.wait_limit_ns ? c.wait_limit_ns : kDefaultWaitNs;
  const int grid_a = (c.T + kTileRows - 1) / kTileRows;
  // the first kernel of the layer is launched plainly (see launch_wide_tmt), the second one behind it
  if (launch_maybe_pdl(false, route_tc_logits_kernel, dim3(grid_a, (p->route_E + 127) / 128), dim3(kTcThreads), kTcSmem, st, mx, mwh,
                       (const __nv_bfloat16*)wr, c.T, c.H, p->route_E, p->s.route_logits, p->s.route_wnorm2, wait_ns,
                       p->s.status) != cudaSuccess)
    return MOE_ERR_CUDA;
  // Tokens per CTA (even: a warp has two): the time is about (waves of CTAs over the SMs) x (tokens + what streaming all
  // of Wr costs a CTA, 10 tokens' worth).
  const int sms = p->sm_count > 0 ? p->sm_count : 148;
  int tpc = 64;
  long long best = 1ll << 60;
  for (int i = 64; i >= 12; i -= 2) {  // (8 tokens per CTA measure slower than 16: T 1024 117 against 110 us)
    const long long ctas = (c.T + i - 1) / i, cost = (ctas + sms - 1) / sms * (i + 10);
    if (cost < best) { best = cost; tpc = i; }
  }
  static SmemAttrOnce once_b[2];
  auto refine = [&](auto kern, SmemAttrOnce& attr) -> int {
    CUtensorMap mxb;  // the tokens' rows of x, one CTA's worth per box
    int r = make_map_2d(enc, &mxb, x, (uint64_t)c.T, (uint64_t)c.H, (uint32_t)tpc);
    if (r != MOE_OK) return r;
    if (ensure_dynamic_smem(kern, rf_smem(tpc), p->device, attr) != cudaSuccess) return MOE_ERR_CUDA;
    return launch_pdl(kern, dim3((c.T + tpc - 1) / tpc), dim3(tpc * 16), rf_smem(tpc), st, mw, mxb, (const __nv_bfloat16*)x, bias,
                      (const float*)p->s.route_logits, (const float*)p->s.route_wnorm2, tpc, c.T, c.H, p->route_E, p->route_K,
                      c.renormalize, topk_idx, topk_w, prep, p->tp, wait_ns, p->s.status) == cudaSuccess
               ? 0 : MOE_ERR_CUDA;
  };
  rc = tpc > 32 ? refine(route_refine_kernel<64>, once_b[0]) : refine(route_refine_kernel<32>, once_b[1]);
  if (rc != 0) return rc;
  p->launches += 2;
  return 0;
}

}  // namespace moehub
