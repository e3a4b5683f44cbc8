// What every router kernel shares: the selection of the K largest logits of a token with its softmax weights,
// and the side job of resetting the dispatch's per-call state (see PrepArgs).
#pragma once
#include <float.h>

#include "common.cuh"

namespace moehub {

// The fp32 chain on bf16 data: acc + x * w with the exact product and one rounding - the same bits as widening both
// operands to fp32 and one fused multiply-add, without the widening instructions.  lo / hi: the half of a 32-bit word.
__device__ __forceinline__ float fma_bf16_lo(uint32_t x, uint32_t w, float acc) {
  float d;
  asm("{\n\t.reg .b16 xl, xh, wl, wh;\n\t"
      "mov.b32 {xl, xh}, %1;\n\tmov.b32 {wl, wh}, %2;\n\t"
      "fma.rn.f32.bf16 %0, xl, wl, %3;\n\t}"
      : "=f"(d) : "r"(x), "r"(w), "f"(acc));
  return d;
}
__device__ __forceinline__ float fma_bf16_hi(uint32_t x, uint32_t w, float acc) {
  float d;
  asm("{\n\t.reg .b16 xl, xh, wl, wh;\n\t"
      "mov.b32 {xl, xh}, %1;\n\tmov.b32 {wl, wh}, %2;\n\t"
      "fma.rn.f32.bf16 %0, xh, wh, %3;\n\t}"
      : "=f"(d) : "r"(x), "r"(w), "f"(acc));
  return d;
}
// A float as an unsigned number of the same order (-0 and +0 equal), so that an integer reduction finds the maximum.
__device__ __forceinline__ unsigned order_key(float v) {
  const unsigned u = __float_as_uint(v + 0.0f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// Maximum / minimum / sum over the G neighbouring lanes of a token (a whole warp: one instruction for the integers).
template <int G> __device__ __forceinline__ unsigned group_max(unsigned v) {
  if (G == 32) return __reduce_max_sync(0xffffffffu, v);
#pragma unroll
  for (int off = G / 2; off > 0; off >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, off));
  return v;
}
template <int G> __device__ __forceinline__ unsigned group_min(unsigned v) {
  if (G == 32) return __reduce_min_sync(0xffffffffu, v);
#pragma unroll
  for (int off = G / 2; off > 0; off >>= 1) v = min(v, __shfl_xor_sync(0xffffffffu, v, off));
  return v;
}
template <int G> __device__ __forceinline__ float group_sum(float v) {
#pragma unroll
  for (int off = G / 2; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

// G lanes per token (8, 16 or a whole warp): the token's logits sit in registers (NJ per lane, experts lane + G j);
// K rounds of an arg-max (largest value, then lowest index), then the softmax weights of the picks.  ls: rows of
// `pitch` logits (shared or global memory); row tl is token t0 + tl.
// s_hist (shared memory, [E], or nullptr): every pick is also counted per expert.
// tp > 1 (expert + tensor parallelism, paper Section VII): every pick is listed once per TP shard, as the
// virtual expert e*tp + s with the pick's weight, so that the dispatch stores the row into every shard's region.
template <int G, int NJ>
__device__ __forceinline__ void select_topk(const float* ls, int pitch, int tvalid, int t0, int E, int K, int renorm,
                                            int* __restrict__ topk_idx, float* __restrict__ topk_w, int* s_hist, int tp) {
  constexpr int PER_WARP = 32 / G;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % G, sub = threadIdx.x % 32 / G;
  for (int base = warp * PER_WARP; base < tvalid; base += blockDim.x / 32 * PER_WARP) {
    const int tl = base + sub;
    const bool live = tl < tvalid;  // (the other tokens of the warp keep it in the shuffles)
    const float* row = ls + (live ? tl : base) * pitch;
    float v[NJ];
    unsigned key[NJ];  // 0: no expert, or picked already
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      const int e = lane + G * j;
      v[j] = (e < E) ? row[e] : -FLT_MAX;
      key[j] = (e < E) ? max(order_key(v[j]), 1u) : 0u;
    }
    float my_v = 0.0f, m = 0.0f;
    int my_e = 0;
    for (int k = 0; k < K; ++k) {
      unsigned bk = key[0];
#pragma unroll
      for (int j = 1; j < NJ; ++j) bk = max(bk, key[j]);
      bk = group_max<G>(bk);
      unsigned be = 0xffffffffu;
#pragma unroll
      for (int j = NJ - 1; j >= 0; --j)
        if (key[j] == bk) be = (unsigned)(lane + G * j);
      be = group_min<G>(be);
#pragma unroll
      for (int j = 0; j < NJ; ++j)
        if (be == (unsigned)(lane + G * j)) key[j] = 0u;
      const float bv = row[be];
      if (k == 0) m = bv;
      if (lane == k) { my_e = (int)be; my_v = bv; }
    }
    float z = 0.0f;
#pragma unroll
    for (int j = 0; j < NJ; ++j)
      if (lane + G * j < E) z += expf(v[j] - m);
    z = group_sum<G>(z);
    float p = (lane < K) ? expf(my_v - m) / z : 0.0f;
    if (renorm) p = p / group_sum<G>(p);
    if (lane < K && live) {
      for (int sh = 0; sh < tp; ++sh) {
        const size_t o = ((size_t)(t0 + tl) * K + lane) * tp + sh;
        topk_idx[o] = my_e * tp + sh;
        topk_w[o] = p;
        if (s_hist != nullptr) atomicAdd(&s_hist[my_e * tp + sh], 1);
      }
    }
  }
}

// The side job of a router that is followed by an ordered dispatch (see PrepArgs): before the chains, clear
// the per-call counters; after the picks, add this CTA's rows per expert to the global counts.
constexpr int kRouteMaxExperts = 256;
__device__ __forceinline__ void route_prep_begin(const PrepArgs& prep, int* s_hist) {
  if (prep.nfill == 0) return;
  for (int e = threadIdx.x; e < kRouteMaxExperts; e += blockDim.x) s_hist[e] = 0;
  prep_reset(prep, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}
__device__ __forceinline__ void route_prep_end(const PrepArgs& prep, const int* s_hist) {
  if (prep.hist == nullptr) return;
  __syncthreads();
  for (int e = threadIdx.x; e < prep.E; e += blockDim.x)
    if (s_hist[e] != 0) atomicAdd(&prep.hist[e], s_hist[e]);
}

}  // namespace moehub
