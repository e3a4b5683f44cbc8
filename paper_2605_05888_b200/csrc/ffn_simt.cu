// Step 3 of the MoE layer (paper Section II-A, expert computation) on plain fp32 FMA units: S = silu(A*Wg^T) .* (A*Wu^T)
// into the intermediate buffer, then O = S*Wd^T, two launches.  Tiles without an owner exit at once, so the weights of
// experts that received no rows are never read.
//
// Two kernels.  ffn_fp32_kernel is the path of dtype fp32 for little work and for few rows per expert (the other shapes go
// to the tensor cores, split into bf16 numbers: ffn_split.cu).  ffn_simt_kernel, slow and simple, is a second, independent device implementation to check the tcgen05
// kernel against on bf16 data (ffn_kernel = 1).
#include "tc_common.cuh"

namespace moehub {

constexpr int kSimtThreads = 256;
constexpr int kSimtBN = 64;
constexpr int kSimtBK = 16;

template <typename XT, bool SWIGLU>
__global__ void __launch_bounds__(kSimtThreads)
ffn_simt_kernel(const XT* __restrict__ A, int lda, const int* __restrict__ tile_expert,
                const XT* __restrict__ B1, const XT* __restrict__ B2, size_t expert_stride, int tp,
                size_t shard_offset, int ldb, int N, int Kd, XT* __restrict__ C, int ldc, int E) {
  const int p = blockIdx.y;
  pdl_wait();
  pdl_trigger();
  const int e = tile_expert[p];
  if (e < 0 || e >= E) return;  // no owner, or no expert at all (a caller's own table): nothing of the weights is read
  const int n0 = blockIdx.x * kSimtBN;
  const size_t row0 = (size_t)p * kTileRows;
  // e is a virtual expert: shard e % tp of expert e / tp (tp = 1: the expert itself)
  const size_t base = (size_t)(e / tp) * expert_stride + (size_t)(e % tp) * shard_offset;
  const XT* b1 = B1 + base;
  const XT* b2 = SWIGLU ? B2 + base : nullptr;
  __shared__ float As[kSimtBK][kTileRows + 1];
  __shared__ float Bs[kSimtBK][kSimtBN + 1];
  __shared__ float Bs2[SWIGLU ? kSimtBK : 1][kSimtBN + 1];
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  float acc[8][4], acc2[SWIGLU ? 8 : 1][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      acc[i][j] = 0.0f;
      if (SWIGLU) acc2[i][j] = 0.0f;
    }
  for (int k0 = 0; k0 < Kd; k0 += kSimtBK) {
#pragma unroll
    for (int i = 0; i < kTileRows * kSimtBK / kSimtThreads; ++i) {
      const int idx = threadIdx.x + i * kSimtThreads;
      const int r = idx / kSimtBK, kk = idx % kSimtBK;
      As[kk][r] = (k0 + kk < Kd) ? to_float(A[(row0 + r) * lda + k0 + kk]) : 0.0f;
    }
#pragma unroll
    for (int i = 0; i < kSimtBN * kSimtBK / kSimtThreads; ++i) {
      const int idx = threadIdx.x + i * kSimtThreads;
      const int r = idx / kSimtBK, kk = idx % kSimtBK;
      const bool ok = (n0 + r < N) && (k0 + kk < Kd);
      Bs[kk][r] = ok ? to_float(b1[(size_t)(n0 + r) * ldb + k0 + kk]) : 0.0f;
      if (SWIGLU) Bs2[kk][r] = ok ? to_float(b2[(size_t)(n0 + r) * ldb + k0 + kk]) : 0.0f;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < kSimtBK; ++kk) {
      float a[8], b[4], c[4];
#pragma unroll
      for (int i = 0; i < 8; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        b[j] = Bs[kk][tx + 16 * j];
        if (SWIGLU) c[j] = Bs2[kk][tx + 16 * j];
      }
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          acc[i][j] = __fmaf_rn(a[i], b[j], acc[i][j]);
          if (SWIGLU) acc2[i][j] = __fmaf_rn(a[i], c[j], acc2[i][j]);
        }
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = n0 + tx + 16 * j;
      if (n >= N) continue;
      float v = acc[i][j];
      if (SWIGLU) v = v / (1.0f + expf(-v)) * acc2[i][j];
      C[(row0 + ty + 16 * i) * ldc + n] = from_float<XT>(v);
    }
}

// ---- dtype fp32 ----------------------------------------------------------------------------------------
// Bound by fp32 FMA issue (128 per clock and SM).  A CTA computes 2 TM WR rows of a tile x 64 TN / WR columns (GEMM1:
// half of them gate, half up columns of the same f); a warp has 2 TM rows and 16 TN columns, a lane TM x TN results.
// Operands stay in their natural K-major rows: TMA brings 128 bytes (32 k) of every row per stage (128-byte swizzle), a lane reads 16 bytes
// (4 k) of its TM rows and TN columns - two pipe cycles each, lanes of a warp being 2 row groups x 16 column groups -
// for TM x TN x 2 packed FMAs (fma.rn.f32x2 on pairs of neighbouring k: a result is the sum of its even and its odd k).
// With scalar FMAs half of them found their accumulator in the register bank of the operand that changes (the four k of
// a 16-byte load alternate between the banks) and ran at two thirds of the rate; an aligned pair spans both banks.  A
// lane of the first warp issues the copies on the side (a warp of its own would cost the others a third of their
// registers); the warps wait per stage on its mbarrier.  A warp whose rows a partly filled tile does not have leaves at
// once.
// Measured against the plain 128 x 64 kernel above on fp32 data: T 1000, H 1024, 16 experts, top-2,
// F 2048: whole layer 1311 -> 735 us (801 with scalar FMAs); T 256, H 128, 8 experts, top-2, F 256: 96 -> 33 us.
constexpr int kF32Warps = 4;
constexpr int kF32Threads = 32 * kF32Warps;
constexpr int kF32K = 32;  // k per stage
// stages and CTAs per SM: 8 x 8 results fill the registers with two CTAs, smaller tiles fit three
template <int TM, int TN, int WR> constexpr int kF32Stages = TM * TN == 32 || WR == 1 ? 3 : 4;
template <int TM, int TN, int WR> constexpr int kF32Ctas = TM * TN == 64 || WR == 1 ? 2 : 3;
template <int TM, int TN, int WR> constexpr int kF32StageBytes = (WR * 2 * TM + kF32Warps / WR * 16 * TN) * kF32K * 4;

struct Fp32Params {
  const int* tile_expert;  // [P]
  const int* tile_count;   // [P] rows per tile, or nullptr
  const int* rows_done;
  int total_rows;
  int P, E, tp, N, Kd;     // tiles, experts (TP shards counted), columns of the result, length of the sums
  float* C;                // [P * 128, N]
  unsigned long long wait_ns;
  int* status;
};

__device__ __forceinline__ void lds_k4(uint32_t addr, unsigned long long& lo, unsigned long long& hi) {
  asm volatile("ld.shared.v2.u64 {%0, %1}, [%2];" : "=l"(lo), "=l"(hi) : "r"(addr));
}
__device__ __forceinline__ void fma_x2(unsigned long long& acc, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
__device__ __forceinline__ float sum_x2(unsigned long long v) {
  return __uint_as_float((uint32_t)v) + __uint_as_float((uint32_t)(v >> 32));
}

struct Fp32Shared {
  unsigned long long full[4], empty[4];
  int abort;
  int col, tile, part, tile_rows;  // the block (col < 0: none)
  int next;                        // the CTA's next block, -1: there is none
};

// Block number id in the order described below: where it lies.  Warp 0 calls; the others see it behind a barrier.
template <int BM, int NOUT>
__device__ __forceinline__ void fp32_find_block(const Fp32Params& p, Fp32Shared& s, int id) {
  constexpr int kParts = kTileRows / BM;
  const int lane = threadIdx.x % 32;
  const bool counted = p.tile_count != nullptr && *p.rows_done >= p.total_rows;
  auto blocks_of = [&](int t) {  // a tile without an owner, or owned by no expert at all (a caller's own table), has none
    const int e = t < p.P ? p.tile_expert[t] : -1;
    return e < 0 || e >= p.E ? 0 : counted ? (min(kTileRows, p.tile_count[t]) + BM - 1) / BM : kParts;
  };
  int total = 0;
  for (int t = lane; t < p.P; t += 32) total += blocks_of(t);
  total = __reduce_add_sync(0xffffffffu, total);
  int col = -1, block = 0;
  if (total > 0) {
    col = id / total;
    block = id - col * total;
  }
  const int cols = (p.N + NOUT - 1) / NOUT;
  if (col >= cols) col = -1;
  if (lane == 0) {
    s.col = col;
    s.next = (long long)id + gridDim.x < (long long)total * cols ? id + (int)gridDim.x : -1;
  }
  for (int t = lane, before = 0; col >= 0 && before <= block; t += 32) {
    const int mine = blocks_of(t);
    int incl = mine;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int o = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += o;
    }
    const int first = before + incl - mine;
    if (block >= first && block < first + mine) {
      s.tile = t;
      s.part = block - first;
      s.tile_rows = counted ? min(kTileRows, p.tile_count[t]) : kTileRows;
    }
    before += __shfl_sync(0xffffffffu, incl, 31);
  }
}

// The block in s.  Warps without rows leave at once; a wait that ran out is left in s.abort.
template <int TM, int TN, int WR, bool SWIGLU>
__device__ __forceinline__ void fp32_block(const CUtensorMap& map_a, const CUtensorMap& map_b1, const CUtensorMap& map_b2,
                                           const Fp32Params& p, Fp32Shared& s, uint8_t* ring) {
  constexpr int WN = kF32Warps / WR, BM = WR * 2 * TM, BN = WN * 16 * TN;  // rows and columns of B per CTA
  constexpr int NOUT = SWIGLU ? BN / 2 : BN;             // columns of the result per CTA
  constexpr int kA = BM * kF32K * 4, kStage = kF32StageBytes<TM, TN, WR>;
  constexpr int kStages = kF32Stages<TM, TN, WR>;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int n0 = s.col * NOUT, tile = s.tile, part = s.part, rows = min(s.tile_rows - part * BM, BM);
  const int e = p.tile_expert[tile];
  const int rw = warp % WR, cw = warp / WR;
  const int live_rows = (rows + 2 * TM - 1) / (2 * TM);
  if (threadIdx.x == 0) {
    for (int i = 0; i < kStages; ++i) {
      mbar_init(smem_u32(&s.full[i]), 1);
      mbar_init(smem_u32(&s.empty[i]), min(live_rows, WR) * WN);
    }
    s.abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (rw >= live_rows) return;
  volatile int* abort_flag = &s.abort;
  const int nk = (p.Kd + kF32K - 1) / kF32K;
  const size_t row0 = (size_t)tile * kTileRows + part * BM;
  int issued = 0, fill = 0;  // copies issued so far (by the first thread), the stage the next one goes to
  auto issue = [&]() {
    const uint32_t bar = smem_u32(&s.full[fill]), dst = smem_u32(ring) + (uint32_t)(fill * kStage);
    const int kc = issued * kF32K;
    mbar_expect_tx(bar, (uint32_t)kStage);  // rows and columns outside a matrix arrive as zeros
    tma_load_2d(dst, &map_a, bar, kc, (int)row0);
    if (SWIGLU) {
      tma_load_3d(dst + kA, &map_b1, bar, kc, n0, e);
      tma_load_3d(dst + kA + (kStage - kA) / 2, &map_b2, bar, kc, n0, e);
    } else {
      tma_load_4d(dst + kA, &map_b1, bar, kc, n0, e % p.tp, e / p.tp);
    }
    ++issued;
    if (++fill == kStages) fill = 0;
  };
  if (threadIdx.x == 0)
    for (int k = 0; k < min(kStages - 1, nk); ++k) issue();
  bool failed = false;
  unsigned long long acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0ull;
  // rows r0 + 2 i; columns of B c0 + 16 j (GEMM1: the first half of the j gate, the others the same columns' up rows)
  constexpr int kCols = SWIGLU ? TN / 2 : TN;
  const int r0 = rw * 2 * TM + lane % 2, c0 = cw * 16 * kCols + lane / 2;
  // the swizzle's row bits: a lane's rows r0 + 2 i take four values of (row % 8), its columns c0 + 16 j only one
  uint32_t aoff[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) aoff[i] = (uint32_t)((r0 + 2 * i) & 7) << 4;
  const uint32_t boff = (uint32_t)(c0 & 7) << 4;
  int b = 0;
  uint32_t phase = 0;
  for (int k = 0; k < nk; ++k) {
    // (After a wait that ran out the stage is computed all the same, on whatever it holds: the vote behind it has the warp
    // leave together.)
    failed = !mbar_wait(smem_u32(&s.full[b]), phase, abort_flag, p.wait_ns);
    const uint32_t a_base = smem_u32(ring) + (uint32_t)(b * kStage) + (uint32_t)r0 * 128u;
    const uint32_t b_base = smem_u32(ring) + (uint32_t)(b * kStage + kA) + (uint32_t)c0 * 128u;
#pragma unroll 1
    for (int half = 0; half < 2; ++half) {
      if (half == 1 && issued > 0 && issued < nk && !failed) {  // the first thread: refill the stage used up in the last iteration
        if (k > 0 && !mbar_wait(smem_u32(&s.empty[fill]), (uint32_t)((k - 1) / kStages) & 1u, abort_flag, p.wait_ns)) failed = true;
        else issue();
      }
#pragma unroll
      for (int uu = 0; uu < kF32K / 8; ++uu) {
        const uint32_t u = (uint32_t)(half * (kF32K / 8) + uu) << 4;
        unsigned long long bl[TN], bh[TN];
#pragma unroll
        for (int j = 0; j < TN; ++j) lds_k4(b_base + (boff ^ u) + (uint32_t)(j < kCols ? 16 * j : BN / 2 + 16 * (j - kCols)) * 128u, bl[j], bh[j]);
#pragma unroll
        for (int i = 0; i < TM; ++i) {
          unsigned long long al, ah;
          lds_k4(a_base + (aoff[i & 3] ^ u) + (uint32_t)i * 2u * 128u, al, ah);
#pragma unroll
          for (int j = 0; j < TN; ++j) fma_x2(acc[i][j], al, bl[j]);
#pragma unroll
          for (int j = 0; j < TN; ++j) fma_x2(acc[i][j], ah, bh[j]);
        }
      }
    }
    failed = __any_sync(0xffffffffu, failed);
    if (failed) break;
    if (lane == 0) mbar_arrive(smem_u32(&s.empty[b]));
    if (++b == kStages) { b = 0; phase ^= 1u; }
  }
  if (failed) {
    s.abort = 1;
    set_status(p.status, MOE_ERR_TIMEOUT, kWaitMbarTma);
    // no copy may still be landing when the CTA's shared memory goes away (only the first thread has issued any)
    for (int g = max(0, issued - kStages); g < issued; ++g) {
      const unsigned long long ts = globaltimer();
      while (!mbar_try(smem_u32(&s.full[g % kStages]), (uint32_t)(g / kStages) & 1u))
        if (globaltimer() - ts > p.wait_ns + 1000000ull) break;
    }
    return;
  }
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    if (r0 + 2 * i >= rows) continue;
    float* crow = p.C + (row0 + r0 + 2 * i) * p.N;
#pragma unroll
    for (int j = 0; j < kCols; ++j) {
      const int n = n0 + c0 + 16 * j;
      if (n >= p.N) continue;
      float v = sum_x2(acc[i][j]);
      if (SWIGLU) v = v / (1.0f + expf(-v)) * sum_x2(acc[i][SWIGLU ? kCols + j : j]);
      crow[n] = v;
    }
  }
}

// A CTA computes one block of rows and columns, and with ANY goes on to the next ones a grid apart while there are any (a grid
// that holds every block a caller's table could ask for would be mostly empty: see launch_fp32_gemm).  The blocks that have
// rows come first, one column of blocks after the other, so they spread over all SMs.  (With a CTA for every block a tile could
// have, the empty ones leave at once but the others stand at every fourth place: 37 of the 148 SMs had work.  T 64, H 1024,
// 32 experts, top-4, F 2048: layer 329 -> 252 us; T 100, H 512, 8 experts, top-2, F 512: 80 -> 69.)
// WR: how many of the four warps stand along the rows (the others beside them, along the columns).
template <int TM, int TN, int WR, bool SWIGLU, bool ANY>
__global__ void __launch_bounds__(kF32Threads, (kF32Ctas<TM, TN, WR>))
ffn_fp32_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b1,
                const __grid_constant__ CUtensorMap map_b2, const Fp32Params p) {
  constexpr int BM = WR * 2 * TM, BN = kF32Warps / WR * 16 * TN, NOUT = SWIGLU ? BN / 2 : BN;
  constexpr int kStages = kF32Stages<TM, TN, WR>;
  static_assert(kStages <= 4, "barriers in Fp32Shared");
  __shared__ Fp32Shared s;
  extern __shared__ uint8_t f32_dyn[];
  uint8_t* ring = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(f32_dyn) + 1023) & ~(uintptr_t)1023);
  pdl_wait();
  pdl_trigger();
  if (threadIdx.x < 32) fp32_find_block<BM, NOUT>(p, s, blockIdx.x);
  __syncthreads();
  if (s.col < 0) return;
  for (;;) {
    fp32_block<TM, TN, WR, SWIGLU>(map_a, map_b1, map_b2, p, s, ring);
    if (!ANY || s.next < 0) return;
    __syncthreads();
    if (s.abort) return;
    if (threadIdx.x == 0) {  // (every copy has been waited for, every arrival made)
      for (int i = 0; i < kStages; ++i) {
        mbar_inval(smem_u32(&s.full[i]));
        mbar_inval(smem_u32(&s.empty[i]));
      }
    }
    if (threadIdx.x < 32) {
      const int id = s.next;
      __syncwarp();  // (the search writes the next one)
      fp32_find_block<BM, NOUT>(p, s, id);
    }
    __syncthreads();
  }
}

// fp32 tensor, innermost dimension first, rows of 32 elements by box_rows, 128-byte swizzle.
static int make_map_f32(EncodeTiledFn enc, CUtensorMap* m, const void* base, int rank, const cuuint64_t* dims,
                        const cuuint64_t* strides, int box_rows) {
  cuuint32_t box[4] = {(cuuint32_t)kF32K, (cuuint32_t)box_rows, 1, 1}, estr[4] = {1, 1, 1, 1};
  CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, (cuuint32_t)rank, const_cast<void*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? MOE_OK : MOE_ERR_CUDA;
}

template <int TM, int TN, int WR, bool SWIGLU>
static int launch_fp32_gemm(moe_plan* p, EncodeTiledFn enc, const void* A, const void* b1, const void* b2,
                            const Fp32Params& q, cudaStream_t st, bool own) {
  constexpr int BM = WR * 2 * TM, BN = kF32Warps / WR * 16 * TN, NOUT = SWIGLU ? BN / 2 : BN;
  const cuuint64_t E = (cuuint64_t)p->cfg.E, K = (cuuint64_t)q.Kd, N = (cuuint64_t)q.N, tp = (cuuint64_t)p->tp;
  CUtensorMap ma, mb1, mb2;
  int rc;
  const cuuint64_t adims[2] = {K, (cuuint64_t)p->P * kTileRows}, astr[1] = {K * 4};
  if ((rc = make_map_f32(enc, &ma, A, 2, adims, astr, BM)) != MOE_OK) return rc;
  if (SWIGLU) {  // gate / up rows of a TP shard are contiguous: [E * tp, F / tp, H]
    const cuuint64_t dims[3] = {K, N, E}, str[2] = {K * 4, N * K * 4};
    if ((rc = make_map_f32(enc, &mb1, b1, 3, dims, str, BN / 2)) != MOE_OK) return rc;
    if ((rc = make_map_f32(enc, &mb2, b2, 3, dims, str, BN / 2)) != MOE_OK) return rc;
  } else {       // a shard of the down matrix is a column slice of it
    const cuuint64_t dims[4] = {K, N, tp, E / tp}, str[3] = {K * tp * 4, K * 4, N * K * tp * 4};
    if ((rc = make_map_f32(enc, &mb1, b1, 4, dims, str, BN)) != MOE_OK) return rc;
    mb2 = mb1;
  }
  // Inside moe_layer a CTA per block that there can be: the counts add up to T * K, so besides full blocks there is at most
  // one per tile.  A caller's table may have any number of whole tiles or of empty ones: a CTA per block that any of its tiles
  // could have, but as each of them walks the table not more than 16 per SM, five times what is resident.  Measured,
  // moe_expert_ffn with counters, us, always a CTA per block / this: 1024 tiles of static regions, 500 tokens, H 256, F 512 193
  // / 83; 31 tiles, T 1000, H 1024, F 2048 722 / 708; 81 tiles, T 700, H 512, F 512 189 / 196; 32 and 64 per SM: 83 and 95 on
  // the first.
  const long long cols = (q.N + NOUT - 1) / NOUT, all = (long long)p->P * (kTileRows / BM) * cols;
  const int sms = p->sm_count > 0 ? p->sm_count : 148;
  const bool any = !own && all > 16ll * sms;
  const dim3 grid((unsigned)(own ? min(all, ((long long)q.total_rows / BM + p->P) * cols) : any ? 16ll * sms : all));
  constexpr size_t smem = 1024 + (size_t)kF32Stages<TM, TN, WR> * kF32StageBytes<TM, TN, WR>;
  p->launches += 1;
  auto launch = [&](auto kern, SmemAttrOnce& once) -> int {
    if (ensure_dynamic_smem(kern, smem, p->device, once) != cudaSuccess) return MOE_ERR_CUDA;
    return launch_pdl(kern, grid, dim3(kF32Threads), smem, st, ma, mb1, mb2, q) == cudaSuccess ? 0 : MOE_ERR_CUDA;
  };
  static SmemAttrOnce once[2];
  return any ? launch(ffn_fp32_kernel<TM, TN, WR, SWIGLU, true>, once[1]) : launch(ffn_fp32_kernel<TM, TN, WR, SWIGLU, false>, once[0]);
}

// Both GEMMs of an fp32 plan.
static int launch_fp32(moe_plan* p, const void* recv, const int* tile_expert, const void* wg, const void* wu, const void* wd,
                       void* out_rows, const int* tile_count, const int* rows_done, cudaStream_t st, bool own) {
  const moe_config_t& c = p->cfg;
  EncodeTiledFn enc;
  int rc = get_encoder(p, &enc);
  if (rc != MOE_OK) return rc;
  Fp32Params q;
  q.tile_expert = tile_expert;
  q.tile_count = tile_count;
  q.rows_done = rows_done;
  q.total_rows = c.T * c.K;
  q.P = (int)p->P;
  q.E = c.E;
  q.tp = p->tp;
  q.wait_ns = kDefaultWaitNs;  // the waits are on this CTA's own copies: nothing a caller's limit is meant for
  q.status = p->s.status;
  const int sms = p->sm_count > 0 ? p->sm_count : 148;
  // Results per lane: 8 x 8 (64 x 128 per CTA) for experts with many rows, 4 x 8 (32 x 128) for experts with about a tile,
  // both where that gives enough CTAs; otherwise 4 x 4 (32 x 64).  Measured, whole layer, us, 8 x 8 / 4 x 8 / 4 x 4: 500 rows
  // per expert 357 / 382 / 383, 250 rows (H 512, F 1024) 248 / 242 / 215, 125 rows 787 / 735 / 766, 66 rows 157 / 143 / 138,
  // 37 rows 470 / 409 / 365.
  // (Without row counts every tile is computed whole: rows as many as a tile per expert has, once most experts have one.
  // Measured without counts, us, by T * K / by this: 36 rows per expert, 256 experts, H 160, F 48 108 / 93; 33, 60 experts, H 512,
  // F 512 417 / 318; 16, 16 experts, H 1024, F 2048 841 / 671.)
  const long long assigned = (long long)c.T * c.K;
  const long long rows = tile_count == nullptr && assigned >= 16ll * c.E ? max(assigned, (long long)kTileRows * c.E) : assigned;
  const long long blocks = rows / 64 + c.E;  // 64-row blocks, about
  const int shape = rows >= 192ll * c.E ? 2 : rows >= 96ll * c.E ? 1 : 0;
  // 4 x 4: how many warps stand along the rows.  An expert's last block of rows leaves warps without rows, and a warp
  // that leaves leaves its scheduler idle, so blocks of eight rows (all warps along the columns) up to 48 rows per expert,
  // of 16 up to 96.  With fewer than eight rows there is one block either way, and the smaller CTAs of 32 rows let GEMM2's
  // start beside GEMM1's.  Measured, whole layer, us, 4 / 2 / 1 warps along the rows, by rows per expert: 4 (H 1024, F 1024)
  // 86 / 109 / 109, 4 (H 512, F 1024) 83 / 85 / 72; 8 (H 1024, F 2048) 252 / 259 / 217; 19 (H 512, F 512) 97 / 83 / 80; 25 (H
  // 512, F 512) 69 / 62 / 56; 33 (H 512, F 256) 102 / 99 / 90; 64 (H 128, F 256) 35 / 33 / 31; 67 (H 512, F 1024) 436 / 429 /
  // 484; 450 (H 256, F 512) 72 / 74 / 80.
  auto along = [&](int n, int cols) {  // cols: the columns of a CTA with all warps along them
    int wr = rows < 8ll * c.E || rows >= 96ll * c.E ? 4 : rows < 48ll * c.E ? 1 : 2;
    while (wr < 4 && cols / wr > n) wr *= 2;
    return wr;
  };
  mark(p, 3, st);
  q.N = c.F;
  q.Kd = c.H;
  q.C = (float*)p->s.inter;
  const bool enough1 = blocks * ((c.F + 63) / 64) >= 2 * sms, enough2 = blocks * ((c.H + 127) / 128) >= 3 * sms / 2;
  if (shape == 2 && enough1) rc = launch_fp32_gemm<8, 8, 4, true>(p, enc, recv, wg, wu, q, st, own);
  else if (shape == 1 && enough1) rc = launch_fp32_gemm<4, 8, 4, true>(p, enc, recv, wg, wu, q, st, own);
  else if (along(c.F, 128) == 1) rc = launch_fp32_gemm<4, 4, 1, true>(p, enc, recv, wg, wu, q, st, own);
  else if (along(c.F, 128) == 2) rc = launch_fp32_gemm<4, 4, 2, true>(p, enc, recv, wg, wu, q, st, own);
  else rc = launch_fp32_gemm<4, 4, 4, true>(p, enc, recv, wg, wu, q, st, own);
  if (rc != 0) return rc;
  mark(p, 4, st);
  q.N = c.H;
  q.Kd = c.F;
  q.C = (float*)out_rows;
  if (shape == 2 && enough2) return launch_fp32_gemm<8, 8, 4, false>(p, enc, p->s.inter, wd, nullptr, q, st, own);
  if (shape == 1 && enough2) return launch_fp32_gemm<4, 8, 4, false>(p, enc, p->s.inter, wd, nullptr, q, st, own);
  if (along(c.H, 256) == 1) return launch_fp32_gemm<4, 4, 1, false>(p, enc, p->s.inter, wd, nullptr, q, st, own);
  if (along(c.H, 256) == 2) return launch_fp32_gemm<4, 4, 2, false>(p, enc, p->s.inter, wd, nullptr, q, st, own);
  return launch_fp32_gemm<4, 4, 4, false>(p, enc, p->s.inter, wd, nullptr, q, st, own);
}

template <typename XT>
static int launch_typed(moe_plan* p, const void* recv, const int* tile_expert, const void* wg,
                        const void* wu, const void* wd, void* out_rows, cudaStream_t st) {
  const moe_config_t& c = p->cfg;
  // c.F is a shard's width; a whole expert's matrices are tp times that.  Gate/up rows of a shard are
  // contiguous ([F/tp, H] at offset s*F/tp*H); a shard of the down matrix is a column slice of it (row pitch: the full width).
  const int tp = p->tp;
  const size_t stride = (size_t)c.F * tp * c.H;
  mark(p, 3, st);
  dim3 g1((c.F + kSimtBN - 1) / kSimtBN, (unsigned)p->P);
  launch_pdl(ffn_simt_kernel<XT, true>, g1, dim3(kSimtThreads), 0, st, (const XT*)recv, c.H, tile_expert,
             (const XT*)wg, (const XT*)wu, stride, tp, (size_t)c.F * c.H, c.H, c.F, c.H, (XT*)p->s.inter, c.F, c.E);
  mark(p, 4, st);
  dim3 g2((c.H + kSimtBN - 1) / kSimtBN, (unsigned)p->P);
  launch_pdl(ffn_simt_kernel<XT, false>, g2, dim3(kSimtThreads), 0, st, (const XT*)p->s.inter, c.F, tile_expert,
             (const XT*)wd, (const XT*)nullptr, stride, tp, (size_t)c.F, c.F * tp, c.H, c.F, (XT*)out_rows, c.H, c.E);
  p->launches += 2;
  return (int)cudaGetLastError();
}

int launch_ffn_simt(moe_plan* p, const void* recv, const int* tile_expert, const void* wg, const void* wu,
                    const void* wd, void* out_rows, const int* tile_count, const int* rows_done, cudaStream_t st, bool own) {
  if (p->P == 0 || p->cfg.T == 0) return 0;
  if (p->cfg.dtype == MOE_DTYPE_BF16)
    return launch_typed<__nv_bfloat16>(p, recv, tile_expert, wg, wu, wd, out_rows, st);
  if (p->s.recv_planes != nullptr) return launch_ffn_split(p, recv, tile_expert, wg, wu, wd, out_rows, tile_count, rows_done, st);
  return launch_fp32(p, recv, tile_expert, wg, wu, wd, out_rows, tile_count, rows_done, st, own);
}

}  // namespace moehub
