// Expert FFN on CTA pairs (paper Section II-A, expert computation; per-tile availability gating as in
// Section IV-D): the cta_group::2 form of the persistent grouped GEMM in ffn_tc.cu.
//
// What bounds the large layers is energy: the part runs at its power limit (SM clock 0.9-1.25 GHz), so a step's time
// is its energy, and the energy is the MMAs that are issued, the operand bytes that travel from L2 to the SMs, and
// the weights' way from HBM.  The form here is chosen for that:
//
//  - The weights are the M side of the MMA, the rows of an expert the N side.  N comes in steps of 32, so a partly
//    filled tile costs what its rows cost; with the rows on the M side every tile costs 128 rows.
//  - A pair of CTAs (a cluster of two SMs) computes 512 weight rows x up to 256 rows of an expert (two of its tiles):
//    tcgen05.mma.cta_group::2 with M = 256, issued by the leader CTA alone, twice per 16 k on the same row operand.
//      GEMM1: gate rows Wg[e, f0:f0+256, :] and up rows Wu[e, f0:f0+256, :];
//      GEMM2: Wd[e, h0:h0+256, :] and Wd[e, h0+256:h0+512, :].
//    Each CTA stages 2 x 128 weight rows and half of the expert's rows: 48 KB per 64 k for 256 x 256 results per SM,
//    half of what one CTA per tile loads, and weights are read once per two tiles.
//  - The accumulators of 512 x 256 results fill tensor memory, so the epilogue of such an item is not hidden behind
//    the next one's MMAs (4-5 us of 30-90; under a power limit a pause costs less than it takes).  Items of at most
//    128 rows need half of it and alternate between the two halves, as the kernel with one CTA per tile does.
//
// Measured against one CTA per tile, whole layer once the clock has settled, us: Mixtral-like T 1024 955 -> 914, T 4096
// 2755 -> 2646; DeepSeek-like T 8192 8237 -> 7870 (Zipf), 8354 -> 7613 (uniform); Phi-like T 4096 1424 -> 1351;
// Qwen-like T 2777 381 -> 361.  Hot and cold experts' items interleaved: no change (energy, not idle pipes).
//
// Roles (576 threads per CTA): warp 0 TMA producer, warp 1 MMA issuer (leader) and TMEM owner, warps 2-17 epilogue.
// The leader's producer claims items dynamically and publishes each to the rings of both CTAs (distributed shared
// memory); every CTA loads its own bytes with plain per-CTA TMA loads.  Per stage, a "full" barrier in the leader (two
// arrivals, both CTAs' loads signal it) and an "empty" barrier in each CTA (the leader's tcgen05.commit arrives on
// both); per accumulator half, a "full" barrier in each CTA (commit to both) and an "empty" barrier in the leader that
// all 32 epilogue warps of the pair arrive on.  Every wait is bounded in time.
#include "tc_common.cuh"

namespace moehub {

constexpr int kPairEpiWarps = 16;
constexpr int kPairThreads = 64 + 32 * kPairEpiWarps;
constexpr int kWHalfBytes = 128 * kBK * 2;             // 16 KB: 128 weight rows
constexpr int kPairStage = 2 * kWHalfBytes + kABytes;  // two weight blocks, then up to 128 of the expert's rows
constexpr int kPairStages = 4;
constexpr int kPairRing = 16;  // the producers are at most 4 items (one per stage) ahead of the MMAs, those 2 ahead of the epilogues
constexpr int kPairPitch = 64;  // bytes of a row of an epilogue warp's staging tile (16 rows x 32 columns)
constexpr int kPairTile = 16 * kPairPitch;
constexpr int kPairSmem = kPairStages * kPairStage + kPairEpiWarps * kPairTile + 1024 + 1024;
// Instruction descriptor: bf16 x bf16 -> fp32, A and B K-major, M = 256 (two CTAs x 128 weight rows), N rows.
__device__ __forceinline__ uint32_t pair_idesc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
}

__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t map_to_cta(uint32_t smem_addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx_cluster(uint32_t cluster_bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cluster.b64 _, [%0], %1;" ::"r"(cluster_bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_bar) : "memory");
}
__device__ __forceinline__ void st_cluster(uint32_t cluster_addr, int v) {
  asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(cluster_addr), "r"(v) : "memory");
}
// Bounded wait that also sees what the other CTA of the pair wrote before it arrived.
__device__ __forceinline__ bool mbar_try_cluster(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity), "r"(kTryHintNs) : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                                  unsigned long long limit_ns) {
  if (mbar_try_cluster(bar, parity)) return true;
  const unsigned long long t0 = globaltimer();
  for (unsigned it = 1;; ++it) {
    if (mbar_try_cluster(bar, parity)) return true;
    if ((it & 31u) == 0u) {
      if (*abort_flag) return false;
      if (globaltimer() - t0 > limit_ns) return false;
    }
  }
}
__device__ __forceinline__ void tma2_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t cluster_bar, int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(dst), "l"(map), "r"(cluster_bar), "r"(c0), "r"(c1) : "memory");
}
// the weights: with an L2 eviction-priority policy (evict-first where they are read this once, else evict-normal)
__device__ __forceinline__ void tma2_load_3d(uint32_t dst, const CUtensorMap* map, uint32_t cluster_bar, int c0, int c1,
                                             int c2, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4, %5}], [%2], %6;"
      ::"r"(dst), "l"(map), "r"(cluster_bar), "r"(c0), "r"(c1), "r"(c2), "l"(policy) : "memory");
}
__device__ __forceinline__ void tma2_load_4d(uint32_t dst, const CUtensorMap* map, uint32_t cluster_bar, int c0, int c1,
                                             int c2, int c3, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4, %5, %6}], [%2], %7;"
      ::"r"(dst), "l"(map), "r"(cluster_bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "l"(policy) : "memory");
}
__device__ __forceinline__ uint64_t l2_policy_evict_normal() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ void tc2_commit_both(uint32_t bar) {  // arrives on `bar` in both CTAs of the pair
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
      ::"r"(bar), "h"((uint16_t)3) : "memory");
}
__device__ __forceinline__ void tc2_commit(uint32_t bar) {  // on `bar` of this CTA
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc2_mma(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                        uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
// Sixteen accumulator columns of the sixteen tensor-memory lanes at taddr: thread l gets lanes l / 4 (r[0], r[1]; r[4], r[5])
// and l / 4 + 8 (r[2], r[3]; r[6], r[7]), columns 2 (l % 4) and + 1, and the same + 8 - the fragment of stmatrix.
__device__ __forceinline__ void tc_ld_frag(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr) : "memory");
}
__device__ __forceinline__ void stmatrix_x4_trans(uint32_t addr, const uint32_t* w) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(w[0]), "r"(w[1]),
               "r"(w[2]), "r"(w[3]) : "memory");
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// Tensor maps: the weights, and the expert's rows (of recv, of the intermediate) in boxes of 128, 64, 32 and 16 rows.
struct PairMaps {
  CUtensorMap wg, wu, wd;
  CUtensorMap rows[2][4];
};

struct PairShared {
  unsigned long long full[kPairStages];   // used in the leader
  unsigned long long empty[kPairStages];  // used in each CTA
  unsigned long long tmem_full[2];        // used in each CTA
  unsigned long long tmem_empty[2];       // used in the leader
  unsigned long long item_bar[kPairRing];
  unsigned long long drain;               // the MMA thread's last commit after an abort
  int item_ring[kPairRing][2];            // item (-1: no more); rows of its two tiles, low and high half-word
  int fills[2];                           // in the leader: the stages' fills that each CTA's producer has issued
  uint32_t tmem_base;
  int abort_flag;                         // set in both CTAs or in neither
  int last_cta;
};
static_assert(sizeof(PairShared) <= 1024, "the epilogue's staging tiles follow");

// An item's rows: r[0] of tile t[0] and r[1] of tile t[1] (t[1] < 0: none).  In the N dimension they stand one after
// the other, each rounded up to 16 (pad[0], pad[1]) and together to n, a multiple of 32.
struct PairRows {
  int t[2], r[2], pad[2], n;
  __device__ __forceinline__ void set(int rows) {
    r[0] = rows & 0xffff;
    r[1] = rows >> 16;
    pad[0] = max(16, (r[0] + 15) & ~15);
    pad[1] = (r[1] + 15) & ~15;
    if ((pad[0] + pad[1]) & 16) {  // (one of them is below 128 then)
      if (pad[0] < kTileRows) pad[0] += 16; else pad[1] += 16;
    }
    n = pad[0] + pad[1];
  }
};

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kPairThreads, 1)
ffn_pair_kernel(const __grid_constant__ PairMaps maps, const FfnParams prm) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* stage_base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  PairShared* sh = reinterpret_cast<PairShared*>(stage_base + kPairStages * kPairStage);
  __shared__ WorkList wl;

  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const uint32_t rank = cluster_ctarank();
  const bool leader = rank == 0;
  const int E = prm.E, F = prm.F, H = prm.H, phase = prm.phase;
  const int nseg = 2 * E;
  const int NB1 = (F + 255) / 256, NB2 = (H + 511) / 512;
  const int KB1 = (H + kBK - 1) / kBK, KB2 = (F + kBK - 1) / kBK;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kPairStages; ++s) {
      mbar_init(smem_u32(&sh->full[s]), 2);
      mbar_init(smem_u32(&sh->empty[s]), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(smem_u32(&sh->tmem_full[a]), 1);
      mbar_init(smem_u32(&sh->tmem_empty[a]), 2 * kPairEpiWarps);
    }
    for (int i = 0; i < kPairRing; ++i) mbar_init(smem_u32(&sh->item_bar[i]), 1);
    mbar_init(smem_u32(&sh->drain), 1);
    sh->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {  // the same warp of both CTAs allocates: 512 columns in each CTA's TMEM
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sh->tmem_base)),
                 "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  pdl_wait();  // everything above needs no global data and overlaps the predecessor's tail
  int* work_counter = prm.work_counter + (phase == 2 ? 1 : 0);
  int first_claim = 0;
  if (leader && threadIdx.x == 0) first_claim = atomicAdd(work_counter, 1);  // in flight while the work list is built
  build_worklist(wl, *reinterpret_cast<WorkScratch*>(stage_base), prm.tile_expert, prm.P, E, NB1, NB2, prm.lag, prm.fused, 2);
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // both CTAs' barriers exist, and both have left the scratch, before anything arrives there
  tc_fence_after();
  const uint32_t tmem_base = sh->tmem_base;
  volatile int* abort_flag = &sh->abort_flag;
  ClockProbe probe(prm.clock_probe);
  const unsigned long long wait_ns = prm.wait_ns;
  int item_begin = 0, item_end = wl.seg_start[nseg];
  if (phase == 1) item_end = wl.n1;
  if (phase == 2) item_begin = wl.n1;

  // item -> (type, expert, column block, its tiles); inside a segment column-block-major, tile-pair-minor.  Only the
  // first lookup searches the segment list: a thread's items only move forward.
  int seg_cursor = -1;
  auto decode = [&](int item, PairRows& rows) {
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
    const int first = wl.estart[it.e], m = wl.estart[it.e + 1] - first, pairs = (m + 1) / 2;
    it.m = m;
    it.cold = m < 3;  // one pair of tiles: the weights are read this once
    const int local = item - wl.seg_start[lo];
    it.nb = local / pairs;
    const int j = 2 * (local - it.nb * pairs);
    rows.t[0] = it.tile = wl.tiles[first + j];
    rows.t[1] = j + 1 < m ? (int)wl.tiles[first + j + 1] : -1;
    return it;
  };
  // Gives up: both CTAs of the pair learn of it.
  auto abort_pair = [&]() {
    sh->abort_flag = 1;
    st_cluster(map_to_cta(smem_u32(&sh->abort_flag), rank ^ 1u), 1);
  };
  volatile int (*item_ring)[2] = sh->item_ring;

  int fail_site = 0;
  if (warp == 0) {
    // ===================== TMA producer (both CTAs; the leader's claims and publishes the items) =====================
    if (lane == 0) {
      int stage = 0;
      uint32_t phase_bit = 0;
      int fills = 0;
      int item = item_begin + first_claim;
      const uint64_t pol_once = l2_policy_evict_first(), pol_keep = l2_policy_evict_normal();
      for (int local_item = 0; !fail_site; ++local_item) {
        const int slot = local_item & (kPairRing - 1);
        PairRows rows;
        Item it;
        if (leader) {
          const bool more = item < item_end;
          int packed = 0, next_item = 0;
          if (more) {
            next_item = item_begin + atomicAdd(work_counter, 1);  // used after this item's loads
            it = decode(item, rows);
            if (rows.t[0] >= prm.P || rows.t[1] >= prm.P || it.e >= E) {  // own index check on what the work list gave
              set_status(prm.status, MOE_ERR_INTERNAL, 211);
              fail_site = kWaitItem;
              break;
            }
            // Availability (Section IV-D) of the tiles' rows: 128 stored, or every assignment of the batch; of their
            // intermediate: every epilogue warp of every GEMM1 block has bumped the tile's counter.  Bounded.
            const int need = 2 * kPairEpiWarps * NB1;
            for (int q = 0; q < 2 && !fail_site; ++q) {
              const int tile = rows.t[q];
              if (tile < 0) continue;
              auto ready = [&]() {
                if (it.type == 1) return ld_acquire(&prm.gemm1_done[tile]) >= need;
                return prm.tile_count == nullptr || ld_acquire(&prm.tile_count[tile]) >= kTileRows ||
                       ld_acquire(prm.rows_done) >= prm.total_rows;
              };
              if (ready()) continue;
              const unsigned long long t0 = globaltimer();
              while (!ready()) {
                if (*abort_flag || globaltimer() - t0 > wait_ns) { fail_site = kWaitTileReady; break; }
                __nanosleep(64);
              }
            }
            if (fail_site) break;
            int r[2];
            for (int q = 0; q < 2; ++q)
              r[q] = rows.t[q] < 0 ? 0 : prm.tile_count == nullptr ? kTileRows : min(kTileRows, prm.tile_count[rows.t[q]]);
            packed = r[0] | (r[1] << 16);
          }
          for (uint32_t c = 0; c < 2; ++c) {
            st_cluster(map_to_cta(smem_u32(&sh->item_ring[slot][0]), c), more ? item : -1);
            st_cluster(map_to_cta(smem_u32(&sh->item_ring[slot][1]), c), packed);
            mbar_arrive_cluster(map_to_cta(smem_u32(&sh->item_bar[slot]), c));
          }
          if (!more) break;
          rows.set(packed);
          item = next_item;
        } else {
          if (!mbar_wait_cluster(smem_u32(&sh->item_bar[slot]), (uint32_t)(local_item / kPairRing) & 1u, abort_flag, wait_ns)) { fail_site = kWaitItem; break; }
          const int got = item_ring[slot][0];
          if (got < 0) break;
          it = decode(got, rows);
          rows.set(item_ring[slot][1]);
        }
        asm volatile("fence.proxy.async.global;" ::: "memory");  // what was seen ready is read through TMA
        const int half = rows.n / 2, lo = (int)rank * half;      // this CTA's share of the N dimension: [lo, lo + half)
        const int len0 = max(0, min(lo + half, rows.pad[0]) - lo), len1 = half - len0;
        const int row0 = rows.t[0] * kTileRows + lo, row1 = rows.t[1] * kTileRows + max(0, lo - rows.pad[0]);
        const CUtensorMap* mr = maps.rows[it.type];
        const int blocks = it.type == 0 || it.nb * 512 + 256 < H ? 2 : 1;
        const uint32_t tx = (uint32_t)(blocks * kWHalfBytes + half * kBK * 2);
        const uint64_t pol = it.cold ? pol_once : pol_keep;
        const int KB = it.type == 0 ? KB1 : KB2;
        for (int kb = 0; kb < KB; ++kb) {
          if (!mbar_wait(smem_u32(&sh->empty[stage]), phase_bit ^ 1u, abort_flag, wait_ns)) { fail_site = kWaitMbarTma; break; }
          const uint32_t full = map_to_cta(smem_u32(&sh->full[stage]), 0);
          const uint32_t dst = smem_u32(stage_base + stage * kPairStage);
          const int kc = kb * kBK;
          mbar_expect_tx_cluster(full, tx);
          if (it.type == 0) {
            const int f = it.nb * 256 + (int)rank * 128;
            tma2_load_3d(dst, &maps.wg, full, kc, f, it.e, pol);
            tma2_load_3d(dst + kWHalfBytes, &maps.wu, full, kc, f, it.e, pol);
          } else {
            const int h = it.nb * 512 + (int)rank * 128, es = it.e % prm.tp, e = it.e / prm.tp;
            tma2_load_4d(dst, &maps.wd, full, kc, h, es, e, pol);
            if (blocks == 2) tma2_load_4d(dst + kWHalfBytes, &maps.wd, full, kc, h + 256, es, e, pol);
          }
          uint32_t rdst = dst + 2 * kWHalfBytes;
          auto load_rows = [&](int row, int len) {  // len: a multiple of 16, at most 128
            if (len == 128) {
              tma2_load_2d(rdst, &mr[0], full, kc, row);
              rdst += 128 * kBK * 2;
              return;
            }
#pragma unroll
            for (int q = 1; q < 4; ++q) {
              const int box = 128 >> q;
              if (len & box) {
                tma2_load_2d(rdst, &mr[q], full, kc, row);
                rdst += box * kBK * 2;
                row += box;
              }
            }
          };
          if (len0 > 0) load_rows(row0, len0);
          if (len1 > 0) load_rows(row1, len1);
          ++fills;
          if (++stage == kPairStages) { stage = 0; phase_bit ^= 1u; }
        }
      }
      if (fail_site) abort_pair();
      st_cluster(map_to_cta(smem_u32(&sh->fills[rank]), 0), fills);
    }
  } else if (warp == 1) {
    // ===================== MMA issuer (leader CTA only) =====================
    if (leader && lane == 0) {
      int stage = 0;
      uint32_t phase_bit = 0;
      uint32_t acc_phase = 0;  // bit a: parity of the uses of accumulator half a so far
      int acc = 0;             // the half the next narrow item takes
      for (int local_item = 0; !fail_site; ++local_item) {
        const int slot = local_item & (kPairRing - 1);
        if (!mbar_wait_cluster(smem_u32(&sh->item_bar[slot]), (uint32_t)(local_item / kPairRing) & 1u, abort_flag, wait_ns)) { fail_site = kWaitItem; break; }
        const int item = item_ring[slot][0];
        if (item < 0) break;
        PairRows rows;
        const Item it = decode(item, rows);
        rows.set(item_ring[slot][1]);
        const bool wide = rows.n > 128;
        const uint32_t halves = wide ? 3u : 1u << acc;
        for (int a = 0; a < 2 && !fail_site; ++a)
          if (((halves >> a) & 1u) && !mbar_wait_cluster(smem_u32(&sh->tmem_empty[a]), ((acc_phase >> a) & 1u) ^ 1u, abort_flag, wait_ns)) fail_site = kWaitMbarTmemFree;
        if (fail_site) break;
        acc_phase ^= halves;
        tc_fence_after();
        const uint32_t d0 = tmem_base + (wide ? 0u : (uint32_t)acc * 256u), d1 = d0 + (wide ? 256u : 128u);
        if (!wide) acc ^= 1;
        const uint32_t idesc = pair_idesc(rows.n);
        const bool two = it.type == 0 || it.nb * 512 + 256 < H;
        const int KB = it.type == 0 ? KB1 : KB2;
        for (int kb = 0; kb < KB; ++kb) {
          if (!mbar_wait_cluster(smem_u32(&sh->full[stage]), phase_bit, abort_flag, wait_ns)) { fail_site = kWaitMbarMma; break; }
          tc_fence_after();
          const uint32_t addr = smem_u32(stage_base + stage * kPairStage);
          const uint64_t w0 = smem_desc_sw128(addr), w1 = smem_desc_sw128(addr + kWHalfBytes);
          const uint64_t rdesc = smem_desc_sw128(addr + 2 * kWHalfBytes);
#pragma unroll
          for (int k = 0; k < kBK / 16; ++k) tc2_mma(d0, w0 + 2 * k, rdesc + 2 * k, idesc, (kb | k) != 0 ? 1u : 0u);
          if (two) {
#pragma unroll
            for (int k = 0; k < kBK / 16; ++k) tc2_mma(d1, w1 + 2 * k, rdesc + 2 * k, idesc, (kb | k) != 0 ? 1u : 0u);
          }
          tc2_commit_both(smem_u32(&sh->empty[stage]));  // both CTAs may refill this stage
          if (++stage == kPairStages) { stage = 0; phase_bit ^= 1u; }
        }
        if (fail_site) break;
        for (int a = 0; a < 2; ++a)  // both CTAs' accumulators complete
          if ((halves >> a) & 1u) tc2_commit_both(smem_u32(&sh->tmem_full[a]));
      }
      if (fail_site) abort_pair();
    }
  } else {
    // ===================== epilogue (both CTAs: their own 128 rows of each weight block) =====================
    // Accumulator lanes are weight rows (F or H columns of the result), its columns the expert's rows.  A warp takes 32
    // columns x 16 rows of the result at a time, transposes them through its own staging tile (stmatrix) and stores 64
    // contiguous bytes of a row with four lanes.  (Stores of 4 bytes after swapping with the neighbour lane need no
    // staging but four times the instructions: 9.7 instead of 4 us for the 512 x 256 results of an item, and that time
    // the tensor pipe waits.)
    const int quarter = warp & 3;             // TMEM lanes this warp may read
    const int which = (warp - 2) / 4;         // it takes every fourth unit of 16 rows (GEMM2: and weight block)
    const uint32_t tile = smem_u32(stage_base + kPairStages * kPairStage + 1024 + (warp - 2) * kPairTile);
    // 16-byte unit u of row r of the tile sits at u ^ (r / 2) % 4: neither the stores nor the loads meet in a bank
    const int st_row = (lane >> 4) * 8 + (lane & 7);
    const uint32_t st_addr = tile + (uint32_t)(st_row * kPairPitch + ((((lane >> 3) & 1) ^ ((st_row >> 1) & 3)) << 4));
    const uint32_t ld_addr = tile + (uint32_t)((lane >> 2) * kPairPitch + (((lane & 3) ^ ((lane >> 3) & 3)) << 4));
    uint32_t acc_phase = 0;
    int acc = 0;
    for (int local_item = 0; !fail_site; ++local_item) {
      const int slot = local_item & (kPairRing - 1);
      if (!warp_agrees(mbar_wait_cluster(smem_u32(&sh->item_bar[slot]), (uint32_t)(local_item / kPairRing) & 1u, abort_flag, wait_ns))) { fail_site = kWaitItem; break; }
      const int item = item_ring[slot][0];
      if (item < 0) break;
      PairRows rows;
      const Item it = decode(item, rows);
      rows.set(item_ring[slot][1]);
      const bool wide = rows.n > 128;
      const uint32_t halves = wide ? 3u : 1u << acc;
      for (int a = 0; a < 2 && !fail_site; ++a)
        if (((halves >> a) & 1u) && !warp_agrees(mbar_wait(smem_u32(&sh->tmem_full[a]), (acc_phase >> a) & 1u, abort_flag, wait_ns))) fail_site = kWaitMbarEpi;
      if (fail_site) break;
      acc_phase ^= halves;
      tc_fence_after();
      const uint32_t base = tmem_base + ((uint32_t)(quarter * 32) << 16) + (wide ? 0u : (uint32_t)acc * 256u);
      const uint32_t second = wide ? 256u : 128u;
      if (!wide) acc ^= 1;
      const bool two = it.type == 1 && it.nb * 512 + 256 < H;  // two results per row (GEMM1: gate and up make one)
      const int ld = it.type == 0 ? F : H;
      __nv_bfloat16* const dst = it.type == 0 ? prm.inter : prm.out;
      const int col0 = (it.type == 0 ? it.nb * 256 : it.nb * 512) + (int)rank * 128 + quarter * 32 + (lane & 3) * 8;
      const int units = rows.n / 16 << (two ? 1 : 0);
      // the accumulators are free for the next item as soon as this warp has read its last values of them
      auto release = [&]() {
        tc_fence_before();
        __syncwarp();
        if (lane == 0)
          for (int a = 0; a < 2; ++a)
            if ((halves >> a) & 1u) mbar_arrive_cluster(map_to_cta(smem_u32(&sh->tmem_empty[a]), 0));  // the leader owns this barrier
      };
      bool released = false;
#pragma unroll 1
      for (int unit = which; unit < units; unit += kPairEpiWarps / 4) {
        const int c = (two ? unit >> 1 : unit) * 16, b = two ? unit & 1 : 0;
        const bool first = c < rows.pad[0];
        const int r0 = first ? c : c - rows.pad[0];
        const int nrow = (first ? rows.r[0] : rows.r[1]) - r0;  // rows of this group that exist
        if (nrow <= 0) continue;
        const int row = (first ? rows.t[0] : rows.t[1]) * kTileRows + r0 + (lane >> 2);  // this lane's rows: row, row + 8
        const bool last = unit + kPairEpiWarps / 4 >= units;
        uint32_t w[8];
        __syncwarp();  // (the loads below want the whole warp; the last unit's stores left it by columns)
        if (it.type == 0) {
          uint32_t g[16], u[16];
          tc_ld_frag(base + c, g);
          tc_ld_frag(base + c + (16u << 16), g + 8);
          tc_ld_frag(base + second + c, u);
          tc_ld_frag(base + second + c + (16u << 16), u + 8);
          tc_wait_ld();
          if (last) release();
#pragma unroll
          for (int i = 0; i < 8; ++i)
            w[i] = pack_bf16(silu_mul(__uint_as_float(g[2 * i]), __uint_as_float(u[2 * i])),
                             silu_mul(__uint_as_float(g[2 * i + 1]), __uint_as_float(u[2 * i + 1])));
        } else {
          uint32_t v[16];
          tc_ld_frag(base + (b ? second : 0u) + c, v);
          tc_ld_frag(base + (b ? second : 0u) + c + (16u << 16), v + 8);
          tc_wait_ld();
          if (last) release();
#pragma unroll
          for (int i = 0; i < 8; ++i) w[i] = pack_bf16(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1]));
        }
        released = last;
        __syncwarp();  // the tile's last contents have been read
        stmatrix_x4_trans(st_addr, w);           // columns 0-15 of the warp's 32
        stmatrix_x4_trans(st_addr ^ 32u, w + 4);  // columns 16-31
        __syncwarp();
        const uint4 lo = lds128(ld_addr), hi = lds128(ld_addr + 8u * kPairPitch);
        const int col = col0 + (b ? 256 : 0);
        if (col < ld) {
          if (it.type == 0 || prm.push_src == nullptr) {
            if ((lane >> 2) < nrow) *reinterpret_cast<uint4*>(dst + (size_t)row * ld + col) = lo;
            if ((lane >> 2) + 8 < nrow) *reinterpret_cast<uint4*>(dst + (size_t)(row + 8) * ld + col) = hi;
          } else {
            // push-style combine: a row goes to its token's position (anything beyond those is none: a stale word after a
            // dispatch that gave up)
            const int s0 = (lane >> 2) < nrow ? __ldcg(prm.push_src + row) : -1;
            const int s1 = (lane >> 2) + 8 < nrow ? __ldcg(prm.push_src + row + 8) : -1;
            if (s0 >= 0 && s0 < prm.total_rows) *reinterpret_cast<uint4*>(dst + (size_t)s0 * ld + col) = lo;
            if (s1 >= 0 && s1 < prm.total_rows) *reinterpret_cast<uint4*>(dst + (size_t)s1 * ld + col) = hi;
          }
        }
      }
      __syncwarp();
      if (!released) release();
      if (it.type == 0) {
        // This warp's part of the block is written: make it visible (also to the async proxy, which
        // is how the GEMM2 producer will read it) and bump the tiles' status counters.
        asm volatile("fence.proxy.async.global;" ::: "memory");
        __threadfence();
        __syncwarp();
        if (lane == 0)
          for (int q = 0; q < 2; ++q)
            if (rows.t[q] >= 0) asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(prm.gemm1_done + rows.t[q]) : "memory");
      }
    }
    if (fail_site && lane == 0) abort_pair();
  }
  if (fail_site) set_status(prm.status, MOE_ERR_TIMEOUT, fail_site);

  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // neither CTA leaves while its partner may still touch its shared memory or TMEM
  tc_fence_after();
  if (sh->abort_flag) {  // (of both CTAs: the barrier above is behind every abort_pair)
    // Whichever role gave up, copies and MMAs that others had issued may still be in flight: all of them have to end before
    // the shared memory and the tensor memory are given up.  The MMAs: the issuing thread's commit comes after them.  The
    // copies: a fill that only one CTA has issued lacks the other one's arrival; with that its phase completes when its bytes
    // are there.  Both waits are bounded.
    if (leader && warp == 1 && lane == 0) {
      tc2_commit(smem_u32(&sh->drain));
      const unsigned long long t0 = globaltimer();
      while (!mbar_try(smem_u32(&sh->drain), 0u))
        if (globaltimer() - t0 > wait_ns + 1000000ull) break;
    }
    if (leader && threadIdx.x == 0) {
      const int all = max(sh->fills[0], sh->fills[1]);
      for (int g = min(sh->fills[0], sh->fills[1]); g < all; ++g) mbar_arrive(smem_u32(&sh->full[g % kPairStages]));
      for (int g = max(0, all - kPairStages); g < all; ++g) {
        const unsigned long long t0 = globaltimer();
        while (!mbar_try(smem_u32(&sh->full[g % kPairStages]), (uint32_t)(g / kPairStages) & 1u))
          if (globaltimer() - t0 > wait_ns + 1000000ull) break;
      }
    }
    __syncthreads();
    cluster_sync_all();
  }
  pdl_trigger();
  probe.finish();
  if (threadIdx.x == 0) {  // the last CTA to leave puts the counters back to zero (see ffn_tc_kernel)
    int* exit_counter = work_counter + 2;
    const bool last = atomicAdd(exit_counter, 1) == (int)gridDim.x - 1;
    if (last) {
      *work_counter = 0;
      *exit_counter = 0;
    }
    sh->last_cta = last ? 1 : 0;
  }
  __syncthreads();
  if (sh->last_cta && phase != 1)
    for (int pt = threadIdx.x; pt < prm.P; pt += kPairThreads) prm.gemm1_done[pt] = 0;
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
}

int launch_ffn_pair(moe_plan* p, const void* recv, const void* wg, const void* wu, const void* wd, FfnParams prm,
                    cudaStream_t st) {
  const moe_config_t& c = p->cfg;
  EncodeTiledFn enc;
  int rc = get_encoder(p, &enc);
  if (rc != MOE_OK) return rc;
  const uint64_t pool_rows = (uint64_t)p->P * kTileRows;
  PairMaps maps;
  if ((rc = make_map_3d(enc, &maps.wg, wg, c.E, c.F, c.H, 128)) != MOE_OK) return rc;
  if ((rc = make_map_3d(enc, &maps.wu, wu, c.E, c.F, c.H, 128)) != MOE_OK) return rc;
  if ((rc = make_map_wd(enc, &maps.wd, wd, c.E / p->tp, p->tp, c.H, c.F, 128)) != MOE_OK) return rc;
  for (int q = 0; q < 4; ++q) {
    if ((rc = make_map_2d(enc, &maps.rows[0][q], recv, pool_rows, c.H, 128u >> q)) != MOE_OK) return rc;
    if ((rc = make_map_2d(enc, &maps.rows[1][q], p->s.inter, pool_rows, c.F, 128u >> q)) != MOE_OK) return rc;
  }
  static SmemAttrOnce once;
  if (ensure_dynamic_smem(ffn_pair_kernel, kPairSmem, p->device, once) != cudaSuccess) return MOE_ERR_CUDA;
  const int grid = p->sm_count & ~1;
  prm.lag = grid;  // two items per pair
  auto launch = [&](int phase) {
    prm.phase = phase;
    p->launches += 1;
    return launch_pdl(ffn_pair_kernel, dim3(grid), dim3(kPairThreads), kPairSmem, st, maps, prm) == cudaSuccess ? 0 : MOE_ERR_CUDA;
  };
  rc = launch(prm.fused ? 0 : 1);
  mark(p, 4, st);
  if (rc == 0 && !prm.fused) rc = launch(2);
  return rc;
}

}  // namespace moehub
