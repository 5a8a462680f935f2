// Grouped expert GEMM on CTA pairs (SwapMoE Section 2: the experts' FFN restricted to the resident slots): two SMs share
// one tile of 256 WEIGHT rows x up to 256 TOKENS through tcgen05 `cta_group::2`.
//
// Why a pair: each CTA stages its own 128 weight rows and half of the tile's tokens; the MMA, issued by the even CTA for
// both, reads the halves from both shared memories and every CTA's tensor core fills the accumulator of its own 128 weight
// rows (all tokens) in its own TMEM.  That is at most 32 KB per CTA and 64-column k-block for 512 tensor clocks (one CTA
// alone: 48 KB), and two accumulator sets fit tensor memory, so the epilogue of one tile overlaps the next tile's MMAs.
// Why the weights are the MMA's rows: its columns then are tokens, whose number is free in steps of 32, so a slot costs
// neither operand bytes nor tensor time for rows it does not have.  A slot's n rows are cut into tiles of equal height
// (write_pair_tiles), and the ring holds more stages where the tiles are small: what a pair pulls per second is bytes in
// flight over the latency of a load (2 us under load).
//
// Roles in each CTA (384 threads): warp 0 = TMA producer (completion is signalled on the EVEN CTA's `full` barrier, which
// expects the bytes of both CTAs), warp 1 = MMA issuer (even CTA only), warp 2 = TMEM allocation, warps 4-11 =
// epilogue of the CTA's own 128 weight rows.  `tcgen05.commit` with a two-CTA mask hands the stage back to both producers
// and announces a finished accumulator to both epilogues; the epilogue warps of both CTAs arrive on the even CTA's
// `acc_empty` barrier.  No load uses cluster multicast.  Every wait is bounded as in tc_gemm_kernel.
#pragma once
#include "gemm_tc.cuh"

namespace swapmoe {

constexpr int kPairTokens = 256;                              // most tokens of a tile
constexpr int kPairMinTokens = 64;                            // ... and the least that pick_tile_height allows it
constexpr int kPairTokenStep = 32;                            // their number is a multiple of this
constexpr int kPairThreads = 384;
constexpr int kPairABytes = kTcBM * kTcBK * 2;                // 16 KB: the CTA's weight rows of a k-block
constexpr int kPairBBytes = kPairTokens / 2 * kTcBK * 2;      // at most 16 KB: its tokens
constexpr int kPairStageArea = 6 * (kPairABytes + kPairBBytes);   // 6 stages of 256 tokens, 8 of 128, 9 of 64
constexpr int kPairMaxStages = 9;
__device__ __forceinline__ int pair_stages(int max_tokens) { return max_tokens > 128 ? 6 : max_tokens > 64 ? 8 : 9; }
// staging of an epilogue warp: a box of 32 tokens x 32 columns (SwiGLU 16), or output row and gate value of its 128 tokens
__host__ __device__ constexpr int pair_warp_bytes(int epi) { return epi == kTcEpiF32 ? 4096 : epi == kTcEpiScatterBf16 ? 1024 : 2048; }
// + alignment slack and barriers (1 KB each).  GEMM-1's leave room for a CTA of the permutation (12 KB).  The ReLU one comes up
// beside it while the permutation still runs (72 registers of 384 threads and 64 of 512: 60416); the gated one does not (89, allocated
// as 96: 69632 of the SM's 65536).
__host__ __device__ constexpr int pair_smem_bytes(int epi) { return kPairStageArea + 2048 + 8 * pair_warp_bytes(epi); }
static_assert(pair_smem_bytes(kTcEpiReluBf16) + 1024 + 12288 <= 228 * 1024, "beside a CTA of the permutation");

namespace ptx {

__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// Address of the same shared-memory location in CTA `rank` of the cluster (shared::cluster window).
__device__ __forceinline__ uint32_t map_to_cta(uint32_t smem_addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// tcgen05.alloc.cta_group::2 takes columns in both SMs, so neither CTA may issue it before the other one has started: without
// this a pair was seen waiting for ever in its allocation (8192 tokens, top-4 of 256 experts, where CTAs of the
// permutation in front still occupy a part of the SMs when the pairs come up).
__device__ __forceinline__ void cluster_start_sync() {
  __syncthreads();
  cluster_sync_all();
}
// Tile load whose completion bytes are credited to a barrier that may live in the peer CTA.
__device__ __forceinline__ void tma_load_2d_pair(void* dst, const CUtensorMap* map, uint32_t bar_cluster_addr, int c0,
                                                 int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(smem_u32(dst)), "l"(map), "r"(bar_cluster_addr), "r"(c0), "r"(c1)
      : "memory");
}
// The same for a box of five dimensions.
__device__ __forceinline__ void tma_load_5d_pair(void* dst, const CUtensorMap* map, uint32_t bar_cluster_addr, int c0,
                                                 int c1, int c2, int c3, int c4) {
  asm volatile(
      "cp.async.bulk.tensor.5d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6, %7}], [%2];"
      ::"r"(smem_u32(dst)), "l"(map), "r"(bar_cluster_addr), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4)
      : "memory");
}
// Arrival on a barrier that may live in the peer CTA, releasing what this thread has done before.
__device__ __forceinline__ void mbar_arrive_release_cluster(uint32_t bar_cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar_cluster_addr) : "memory");
}
// A box of shared memory to global memory; columns and rows outside the matrix are left out.
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, const void* src, int c0, int c1) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];\ncp.async.bulk.commit_group;" ::"l"(map),
               "r"(smem_u32(src)), "r"(c0), "r"(c1)
               : "memory");
}
// This thread's stores have read their shared memory.
__device__ __forceinline__ void tma_store_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void tma_store_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
// Arrival on a barrier that the peer CTA's threads wait on (mbar_try_wait_cluster).  Relaxed at cluster scope: with the tcgen05
// fences on either side it orders this warp's tcgen05 accesses (the accumulator has been read, tcgen05.wait::ld has
// returned) before the waiter's, and nothing else is handed over: nobody in this kernel reads the stores of the epilogue.  With
// .release every epilogue warp waited here until its tile's global stores had been performed, behind the operand loads in
// flight (24044 rows, d_model 1024, d_ff 512, y in fp32: GEMM-2 alone 49 -> 42 us; 8192 rows 768 x 3072: GEMM-1 49.5 -> 46.0).
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar_cluster_addr) {
  asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar_cluster_addr) : "memory");
}
__device__ __forceinline__ void tmem_alloc_pair(uint32_t* dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)),
               "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish_pair() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void umma_bf16_pair(uint32_t tmem_d, uint64_t desc_a, uint64_t desc_b, uint32_t idesc,
                                               uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
      "l"(desc_a), "l"(desc_b), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrives on the barrier at this shared-memory offset in both CTAs of the pair once the MMAs issued so far are done.
__device__ __forceinline__ void umma_commit_pair(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
          smem_u32(bar)),
      "h"((unsigned short)3)
      : "memory");
}

}  // namespace ptx

struct TcPairArgs {
  void* C;                  // [rows, ldc]
  const TileDesc* tiles;    // token tiles: up to 256 rows, multiples of 32 but for a slot's last one
  const int32_t* n_tiles;   // [0] their number, [1] what they hold at most (256, 128 or 64 tokens)
  int32_t* status;
  int32_t ldc;              // columns of C
  int32_t n_col_tiles;      // weight tiles per slot (256 rows; SwiGLU 128 of either matrix)
  int32_t k_blocks;
  int32_t w_rows;           // weight rows per arena entry
  int32_t row_group;        // token tiles per scheduling group (see decode_tile)
  const int32_t* row_pair;  // [rows] pair index of each padded row (scatter epilogue)
  const float* gate;        // [T*k] masked gate values (scatter epilogue)
  int32_t early_w;          // 1: the tile list is final when the CTAs start: weights are requested early
};

// C[token, 256 (128 for SwiGLU) weight rows] = epi(W[256 rows, :] * x[tokens, :]^T); weight rows 128 r .. + 127 of the tile
// belong to CTA r of the pair.  The even CTA stages the first half of the tile's tokens, the odd CTA the second.
// SwiGLU: the 128 lanes hold sixteen rows of W1, the same sixteen of W3, the next sixteen of W1 ... (one 5-D TMA box), so the
// two products of a hidden unit sit in lanes l and l + 16 of one epilogue warp.
template <int EPI>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kPairThreads, 1)
tc_gemm_pair_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX128,
                    const __grid_constant__ CUtensorMap tmX64, const __grid_constant__ CUtensorMap tmX32,
                    const __grid_constant__ CUtensorMap tmX16, const __grid_constant__ CUtensorMap tmC, const TcPairArgs a) {
  constexpr bool kSwiglu = EPI == kTcEpiSwigluBf16;
  constexpr uint32_t kTmemCols = 2 * kPairTokens;             // two accumulator sets

  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  unsigned char* sW = smem;                                   // [stages][128][64] bf16
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kPairStageArea);
  uint64_t* full = bars;                    // [stages]  used in the even CTA
  uint64_t* empty = bars + kPairMaxStages;  // [stages]  one in each CTA (the commit reaches both)
  uint64_t* acc_full = bars + 2 * kPairMaxStages;  // [2]  one in each CTA
  uint64_t* acc_empty = acc_full + 2;       // [2]       used in the even CTA
  uint64_t* tmem_ready = acc_empty + 2;     // used in the even CTA: the odd one has allocated its half
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tmem_ready + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // warp-uniform
  const uint32_t rank = ptx::cluster_ctarank();               // 0: issues the MMAs
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;

  constexpr int kTr = (EPI == kTcEpiReluBf16 || EPI == kTcEpiSwigluBf16) ? 2 : 3;   // trace id: GEMM-1 or GEMM-2
  (void)kTr;
  // The producer's first tile: the number of tiles and the first 32 descriptors (the list holds at least so many) in one round
  // trip, for GEMM-2 underneath the barriers below.
  int4 first_raw = make_int4(0, 0, 0, 0);
  int2 first_n = make_int2(0, 0);
  auto fetch_list = [&]() {
    first_raw = __ldcg(reinterpret_cast<const int4*>(a.tiles + lane));
    first_n = __ldcg(reinterpret_cast<const int2*>(a.n_tiles));
  };
  auto tile_at = [&](int rt) -> TileDesc {                   // by the whole producer warp
    const int src = rt & 31;
    const int4 raw = rt < 32 ? make_int4(__shfl_sync(0xffffffffu, first_raw.x, src), __shfl_sync(0xffffffffu, first_raw.y, src),
                                         __shfl_sync(0xffffffffu, first_raw.z, src), __shfl_sync(0xffffffffu, first_raw.w, src))
                             : __ldcg(reinterpret_cast<const int4*>(a.tiles + rt));
    return *reinterpret_cast<const TileDesc*>(&raw);
  };
  if (warp == 0 && a.early_w) fetch_list();
  if (threadIdx.x == 0) {
    SWAPMOE_STAMP(kTr, 0);
    ptx::mbar_init(tmem_ready, 1);
    for (int s = 0; s < kPairMaxStages; ++s) { ptx::mbar_init(&full[s], 1); ptx::mbar_init(&empty[s], 1); }
    for (int b = 0; b < 2; ++b) { ptx::mbar_init(&acc_full[b], 1); ptx::mbar_init(&acc_empty[b], 16); }
    *abort_flag = 0;
    ptx::fence_barrier_init();
    ptx::prefetch_tmap(&tmW);
    ptx::prefetch_tmap(&tmX128);
  }
  ptx::cluster_start_sync();                                  // both CTAs run and their barriers are initialised
  // Tensor memory: who needs it waits for this CTA's allocation, the MMA issuer also for the peer's; the producers go on.
  uint32_t tmem_base = 0;
  if (warp != 0 && warp != 3) {
    if (warp == 2) {
      ptx::tmem_alloc_pair(tmem_slot, kTmemCols);             // issued in both CTAs: one allocation for the pair
      ptx::tmem_relinquish_pair();
      if (rank == 1 && lane == 0) ptx::mbar_arrive_release_cluster(ptx::map_to_cta(ptx::smem_u32(tmem_ready), 0u));
    }
    ptx::tc_fence_before();
    asm volatile("bar.sync 1, %0;" ::"n"(kPairThreads - 64) : "memory");
    ptx::tc_fence_after();
    tmem_base = *tmem_slot;
  }

  // tokens of a tile in the MMA's columns; each CTA stages half of them
  auto tile_cols = [](int rows) { return (rows + kPairTokenStep - 1) & ~(kPairTokenStep - 1); };
  const uint32_t full0 = ptx::map_to_cta(ptx::smem_u32(full), 0u);
  auto load_w = [&](int stage, int kb, int phys, int ct) {
    const uint32_t bar = full0 + 8u * (uint32_t)stage;
    if (kSwiglu)
      ptx::tma_load_5d_pair(sW + stage * kPairABytes, &tmW, bar, kb * kTcBK, 0, 0, ct * 8 + (int)rank * 4, phys);
    else
      ptx::tma_load_2d_pair(sW + stage * kPairABytes, &tmW, bar, kb * kTcBK,
                            phys * a.w_rows + ct * 2 * kTcBM + (int)rank * kTcBM);
  };

  // As in tc_gemm_kernel: with `early_w` each producer requests the weight boxes of its first stages before the
  // dependent-launch wait.
  int pre = 0;
  if (warp == 0 && a.early_w) {
    const int n_rt = first_n.x, early_stages = pair_stages(first_n.y);
    if (pair < n_rt * a.n_col_tiles) {
      int rt, ct;
      decode_tile(pair, n_rt, a.n_col_tiles, a.row_group, &rt, &ct);
      const TileDesc td = tile_at(rt);
      const uint32_t bytes = (uint32_t)(2 * kPairABytes + tile_cols(td.rows) * kTcBK * 2);
      pre = a.k_blocks < early_stages ? a.k_blocks : early_stages;
      for (int kb = 0; kb < pre; ++kb) {
        if (ptx::elect_one()) {
          if (rank == 0) ptx::mbar_expect_tx(&full[kb], bytes);
          load_w(kb, kb, td.phys, ct);
        }
        __syncwarp();
      }
    }
  }
  if (threadIdx.x == 0) SWAPMOE_STAMP(kTr, 1);
  pdl_wait();      // the activations come from the preceding kernel
  pdl_trigger();
  if (threadIdx.x == 0) SWAPMOE_STAMP(kTr, 2);
  if (warp == 0 && !a.early_w) fetch_list();
  else if (warp != 0) first_n = __ldcg(reinterpret_cast<const int2*>(a.n_tiles));
  const int n_row_tiles = first_n.x, max_tokens = first_n.y;
  const int total = n_row_tiles * a.n_col_tiles;
  const int n_stages = pair_stages(max_tokens), x_bytes = max_tokens / 2 * kTcBK * 2;
  unsigned char* sX = smem + n_stages * kPairABytes;          // [stages][max_tokens / 2][64] bf16

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer (both CTAs)
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    for (int t = pair; t < total && ok; t += n_pairs) {
      int rt, ct;
      decode_tile(t, n_row_tiles, a.n_col_tiles, a.row_group, &rt, &ct);
      const TileDesc td = t == pair ? tile_at(rt) : a.tiles[rt];
      const int cols = tile_cols(td.rows), half = cols / 2;     // half: a multiple of 16, at most 128
      const int xrow = td.row0 + (int)rank * half;
      const uint32_t bytes = (uint32_t)(2 * kPairABytes + cols * kTcBK * 2);
      for (int kb = 0; kb < a.k_blocks; ++kb) {
        const bool early = t == pair && kb < pre;          // armed and weights requested above
        if (!early) {
          ok = warp_wait<true>(&empty[stage], phase ^ 1u, abort_flag, a.status, 11);
          if (!ok) break;
        }
        if (ptx::elect_one()) {
          if (rank == 0 && !early) ptx::mbar_expect_tx(&full[stage], bytes);
          const uint32_t bar = full0 + 8u * (uint32_t)stage;
          unsigned char* dst = sX + stage * x_bytes;
          if (half == 128) {
            ptx::tma_load_2d_pair(dst, &tmX128, bar, kb * kTcBK, xrow);
          } else {                                             // boxes of 64, 32 and 16 rows
            if (half & 64) ptx::tma_load_2d_pair(dst, &tmX64, bar, kb * kTcBK, xrow);
            if (half & 32) ptx::tma_load_2d_pair(dst + (half & 64) * 128, &tmX32, bar, kb * kTcBK, xrow + (half & 64));
            if (half & 16) ptx::tma_load_2d_pair(dst + (half & 96) * 128, &tmX16, bar, kb * kTcBK, xrow + (half & 96));
          }
          if (!early) load_w(stage, kb, td.phys, ct);
        }
        __syncwarp();
        if (++stage == n_stages) { stage = 0; phase ^= 1u; }
      }
      if (lane == 0) SWAPMOE_STAMP(kTr, 3);
    }
    if (!ok) {
      // Give copies that are still in flight time to land before shared memory is released.
      const uint64_t t0 = ptx::globaltimer_ns();
      while (ptx::globaltimer_ns() - t0 < 2000000ull) __nanosleep(1000);
    }
  } else if (warp == 1) {
    if (rank == 0) {
      // ------------------------------------------------------------------ MMA issuer (even CTA, for the pair)
      int stage = 0, acc = 0;
      uint32_t phase = 0, acc_phase = 0;
      bool ok = warp_wait<true>(tmem_ready, 0u, abort_flag, a.status, 15);
      ptx::tc_fence_after();
      for (int t = pair; t < total && ok; t += n_pairs) {
        int rt, ct_unused;
        decode_tile(t, n_row_tiles, a.n_col_tiles, a.row_group, &rt, &ct_unused);
        const uint32_t idesc = make_idesc_bf16(2 * kTcBM, tile_cols(a.tiles[rt].rows));
        ok = warp_wait<true>(&acc_empty[acc], acc_phase ^ 1u, abort_flag, a.status, 12);
        if (!ok) break;
        ptx::tc_fence_after();
        const uint32_t tmem_d = tmem_base + (uint32_t)(acc * kPairTokens);
        for (int kb = 0; kb < a.k_blocks; ++kb) {
          ok = warp_wait<true>(&full[stage], phase, abort_flag, a.status, 13);
          if (!ok) break;
          ptx::tc_fence_after();
          if (lane == 0 && t == pair && kb == 0) SWAPMOE_STAMP(kTr, 4);
          const uint64_t dw = make_kmajor_sw128_desc(ptx::smem_u32(sW + stage * kPairABytes));
          const uint64_t dx = make_kmajor_sw128_desc(ptx::smem_u32(sX + stage * x_bytes));
          if (ptx::elect_one()) {
#pragma unroll
            for (int k = 0; k < kTcBK / kTcUmmaK; ++k)
              ptx::umma_bf16_pair(tmem_d, dw + (uint64_t)(2 * k), dx + (uint64_t)(2 * k), idesc, (kb > 0 || k > 0) ? 1u : 0u);
            ptx::umma_commit_pair(&empty[stage]);   // frees the stage in both CTAs once these MMAs have read it
            if (kb + 1 == a.k_blocks) ptx::umma_commit_pair(&acc_full[acc]);    // accumulator complete, in both CTAs
          }
          __syncwarp();
          if (++stage == n_stages) { stage = 0; phase ^= 1u; }
        }
        if (!ok) break;
        if (lane == 0) SWAPMOE_STAMP(kTr, 5);
        if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
      }
    }
  } else if (warp >= 4) {
    // -------------------------------------------------------------------- epilogue (own 128 weight rows)
    const int q = warp & 3;                    // TMEM lane quarter this warp may read
    const int part = (warp - 4) >> 2;          // two warps per quarter take turns with the chunks of 32 tokens
    const int odd = lane & 1, hi = lane >> 4;
    unsigned char* s_stage = smem + kPairStageArea + 1024 + (warp - 4) * pair_warp_bytes(EPI);
    int2* s_dest = reinterpret_cast<int2*>(s_stage);
    const uint32_t acc_empty0 = ptx::map_to_cta(ptx::smem_u32(acc_empty), 0u);
    int acc = 0;
    uint32_t acc_phase = 0;
    bool ok = true;
    for (int t = pair; t < total && ok; t += n_pairs) {
      int rt, ct;
      decode_tile(t, n_row_tiles, a.n_col_tiles, a.row_group, &rt, &ct);
      const TileDesc td = a.tiles[rt];
      // first of this warp's output columns (32; SwiGLU 16), all of them in the matrix or none
      const int col0 = kSwiglu ? (ct * 8 + (int)rank * 4 + q) * 16 : ct * 2 * kTcBM + (int)rank * kTcBM + q * 32;
      const bool col_ok = col0 < a.ldc;
      if (EPI == kTcEpiScatterBf16) {
        // where the tokens of this warp's chunks go and their gate values: two dependent global loads that the tile's MMAs
        // hide (fetched a chunk ahead they set the pace: d_model 1536, d_ff 1088, 10000 tokens, GEMM-2 61 us)
        __syncwarp();                                          // the tile before has been read out
#pragma unroll
        for (int i = 0; i < kPairTokens / 64; ++i) {
          const int token = (2 * i + part) * 32 + lane;
          const int p = token < td.rows ? a.row_pair[td.row0 + token] : 0;      // top-1: the pair is the token
          s_dest[i * 32 + lane] = make_int2(p, token < td.rows ? __float_as_int(a.gate[p]) : 0);
        }
      }
      ok = warp_wait<true>(&acc_full[acc], acc_phase, abort_flag, a.status, 14);
      if (!ok) break;
      ptx::tc_fence_after();
      const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * kPairTokens);
      const int last = (td.rows - 1) >> 5;                   // the tile's last chunk
      const int my_last = last - ((last ^ part) & 1);        // this warp's last one (-1: none)
      if (my_last < 0 && lane == 0) ptx::mbar_arrive_cluster(acc_empty0 + 8u * (uint32_t)acc);
#pragma unroll 1
      for (int c = part; c <= last; c += 2) {
        const int t0 = 32 * c, left = td.rows - t0;          // valid tokens of this chunk (may exceed 32)
        uint32_t v[32];
        __syncwarp();                                        // the tensor-memory load is one of the whole warp
        ptx::tmem_ld32(taddr + (uint32_t)t0, v);
        ptx::tmem_ld_wait();
        if (c == my_last) {
          // last read of this accumulator: one arrival per warp on the even CTA's barrier, 16 hand it back to the MMA issuer
          ptx::tc_fence_before();
          __syncwarp();
          if (lane == 0) ptx::mbar_arrive_cluster(acc_empty0 + 8u * (uint32_t)acc);
        }
        if (!col_ok) continue;
        // Boxes of 32 tokens leave through the TMA unit (stored by the lanes themselves, eight warps' stores held up the
        // operand loads: fp32 y, 24044 rows of 1024, GEMM-2 45.7 us against 41.2).  Rows up to the next multiple of 32 are
        // stored with the valid ones: they lie in the slot's own segment, and nobody reads a row that no pair occupies.
        unsigned char* stg = s_stage;
        if (EPI != kTcEpiScatterBf16) {
          if (lane == 0) ptx::tma_store_wait_read();
          __syncwarp();
        }
        if (EPI == kTcEpiF32) {
          float* w = reinterpret_cast<float*>(stg) + lane;     // [32 tokens][32 columns]
#pragma unroll
          for (int j = 0; j < 32; ++j) w[32 * j] = __uint_as_float(v[j]);
        } else if (EPI == kTcEpiSwigluBf16) {
          // lanes l and l + 16 hold the two products of hidden unit l & 15: the lower one finishes token 2 i, the upper one
          // token 2 i + 1; then neighbours trade, so that each has two units of one token
          uint32_t* w = reinterpret_cast<uint32_t*>(stg) + (2 * odd + hi) * 8 + ((lane & 14) >> 1);    // [32 tokens][16 units]
          float o[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const float v0 = __uint_as_float(v[2 * i]), v1 = __uint_as_float(v[2 * i + 1]);
            const float r = __shfl_xor_sync(0xffffffffu, hi ? v0 : v1, 16);
            const float x1 = hi ? r : v0, x3 = hi ? v1 : r;
            o[i] = silu_from_exp(x1, __expf(-x1)) * x3;
          }
#pragma unroll
          for (int m = 0; m < 8; ++m) {
            const float r = __shfl_xor_sync(0xffffffffu, odd ? o[2 * m] : o[2 * m + 1], 1);
            w[32 * m] = odd ? pack_bf16x2(r, o[2 * m + 1]) : pack_bf16x2(o[2 * m], r);
          }
        } else {
          // neighbouring lanes trade, so that each holds two output columns of one token (scatter: 64 contiguous bytes of
          // two tokens per instruction)
          uint32_t* w = reinterpret_cast<uint32_t*>(stg) + odd * 16 + (lane >> 1);      // [32 tokens][32 columns]
          bf16* dst = static_cast<bf16*>(a.C) + col0 + (lane & 30);
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const float v0 = __uint_as_float(v[2 * i]), v1 = __uint_as_float(v[2 * i + 1]);
            const float r = __shfl_xor_sync(0xffffffffu, odd ? v0 : v1, 1);
            const float lo = odd ? r : v0, up = odd ? v1 : r;
            if (EPI == kTcEpiReluBf16) {
              w[32 * i] = pack_bf16x2(fmaxf(lo, 0.f), fmaxf(up, 0.f));
            } else {
              const int j = 2 * i + odd;
              const int2 to = s_dest[(c >> 1) * 32 + j];
              const float g = __int_as_float(to.y);
              if (j < left) *reinterpret_cast<uint32_t*>(dst + (size_t)to.x * a.ldc) = pack_bf16x2(lo * g, up * g);
            }
          }
        }
        if (EPI != kTcEpiScatterBf16) {
          ptx::fence_proxy_async();                            // the staged box is read by the TMA unit
          __syncwarp();
          if (lane == 0) ptx::tma_store_2d(&tmC, stg, col0, td.row0 + t0);
        }
      }
      if (q == 0 && lane == 0) SWAPMOE_STAMP(kTr, 6);
      if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
    }
    if (EPI != kTcEpiScatterBf16 && lane == 0) ptx::tma_store_wait_all();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::cluster_sync_all();       // neither CTA's shared memory, barriers or TMEM go away while the peer may touch them
  if (warp == 2) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc_pair(tmem_base, kTmemCols);
  }
}

typedef void (*TcPairKernel)(const CUtensorMap, const CUtensorMap, const CUtensorMap, const CUtensorMap, const CUtensorMap,
                             const CUtensorMap, const TcPairArgs);

template <int EPI>
inline bool tc_pair_set_smem_attr() {
  return cudaFuncSetAttribute(tc_gemm_pair_kernel<EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, pair_smem_bytes(EPI)) ==
         cudaSuccess;
}

// CTA pairs that can be resident at once (0 when the kernels cannot be launched).
inline int tc_pair_init(int sm_count) {
  if (!(tc_pair_set_smem_attr<kTcEpiReluBf16>() && tc_pair_set_smem_attr<kTcEpiSwigluBf16>() &&
        tc_pair_set_smem_attr<kTcEpiF32>() && tc_pair_set_smem_attr<kTcEpiScatterBf16>())) {
    cudaGetLastError();
    return 0;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * (sm_count / 2)); cfg.blockDim = dim3(kPairThreads); cfg.dynamicSmemBytes = pair_smem_bytes(kTcEpiF32);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, tc_gemm_pair_kernel<kTcEpiF32>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n < sm_count / 2 ? n : sm_count / 2;
}

// Launches GEMM-1 (which = 1) or GEMM-2 (2) of a layer on CTA pairs over its list of token tiles.  With top_k == 1 the second
// GEMM writes gate * y straight into `out` and no combine kernel is needed.
inline int32_t tc_gemm_pair(TcState& s, int n_pairs, const swapmoe_config_t& c, int which, void* out, const TileDesc* tiles,
                            const int32_t* n_tiles, int max_tiles, const int32_t* row_pair, const float* mgate,
                            int n_tokens, int32_t* status, cudaStream_t st, bool pdl, int row_group_forced) {
  if (!s.enabled || !s.arena_bound || n_pairs < 1) return SWAPMOE_ERR_NOT_READY;
  const bool swiglu = c.act == SWAPMOE_ACT_SWIGLU, scatter = c.top_k == 1;
  const long long pairs = (long long)n_tokens * c.top_k;
  TcPairArgs g;
  g.C = out; g.status = status; g.tiles = tiles; g.n_tiles = n_tiles; g.row_pair = row_pair; g.gate = mgate;
  g.row_group = 1 << 30;
  if (row_group_forced > 0) g.row_group = row_group_forced;
  else if (pairs * (long long)c.d_model * 2 > (48ll << 20)) {
    // Token rows of a group stay in L2 across its weight tiles: as many tiles as make 20 MB when they hold 256 rows each (slots cut
    // into lower tiles make smaller groups, down to half of that just above 256 rows a slot, a quarter under a cap of 64).  The
    // optimum is flat: us per forward at 5 / 10 / 20 / 40 / all tiles per group, 1024 x 512 top-4, 64 slots, 16000 tokens 289 / 291
    // / 290 / 295 / 322 (40 is what this rule gives); 2048 x 1024 top-2, 12000 tokens, slots of 330 to 420 rows 355 / 355 / 357 / 362 /
    // 393 (20); SwiGLU 4096 x 14336, 4096 tokens, 4 / 10 / 16 / 32 / all 2592 / 2456 / 2469 / 2454 / 2490 (10).
    g.row_group = (int)((20ll << 20) / (2ll * kTcBM * c.d_model * 2));
    if (g.row_group < 4) g.row_group = 4;
  }
  const CUtensorMap *mw, *mx, *mc;
  TcPairKernel k;
  int epi;
  if (which == 1) {
    const int out1 = swiglu ? kTcBM : 2 * kTcBM;
    g.ldc = c.d_ff; g.n_col_tiles = (c.d_ff + out1 - 1) / out1; g.k_blocks = c.d_model / kTcBK;
    g.w_rows = c.d_ff; g.early_w = 0;
    epi = swiglu ? kTcEpiSwigluBf16 : kTcEpiReluBf16;
    k = swiglu ? tc_gemm_pair_kernel<kTcEpiSwigluBf16> : tc_gemm_pair_kernel<kTcEpiReluBf16>;
    mw = swiglu ? &s.map_win_gated : &s.map_win[1]; mx = s.map_xp; mc = &s.map_h_out;
  } else {
    g.ldc = c.d_model; g.n_col_tiles = (c.d_model + 2 * kTcBM - 1) / (2 * kTcBM); g.k_blocks = c.d_ff / kTcBK;
    g.w_rows = c.d_model; g.early_w = 1;
    epi = scatter ? kTcEpiScatterBf16 : kTcEpiF32;
    k = scatter ? tc_gemm_pair_kernel<kTcEpiScatterBf16> : tc_gemm_pair_kernel<kTcEpiF32>;
    mw = &s.map_wout[1]; mx = s.map_h; mc = &s.map_y_out;
  }
  const long long work = (long long)max_tiles * g.n_col_tiles;
  return launch_kernel(k, dim3(2 * (work > n_pairs ? n_pairs : (int)work)), dim3(kPairThreads), pair_smem_bytes(epi), st, pdl, *mw,
                       mx[0], mx[1], mx[2], mx[3], *mc, g) == cudaSuccess ? SWAPMOE_OK : SWAPMOE_ERR_CUDA;
}

}  // namespace swapmoe
