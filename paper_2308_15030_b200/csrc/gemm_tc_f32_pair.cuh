// Grouped expert GEMM for fp32 layers on CTA pairs (SwapMoE Section 2), for slots of well over one 128-row tile: the
// products and the operand split of tc_gemm_f32_kernel, on 256 x 192 tiles with tcgen05 `cta_group::2`.
//
// What bounds tc_gemm_f32_kernel on such slots is neither the tensor core nor the conversion but what the SMs pull from
// L2: 32 KB of fp32 operands per k-block of 32 and 128 x 128 tile, 9.3 TB/s over all SMs (3062 rows, d_model 1024, d_ff
// 2816, SwiGLU: 1.25 GB in 134 us; halving the conversion time changed nothing).  Here a CTA stages its own 128
// token rows and half of the tile's 192 weight rows: 28 KB for one and a half times the work.  192 columns, because two
// accumulator sets of 192 and four slots of converted A (32 columns each) fill the 512 columns of tensor memory exactly,
// so the epilogue stays overlapped.  3062 rows of that layer: GEMM-1 134 -> 117 us, forward 252 -> 225; 6400 rows of
// 768 x 3072, ReLU, forward 287 -> 224.
//
// Roles in each CTA (768 threads): warp 0 TMA producer (own rows and own half of the weights, completion on the CTA's own
// `full` barrier), warp 1 MMA issuer (even CTA only, for both), warp 2 TMEM allocation, warps 4-7 epilogue of the CTA's own
// 128 rows, warps 8-15 and 16-23 two converter groups that take alternate k-blocks (four warps split A into tensor
// memory, four rewrite B in place).  The converters of both CTAs arrive on the even CTA's `conv_done`; commits with
// a two-CTA mask free stages and slots in both.  SwiGLU: the even CTA stages W1 rows, the odd one the same W3 rows.  Every
// wait is bounded; no load uses cluster multicast.
#pragma once
#include "gemm_tc_f32.cuh"
#include "gemm_tc_pair.cuh"

namespace swapmoe {

constexpr int kF32PairBN = 192;                                        // accumulator columns of the pair's tile
constexpr int kF32PairHalf = kF32PairBN / 2;                           // weight rows each CTA stages
constexpr int kF32PairBBytes = kF32PairHalf * kF32BK * 4;              // 12 KB
constexpr int kF32PairStageBytes = kF32ABytes + kF32PairBBytes;
constexpr int kF32PairStages = 7;
constexpr int kF32PairThreads = 768;
constexpr int kF32PairASlotBase = 2 * kF32PairBN;                      // first TMEM column of the A slots
constexpr int kF32PairSmemBytes = kF32PairStages * kF32PairStageBytes + 2048 + kTcEpiStageBytes;
static_assert(kF32PairASlotBase + kF32ASlots * kF32ASlotCols <= 512, "tensor memory");
static_assert(kF32PairSmemBytes <= 227 * 1024 && kF32PairStageBytes % 1024 == 0, "shared memory per CTA, swizzle atoms");

namespace ptx {
__device__ __forceinline__ void umma_bf16_ts_pair(uint32_t tmem_d, uint32_t tmem_a, uint64_t desc_b, uint32_t idesc,
                                                  uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(tmem_d),
      "r"(tmem_a), "l"(desc_b), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrival of a converter warp on the even CTA's barrier, whose waiter issues MMAs that read what the warp has written: tensor
// memory, ordered by the tcgen05 fences on either side, and shared memory, for which the release has to reach the cluster.
// It is restricted to this CTA's shared memory: an unrestricted one is a full memory fence behind the loads in flight (us per
// forward, 3062 rows of 1024 x 2816 SwiGLU 386 against 256, 6400 of 768 x 3072 ReLU 380 against 260; with no release beyond the
// CTA, which the waiter's SM is not bound to see, 254 and 256).
__device__ __forceinline__ void mbar_arrive_converted(uint32_t bar_cluster_addr) {
  asm volatile("fence.release.sync_restrict::shared::cta.cluster;" ::: "memory");
  mbar_arrive_cluster(bar_cluster_addr);
}
}  // namespace ptx

template <int EPI>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kF32PairThreads, 1)
tc_gemm_f32_pair_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const TcF32Args a) {
  constexpr int kStages = kF32PairStages, kSlots = kF32ASlots;
  constexpr bool kGated = EPI == kTcEpiSwigluF32;
  constexpr int kOutCols = kGated ? kF32PairHalf : kF32PairBN;
  constexpr uint32_t kIdesc = make_idesc_bf16(2 * kTcBM, kF32PairBN);

  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  unsigned char* raw = smem;                                  // [stages][A 16 KB | B 12 KB]
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kStages * kF32PairStageBytes);
  uint64_t* full = bars;                          // [stages]   own TMA -> own converters
  uint64_t* empty = full + kStages;               // [stages]   one in each CTA
  uint64_t* conv_done = empty + kStages;          // [slots]    used in the even CTA: 16 converter warps
  uint64_t* lo_empty = conv_done + kSlots;        // [slots]    one in each CTA
  uint64_t* acc_full = lo_empty + kSlots;         // [2]        one in each CTA
  uint64_t* acc_empty = acc_full + 2;             // [2]        used in the even CTA
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  unsigned char* epi_stage = reinterpret_cast<unsigned char*>(bars) + 1024;

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // warp-uniform
  const uint32_t rank = ptx::cluster_ctarank();
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) { ptx::mbar_init(&full[s], 1); ptx::mbar_init(&empty[s], 1); }
    for (int s = 0; s < kSlots; ++s) { ptx::mbar_init(&conv_done[s], 16); ptx::mbar_init(&lo_empty[s], 1); }
    for (int b = 0; b < 2; ++b) { ptx::mbar_init(&acc_full[b], 1); ptx::mbar_init(&acc_empty[b], 8); }
    *abort_flag = 0;
    ptx::fence_barrier_init();
    ptx::prefetch_tmap(&tmA);
    ptx::prefetch_tmap(&tmB);
  }
  ptx::cluster_start_sync();                      // both CTAs run and their barriers are initialised
  // Who needs tensor memory waits for this CTA's allocation (the MMA issuer learns of the peer's by its converters' first
  // arrivals); the producers go on.
  uint32_t tmem_base = 0;
  if (warp != 0 && warp != 3) {
    if (warp == 2) {
      ptx::tmem_alloc_pair(tmem_slot, 512);
      ptx::tmem_relinquish_pair();
    }
    ptx::tc_fence_before();
    asm volatile("bar.sync 1, %0;" ::"n"(kF32PairThreads - 64) : "memory");
    ptx::tc_fence_after();
    tmem_base = *tmem_slot;
  }

  // weight rows of column tile ct that this CTA stages
  auto weight_row = [&](const TileDesc& td, int ct) {
    return td.phys * a.b_rows_per_phys +
           (kGated ? ct * kF32PairHalf + (int)rank * a.b_rows_gate : ct * kF32PairBN + (int)rank * kF32PairHalf);
  };
  // With `early_b` the weight boxes of the first stages are requested before the wait (see tc_gemm_f32_kernel).
  int pre = 0;
  if (warp == 0 && a.early_b) {
    const int n_rt = __ldcg(a.n_tiles), per = n_rt * a.n_col_tiles;
    if (pair < per * a.n_split) {
      const int z = pair / per, u = pair - z * per, ct = u / n_rt;
      const int4 rawd = __ldcg(reinterpret_cast<const int4*>(a.tiles + (u - ct * n_rt)));
      const int brow = weight_row(*reinterpret_cast<const TileDesc*>(&rawd), ct);
      pre = a.k_blocks < kStages ? a.k_blocks : kStages;
      for (int kb = 0; kb < pre; ++kb) {
        if (ptx::elect_one()) {
          ptx::mbar_expect_tx(&full[kb], (uint32_t)kF32PairStageBytes);
          ptx::tma_load_2d(raw + kb * kF32PairStageBytes + kF32ABytes, &tmB, &full[kb], (z * a.k_blocks + kb) * kF32BK, brow);
        }
        __syncwarp();
      }
    }
  }
  pdl_wait();
  pdl_trigger();
  const int n_row_tiles = *a.n_tiles;
  const int per_slice = n_row_tiles * a.n_col_tiles;
  const int total = per_slice * a.n_split;        // item = slice * per_slice + (col tile * n_row_tiles + row tile)

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer (both CTAs)
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    for (int t = pair; t < total && ok; t += n_pairs) {
      const int z = t / per_slice, u = t - z * per_slice;
      const int ct = u / n_row_tiles;
      const TileDesc td = a.tiles[u - ct * n_row_tiles];
      const int brow = weight_row(td, ct), arow = td.row0 + (int)rank * kTcBM;
      for (int kb = 0; kb < a.k_blocks; ++kb) {
        const bool early = t == pair && kb < pre;
        if (!early) {
          ok = warp_wait<true>(&empty[stage], phase ^ 1u, abort_flag, a.status, 51);
          if (!ok) break;
        }
        if (ptx::elect_one()) {
          unsigned char* st = raw + stage * kF32PairStageBytes;
          const int col = (z * a.k_blocks + kb) * kF32BK;
          if (!early) {
            ptx::mbar_expect_tx(&full[stage], (uint32_t)kF32PairStageBytes);
            ptx::tma_load_2d(st + kF32ABytes, &tmB, &full[stage], col, brow);
          }
          ptx::tma_load_2d(st, &tmA, &full[stage], col, arow);     // (rows behind the slot or the workspace: never stored)
        }
        __syncwarp();
        if (++stage == kStages) { stage = 0; phase ^= 1u; }
      }
    }
    if (!ok) {
      // Give copies that are still in flight time to land before shared memory is released.
      const uint64_t t0 = ptx::globaltimer_ns();
      while (ptx::globaltimer_ns() - t0 < 2000000ull) __nanosleep(1000);
    }
  } else if (warp == 1) {
    if (rank == 0) {
      // ------------------------------------------------------------------ MMA issuer (even CTA, for the pair)
      int stage = 0, slot = 0, acc = 0;
      uint32_t slot_phase = 0, acc_phase = 0;
      bool ok = true;
      for (int t = pair; t < total && ok; t += n_pairs) {
        ok = warp_wait<true>(&acc_empty[acc], acc_phase ^ 1u, abort_flag, a.status, 52);
        if (!ok) break;
        ptx::tc_fence_after();
        const uint32_t tmem_d = tmem_base + (uint32_t)(acc * kF32PairBN);
        for (int kb = 0; kb < a.k_blocks; ++kb) {
          ok = warp_wait<true>(&conv_done[slot], slot_phase, abort_flag, a.status, 53);
          if (!ok) break;
          ptx::tc_fence_after();
          // layouts of a converted stage and slot: see tc_gemm_f32_kernel; small terms first
          const uint64_t db = make_kmajor_sw128_desc(ptx::smem_u32(raw + stage * kF32PairStageBytes + kF32ABytes));
          const uint32_t a1 = tmem_base + (uint32_t)(kF32PairASlotBase + slot * kF32ASlotCols), a2 = a1 + 16;
          if (ptx::elect_one()) {
            ptx::umma_bf16_ts_pair(tmem_d, a2, db, kIdesc, kb > 0 ? 1u : 0u);
            ptx::umma_bf16_ts_pair(tmem_d, a2 + 8, db + 2, kIdesc, 1u);
            ptx::umma_bf16_ts_pair(tmem_d, a1, db + 4, kIdesc, 1u);
            ptx::umma_bf16_ts_pair(tmem_d, a1 + 8, db + 6, kIdesc, 1u);
            ptx::umma_bf16_ts_pair(tmem_d, a1, db, kIdesc, 1u);
            ptx::umma_bf16_ts_pair(tmem_d, a1 + 8, db + 2, kIdesc, 1u);
            ptx::umma_commit_pair(&empty[stage]);       // the raw stage may be refilled, in both CTAs
            ptx::umma_commit_pair(&lo_empty[slot]);     // the TMEM slot may be rewritten, in both CTAs
            if (kb + 1 == a.k_blocks) ptx::umma_commit_pair(&acc_full[acc]);
          }
          __syncwarp();
          if (++stage == kStages) stage = 0;
          if (++slot == kSlots) { slot = 0; slot_phase ^= 1u; }
        }
        if (!ok) break;
        if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
      }
    }
  } else if (warp >= 8) {
    // ---------------------------------------------------------------------- converters
    const int grp = (warp - 8) >> 3;
    const bool does_b = ((warp - 8) >> 2) & 1;
    const int ctid = threadIdx.x & 127;                // row inside the operand (A: = TMEM lane)
    const uint32_t done0 = ptx::map_to_cta(ptx::smem_u32(conv_done), 0u);
    int stage = 0, slot = 0;
    uint32_t phase = 0, slot_phase = 0;
    bool ok = true;
    for (int t = pair; t < total && ok; t += n_pairs) {
      for (int kb = 0; kb < a.k_blocks; ++kb) {
        if ((slot & 1) == grp) {
          ok = warp_wait(&full[stage], phase, abort_flag, a.status, 54);
          if (ok) ok = warp_wait<true>(&lo_empty[slot], slot_phase ^ 1u, abort_flag, a.status, 55);
          if (!ok) break;
          ptx::tc_fence_after();
          if (!does_b) {
            // thread = row = TMEM lane; 32 values -> 16 packed b1 columns and 16 packed b2 columns
            const unsigned char* arow = raw + stage * kF32PairStageBytes + ctid * 128;
            uint32_t hm[32];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const uint4 x = *reinterpret_cast<const uint4*>(arow + ((j ^ (ctid & 7)) << 4));
              split_bf16_pair(x.x, x.y, &hm[2 * j], &hm[16 + 2 * j]);
              split_bf16_pair(x.z, x.w, &hm[2 * j + 1], &hm[16 + 2 * j + 1]);
            }
            ptx::tmem_st32(tmem_base + ((uint32_t)((ctid >> 5) * 32) << 16) +
                               (uint32_t)(kF32PairASlotBase + slot * kF32ASlotCols), hm);
            ptx::tmem_st_wait();
          } else if (ctid < kF32PairHalf) {
            // 32 fp32 -> [32 x b1 | 32 x b2] in place, 16-byte piece c at physical piece c ^ (row & 7)
            unsigned char* brow = raw + stage * kF32PairStageBytes + kF32ABytes + ctid * 128;
            uint32_t p1[16], p2[16];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const uint4 x = *reinterpret_cast<const uint4*>(brow + ((j ^ (ctid & 7)) << 4));
              split_bf16_pair(x.x, x.y, &p1[2 * j], &p2[2 * j]);
              split_bf16_pair(x.z, x.w, &p1[2 * j + 1], &p2[2 * j + 1]);
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              *reinterpret_cast<uint4*>(brow + ((c ^ (ctid & 7)) << 4)) =
                  make_uint4(p1[4 * c], p1[4 * c + 1], p1[4 * c + 2], p1[4 * c + 3]);
              *reinterpret_cast<uint4*>(brow + (((4 + c) ^ (ctid & 7)) << 4)) =
                  make_uint4(p2[4 * c], p2[4 * c + 1], p2[4 * c + 2], p2[4 * c + 3]);
            }
          }
          ptx::tc_fence_before();
          ptx::fence_proxy_async();                    // these writes are read by the tensor cores (async proxy)
          __syncwarp();
          if (lane == 0) ptx::mbar_arrive_converted(done0 + 8u * (uint32_t)slot);
        }
        if (++stage == kStages) { stage = 0; phase ^= 1u; }
        if (++slot == kSlots) { slot = 0; slot_phase ^= 1u; }
      }
    }
  } else if (warp >= 4) {
    // ---------------------------------------------------------------------- epilogue (own 128 rows)
    const int q = warp - 4;
    const int rr = (int)rank * kTcBM + q * 32 + lane;  // row inside the 256-row tile
    int acc = 0;
    uint32_t acc_phase = 0;
    bool ok = true;
    for (int t = pair; t < total && ok; t += n_pairs) {
      const int z = t / per_slice, u = t - z * per_slice;
      const int ct = u / n_row_tiles;
      const TileDesc td = a.tiles[u - ct * n_row_tiles];
      ok = warp_wait<true>(&acc_full[acc], acc_phase, abort_flag, a.status, 56);
      if (!ok) break;
      ptx::tc_fence_after();
      if (rank == 0 || td.rows > kTcBM) {              // the odd CTA has nothing to store for a tile of <= 128 rows
        const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * kF32PairBN);
        unsigned char* dst[8];
        epi_row_pointers(dst, rr < td.rows ? td.row0 + rr : -1, lane,
                         static_cast<float*>(a.C) + (size_t)z * a.split_stride, (size_t)a.ldc, (size_t)ct * kOutCols, 4);
#pragma unroll 1
        for (int c0 = 0; c0 < min(kOutCols, a.ldc - ct * kOutCols); c0 += 32) {
          uint4 pc[8];
          epi_load_pieces_f32<EPI>(taddr, c0, kOutCols, pc);
          epi_store_chunk(epi_stage + q * kTcEpiWarpStage, pc, lane, dst, c0 * 4);
        }
      }
      ptx::tc_fence_before();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive_cluster(ptx::map_to_cta(ptx::smem_u32(&acc_empty[acc]), 0u));
      if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
    }
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::cluster_sync_all();       // neither CTA's shared memory, barriers or TMEM go away while the peer may touch them
  if (warp == 2) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc_pair(tmem_base, 512);
  }
}

// ----------------------------------------------------------------------------- host side
typedef void (*TcF32Kernel)(const CUtensorMap, const CUtensorMap, const TcF32Args);

// CTA pairs that can be resident at once (0 when the kernels cannot be launched).
inline int tc_f32_pair_init(int sm_count) {
  const TcF32Kernel all[3] = {tc_gemm_f32_pair_kernel<kTcEpiReluF32>, tc_gemm_f32_pair_kernel<kTcEpiSwigluF32>,
                              tc_gemm_f32_pair_kernel<kTcEpiF32>};
  for (TcF32Kernel k : all)
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kF32PairSmemBytes) != cudaSuccess) {
      cudaGetLastError();
      return 0;
    }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * (sm_count / 2)); cfg.blockDim = dim3(kF32PairThreads); cfg.dynamicSmemBytes = kF32PairSmemBytes;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, tc_gemm_f32_pair_kernel<kTcEpiF32>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n < sm_count / 2 ? n : sm_count / 2;
}

// Slices of GEMM-2's contraction (copies of y): until every unit (CTA or pair) has an item, eight k-blocks at least.
inline int tc_f32_split(long long tiles, int units, int k_blocks, int y_copies) {
  int split = 1;
  while (split * 2 <= y_copies && tiles * split < units && k_blocks % (split * 2) == 0 && k_blocks / (split * 2) >= 8) split *= 2;
  return split;
}

// Whether the GEMMs of a forward over `rows` pairs run on CTA pairs rather than on one CTA per 128 x 128 tile: rounds of
// tiles times the measured time of a round on either side, in 10 ns (48 per k-block for one CTA, 52 for a pair; a round of
// short SwiGLU tiles takes 6 and 11.8 us whatever its contraction: the epilogue's exponentials share the issue slots with
// the converters).  us per forward one CTA / pairs, top-1 ReLU 768 x 3072 at 110, 170, 260, 420, 800 rows on each of 8 slots:
// 75 / 80, 115 / 90, 127 / 118, 186 / 140, 287 / 224; SwiGLU 512 x 2048 98 / 94 at 260 and 195 / 199 at 800.  Over 100 such
// shapes the rule is 0.4 % from the better side; one side always: 4 % (pairs) and 9 %.
inline bool tc_f32_use_pairs(const swapmoe_config_t& c, int n_pairs, int sm_count, long long rows, int y_copies) {
  if (n_pairs < 1 || rows < 130ll * c.K) return false;
  const bool gated = c.act == SWAPMOE_ACT_SWIGLU;
  const long long half_tiles = (rows < c.K ? rows : c.K) / 2;
  long long cost[2];
  for (int p = 0; p < 2; ++p) {
    const int tile = p ? 2 * kTcBM : kTcBM, bn = p ? kF32PairBN : kF32BN, units = p ? n_pairs : sm_count;
    const int out1 = gated ? bn / 2 : bn, per_kb = p ? 52 : 48, least = gated ? (p ? 1180 : 600) : (p ? 400 : 300);
    const long long rt = rows / tile + half_tiles;
    const long long n1 = rt * ((c.d_ff + out1 - 1) / out1), n2 = rt * ((c.d_model + bn - 1) / bn);
    const int kb1 = c.d_model / kF32BK, kb2 = c.d_ff / kF32BK, split = tc_f32_split(n2, units, kb2, y_copies);
    cost[p] = (n1 + units - 1) / units * (per_kb * kb1 > least ? per_kb * kb1 : least) +
              (n2 * split + units - 1) / units * per_kb * (kb2 / split);
  }
  return cost[1] < cost[0];
}

// Both grouped GEMMs of an fp32 layer on CTA pairs, over a list of 256-row tiles; same contract as tc_ffn_f32.
inline int32_t tc_ffn_f32_pair(TcF32State& s, const swapmoe_config_t& c, void* h, float* y, long long y_copy_stride,
                               int y_copies, const TileDesc* tiles, const int32_t* n_tiles, int max_tiles, int n_tokens,
                               int32_t* status, cudaStream_t st, bool pdl, int64_t* launches, int* y_split,
                               cudaEvent_t between) {
  if (!s.enabled || !s.arena_bound || s.n_pairs < 1) return SWAPMOE_ERR_NOT_READY;
  const bool swiglu = c.act == SWAPMOE_ACT_SWIGLU;
  const int out1 = swiglu ? kF32PairHalf : kF32PairBN;
  TcF32Args g;
  g.tiles = tiles; g.n_tiles = n_tiles; g.status = status;
  g.C = h; g.split_stride = 0; g.n_split = 1; g.early_b = 0;
  g.ldc = c.d_ff; g.n_col_tiles = (c.d_ff + out1 - 1) / out1; g.k_blocks = c.d_model / kF32BK;
  g.b_rows_per_phys = swiglu ? 2 * c.d_ff : c.d_ff;
  g.b_rows_gate = swiglu ? c.d_ff : 0;
  long long work = (long long)max_tiles * g.n_col_tiles;
  int grid = 2 * (int)(work > s.n_pairs ? s.n_pairs : work);
  if (s.only != 2) {
    if (launch_kernel(swiglu ? tc_gemm_f32_pair_kernel<kTcEpiSwigluF32> : tc_gemm_f32_pair_kernel<kTcEpiReluF32>, dim3(grid),
                      dim3(kF32PairThreads), kF32PairSmemBytes, st, pdl, s.map_xp, s.map_win_pair, g) != cudaSuccess)
      return SWAPMOE_ERR_CUDA;
    ++*launches;
  }
  if (between) cudaEventRecord(between, st);
  // GEMM-2: few output tiles, long contraction: slice it until every pair has an item
  const long long rows = (long long)n_tokens * c.top_k;
  const long long row_tiles_est = rows / (2 * kTcBM) + (rows < c.K ? rows : c.K) / 2;
  g.n_col_tiles = (c.d_model + kF32PairBN - 1) / kF32PairBN;
  const int split = tc_f32_split(row_tiles_est * g.n_col_tiles, s.n_pairs, c.d_ff / kF32BK, y_copies);
  *y_split = split;
  if (s.only == 1) return SWAPMOE_OK;
  g.C = y; g.split_stride = y_copy_stride; g.n_split = split; g.early_b = 1;
  g.ldc = c.d_model; g.k_blocks = c.d_ff / kF32BK / split;
  g.b_rows_per_phys = c.d_model; g.b_rows_gate = 0;
  work = (long long)max_tiles * g.n_col_tiles * split;
  grid = 2 * (int)(work > s.n_pairs ? s.n_pairs : work);
  if (launch_kernel(tc_gemm_f32_pair_kernel<kTcEpiF32>, dim3(grid), dim3(kF32PairThreads), kF32PairSmemBytes, st,
                    pdl && between == nullptr, s.map_h, s.map_wout_pair, g) != cudaSuccess)
    return SWAPMOE_ERR_CUDA;
  ++*launches;
  return SWAPMOE_OK;
}

}  // namespace swapmoe
