// Launch logic of the two grouped GEMMs of a bf16 layer on one CTA per tile (tc_gemm_kernel), and the rule that sends them to
// CTA pairs.
// SwapMoE Section 2: E_i(x) per slot.
#pragma once
#include "gemm_tc_pair.cuh"

namespace swapmoe {

// Weight tiles per token tile where a grouped GEMM (which = 1 or 2) runs on CTA pairs, 0: one CTA per tile.  Pairs take
// every forward of more than 64 (token, expert) pairs (up to there the small-batch kernel fills the SMs better: SwiGLU 960 x
// 2624, four slots, 13 tokens 31.0 us per forward against 39.6) whose matrices leave at most a fifth of the width of all
// weight tiles together empty (tc_wide_ok).  us per forward, the tree in which they
// took slots of 160 rows and more only / here: 768 x 3072, 16 slots, 70 tokens 48.6 / 42.7, 500 53.2 / 46.5, 2048 55.8 / 54.3, 5000
// 92.8 / 83.7; 512 x 2048 at 90 33.8 / 31.7; 1536 x 1088, 48 slots, 110 tokens 95.7 / 93.5; 1024 x 512 top-4, 64 slots, 3000 92.4 /
// 87.7; SwiGLU top-2, four slots, 1024 x 3584, 300 62.8 / 50.6, 4096 x 14336, 700 647 / 568.
inline int tc_pair_cols(const swapmoe_config_t& c, int which, long long pairs, int min_rows) {
  const int width = which == 2 ? c.d_model : c.act == SWAPMOE_ACT_SWIGLU ? 2 * c.d_ff : c.d_ff;
  if (pairs <= 64 || pairs < (long long)min_rows * c.K || !tc_wide_ok(width)) return 0;
  return (width + 2 * kTcBM - 1) / (2 * kTcBM);
}

// What a forward's row count says about either GEMM on one CTA per tile.
struct TcRowPlan {
  int ia, a_box_bytes, row_group;
  long long row_tiles_est;
};
inline void tc_plan_rows(const swapmoe_config_t& c, int n_tokens, int row_group_forced, TcRowPlan* p) {
  // row tiles expected: every touched slot (at most min(pairs, K)) has at least one, and large slots
  // have pairs / 128 in total plus on average half a ragged tile each
  const long long pairs = (long long)n_tokens * c.top_k;
  const long long touched = pairs < c.K ? pairs : c.K;
  const long long by_rows = pairs / kTcBM + touched / 2;
  p->row_tiles_est = touched > by_rows ? touched : by_rows;
  // no tile holds more rows than there are pairs: small batches fetch only the rows that can be valid
  p->ia = 0;
  while (p->ia < 3 && (kTcBM >> (p->ia + 1)) >= pairs) ++p->ia;
  p->a_box_bytes = (kTcBM >> p->ia) * kTcBK * 2;
  // Large activation matrices (tens of MB) are walked in groups of 32 row tiles so that a group's
  // rows stay in L2 across its column tiles; small ones are a single group.
  p->row_group = 1 << 30;
  if (row_group_forced > 0) p->row_group = row_group_forced;
  else if (pairs * (long long)c.d_model * 2 > (48ll << 20)) p->row_group = 32;
}
// How tc_gemm1 launches GEMM-1 for a forward of n_tokens.
struct TcGemm1Plan : TcRowPlan {
  int i1, bn1;              // index into kBn1Options, tile width
  int n_col_tiles, grid;
};
inline bool tc_plan_gemm1(const TcState& s, const swapmoe_config_t& c, int n_tokens, int max_tiles, int row_group_forced,
                          TcGemm1Plan* p) {
  const bool swiglu = c.act == SWAPMOE_ACT_SWIGLU;
  tc_plan_rows(c, n_tokens, row_group_forced, p);
  // (SwiGLU counts the rows of both matrices; with one matrix's the model saw half the tiles: 13 tokens, d_model 4096,
  // d_ff 14336, four slots, GEMM-1 alone 187 us at 448 tiles on 148 SMs, 174 at 896 narrower ones)
  p->i1 = tc_pick_bn(kBn1Options, 3, swiglu ? 2 * c.d_ff : c.d_ff, p->row_tiles_est, s.sm_count, p->a_box_bytes,
                     swiglu ? 64 : 32);
  if (p->i1 < 0) return false;
  p->bn1 = kBn1Options[p->i1];
  const int out1 = swiglu ? p->bn1 / 2 : p->bn1;
  p->n_col_tiles = (c.d_ff + out1 - 1) / out1;
  const long long work = (long long)max_tiles * p->n_col_tiles;
  p->grid = work > s.sm_count ? s.sm_count : (int)work;
  return true;
}

// GEMM-1, h = act(xp * W_in^T), over a list of 128-row tiles.  Its k-loop is short (d_model / 64 blocks), so its epilogue must
// overlap the next tile's MMAs: two TMEM buffers.
inline int32_t tc_gemm1(TcState& s, const swapmoe_config_t& c, void* h, const TileDesc* tiles, const int32_t* n_tiles,
                        int max_tiles, int n_tokens, int32_t* status, cudaStream_t st, bool pdl, int row_group_forced) {
  if (!s.enabled || !s.arena_bound) return SWAPMOE_ERR_NOT_READY;
  const bool swiglu = c.act == SWAPMOE_ACT_SWIGLU;
  TcGemm1Plan plan;
  if (!tc_plan_gemm1(s, c, n_tokens, max_tiles, row_group_forced, &plan)) return SWAPMOE_ERR_UNSUPPORTED;
  TcGemmArgs g;
  g.C = h; g.status = status; g.ldc = c.d_ff; g.tiles = tiles; g.n_tiles = n_tiles;
  g.n_col_tiles = plan.n_col_tiles;
  g.k_blocks = c.d_model / kTcBK;
  g.b_rows_per_phys = swiglu ? 2 * c.d_ff : c.d_ff;
  g.b_rows_gate = swiglu ? c.d_ff : 0;
  g.row_pair = nullptr; g.gate = nullptr; g.top_k = c.top_k;
  g.row_group = plan.row_group;
  g.a_box_bytes = plan.a_box_bytes;
  g.early_b = 0;
  static const TcGemmKernel kernels[2][3] = {
      {tc_gemm_kernel<256, kTcEpiReluBf16>, tc_gemm_kernel<128, kTcEpiReluBf16>, tc_gemm_kernel<64, kTcEpiReluBf16>},
      {tc_gemm_kernel<256, kTcEpiSwigluBf16>, tc_gemm_kernel<128, kTcEpiSwigluBf16>,
       tc_gemm_kernel<64, kTcEpiSwigluBf16>}};
  static const int smem[3] = {TcSmem<256>::kBytes, TcSmem<128>::kBytes, TcSmem<64>::kBytes};
  return launch_kernel(kernels[swiglu ? 1 : 0][plan.i1], dim3(plan.grid), dim3(kTcThreads), smem[plan.i1], st, pdl,
                       s.map_xp[plan.ia], s.map_win[plan.i1], g) == cudaSuccess ? SWAPMOE_OK : SWAPMOE_ERR_CUDA;
}

// GEMM-2, y = h * W_out^T, or out = gate * y for top-1 layers (no combine kernel is needed then).
inline int32_t tc_gemm2(TcState& s, const swapmoe_config_t& c, void* dst, const TileDesc* tiles, const int32_t* n_tiles,
                        int max_tiles, const int32_t* row_pair, const float* mgate, int n_tokens, int32_t* status,
                        cudaStream_t st, bool pdl, int row_group_forced) {
  if (!s.enabled || !s.arena_bound) return SWAPMOE_ERR_NOT_READY;
  const bool scatter = c.top_k == 1;
  TcRowPlan rp;
  tc_plan_rows(c, n_tokens, row_group_forced, &rp);
  const int i2 = tc_pick_bn(kBn2Options, 4, c.d_model, rp.row_tiles_est, s.sm_count, rp.a_box_bytes, 32);
  if (i2 < 0) return SWAPMOE_ERR_UNSUPPORTED;
  const int bn2 = kBn2Options[i2];
  TcGemmArgs g;
  g.C = dst; g.tiles = tiles; g.n_tiles = n_tiles; g.status = status; g.ldc = c.d_model;
  g.n_col_tiles = (c.d_model + bn2 - 1) / bn2;
  g.k_blocks = c.d_ff / kTcBK;
  g.b_rows_per_phys = c.d_model;
  g.b_rows_gate = 0;
  g.row_pair = row_pair; g.gate = mgate; g.top_k = c.top_k;
  g.row_group = rp.row_group;
  g.a_box_bytes = rp.a_box_bytes;
  g.early_b = 1;
  const long long work = (long long)max_tiles * g.n_col_tiles;
  const int grid = work > s.sm_count ? s.sm_count : (int)work;
  static const TcGemmKernel kernels[2][4] = {
      {tc_gemm_kernel<256, kTcEpiF32>, tc_gemm_kernel<128, kTcEpiF32>, tc_gemm_kernel<64, kTcEpiF32>,
       tc_gemm_kernel<32, kTcEpiF32>},
      {tc_gemm_kernel<256, kTcEpiScatterBf16>, tc_gemm_kernel<128, kTcEpiScatterBf16>, tc_gemm_kernel<64, kTcEpiScatterBf16>,
       tc_gemm_kernel<32, kTcEpiScatterBf16>}};
  static const int smem[4] = {TcSmem<256>::kBytes, TcSmem<128>::kBytes, TcSmem<64>::kBytes, TcSmem<32>::kBytes};
  return launch_kernel(kernels[scatter ? 1 : 0][i2], dim3(grid), dim3(kTcThreads), smem[i2], st, pdl, s.map_h[rp.ia],
                       s.map_wout[i2], g) == cudaSuccess ? SWAPMOE_OK : SWAPMOE_ERR_CUDA;
}

}  // namespace swapmoe
