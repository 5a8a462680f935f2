// Gate of one token tile, shared by both router kernels (SwapMoE Section 2: G(x); Fig. 4:
// Masked Gating; Eq. 1: importance terms).  Input: the tile's logits in shared memory; output:
// both selections with their gate values, the slot of every pair, ||x||, and the CTA's partial
// sums for the slot scan.  256 threads; tok = 32, 64 or 128 tokens per CTA.
#pragma once
#include "common.cuh"
#include "permute.cuh"
#include "router_args.cuh"

namespace swapmoe {

constexpr int kGateTokMax = 128;   // largest token tile
constexpr int kGateThreads = 256;

// Order-preserving key of a logit, as gate_key (equal for -0 and +0, never 0), with NaN as -inf: a logit that is NaN is chosen
// only if no number is left.  (gate_key promises nothing about NaN: the sign of the sum it starts from is the compiler's
// choice, and NaN came out above the negative logits.)
__device__ __forceinline__ uint32_t gate_scan_key(float x) {
  const uint32_t b = __float_as_uint(fmaxf(x, -INFINITY));
  return (b & 0x80000000u) ? 0u - b : b + 0x80000000u;
}

// Running list of the N best logits, descending, as order-preserving keys (gate_scan_key; 0 = nothing).  A candidate goes
// below every entry that is >= it, so equal values stay in arrival (= expert index) order.  Without branches: on a warp of
// 32 tokens some token takes nearly every candidate, so a branch only adds its own cost (256 experts, top-4, 64
// tokens per CTA: logits copy and this scan 23 -> 9.2 us).
template <int N>
struct TopK {
  uint32_t v[N];
  int e[N];
  __device__ __forceinline__ void init() {
#pragma unroll
    for (int j = 0; j < N; ++j) { v[j] = 0u; e[j] = -1; }
  }
  __device__ __forceinline__ void push(uint32_t cv, int ce) {
    bool beats[N];
#pragma unroll
    for (int j = 0; j < N; ++j) beats[j] = cv > v[j];
#pragma unroll
    for (int j = N - 1; j > 0; --j) {
      v[j] = beats[j - 1] ? v[j - 1] : (beats[j] ? cv : v[j]);
      e[j] = beats[j - 1] ? e[j - 1] : (beats[j] ? ce : e[j]);
    }
    v[0] = beats[0] ? cv : v[0];
    e[0] = beats[0] ? ce : e[0];
  }
};

// The logit behind a list entry (an empty one, possible with fewer allowed experts than k, weighs nothing).
__device__ __forceinline__ float gate_entry_value(const float* row, int e) { return e >= 0 ? row[e] : -INFINITY; }

// The best N of the allowed experts [e_lo, e_hi) (e_lo a multiple of 32) of one logits row; at most seven floats
// behind the row's end are read.
template <int N>
__device__ __forceinline__ void gate_scan(const float* row, const uint32_t* allow, int e_lo, int e_hi, uint32_t* cand_v,
                                          int* cand_e) {
  TopK<N> tk;
  tk.init();
#pragma unroll 1
  for (int e0 = e_lo; e0 < e_hi; e0 += 8) {
    const uint32_t w = (allow[e0 >> 5] >> (e0 & 31)) & 0xffu;
    if (w == 0u) continue;                         // the same for all threads of a warp
    float l[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) l[i] = row[e0 + i];
#pragma unroll
    for (int i = 0; i < 8; ++i) tk.push((w >> i) & 1u ? gate_scan_key(l[i]) : 0u, e0 + i);
  }
#pragma unroll
  for (int j = 0; j < kMaxTopK; ++j) {
    cand_v[j] = j < N ? tk.v[j < N ? j : 0] : 0u;
    cand_e[j] = j < N ? tk.e[j < N ? j : 0] : -1;
  }
}

// Shared-memory arrays of the gate, carved from one block by gate_smem_carve().
struct GateSmem {
  int* pe;             // [tok*k] unmasked expert per pair
  int* ps;             // [tok*k] slot per pair
  float* pt;           // [tok*k] Eq. (1) term per pair
  float* pm;           // [tok*k] Eq. (1) term under the masked routing
  float* snorm;        // [tok] ||x_t||
  int* s_e2s;          // [256] expert -> slot
  float* s_enorm;      // [256] ||E_e||
  uint32_t* s_mask;    // [2][8] valid / resident expert bits
  uint32_t* cand_v;    // [256 threads][kMaxTopK] per-thread top-k keys
  int* cand_e;         //  ... and experts
  float* part_den;     // [256] partial softmax denominators
  float* s_m;          // [tok][2] row maximum per gate
};

__host__ __device__ constexpr size_t gate_smem_bytes() {
  return (size_t)4 * (4 * kGateTokMax * kMaxTopK + kGateTokMax + 2 * kMaxE + 16 +
                      2 * kGateThreads * kMaxTopK + kGateThreads + 2 * kGateTokMax);
}

__device__ __forceinline__ GateSmem gate_smem_carve(void* base) {
  GateSmem g;
  g.pe = static_cast<int*>(base);
  g.ps = g.pe + kGateTokMax * kMaxTopK;
  g.pt = reinterpret_cast<float*>(g.ps + kGateTokMax * kMaxTopK);
  g.pm = g.pt + kGateTokMax * kMaxTopK;
  g.snorm = g.pm + kGateTokMax * kMaxTopK;
  g.s_e2s = reinterpret_cast<int*>(g.snorm + kGateTokMax);
  g.s_enorm = reinterpret_cast<float*>(g.s_e2s + kMaxE);
  g.s_mask = reinterpret_cast<uint32_t*>(g.s_enorm + kMaxE);
  g.cand_v = g.s_mask + 16;
  g.cand_e = reinterpret_cast<int*>(g.cand_v + kGateThreads * kMaxTopK);
  g.part_den = reinterpret_cast<float*>(g.cand_e + kGateThreads * kMaxTopK);
  g.s_m = g.part_den + kGateThreads;
  return g;
}

// Copies the slot table and the expert norms into shared memory and builds the bit masks of
// valid and of resident experts.  All 256 threads; the caller synchronises afterwards.
__device__ __forceinline__ void gate_load_tables(const RouterArgs& a, const GateSmem& g) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // (a table entry outside [0, K) - possible only when the caller hands in its own table, as swapmoe_route_static
  // allows - counts as "not resident")
  for (int e = tid; e < kMaxE; e += kGateThreads) {
    const int sl = e < a.E ? a.e2s[e] : -1;
    g.s_e2s[e] = sl < a.K ? sl : -1;
    g.s_enorm[e] = e < a.E ? a.enorm[e] : 0.f;
  }
  // warp w builds word w of the valid-expert mask and of the resident-expert mask
  const int e = warp * 32 + lane;
  int sl = e < a.E ? a.e2s[e] : -1;
  if (sl >= a.K) sl = -1;
  const uint32_t wv = __ballot_sync(0xffffffffu, e < a.E), wr = __ballot_sync(0xffffffffu, sl >= 0);
  if (lane == 0) { g.s_mask[warp] = wv; g.s_mask[8 + warp] = wr; }
}

// The gate proper.  slog holds the tile's logits, row stride E + 1 floats (with at least 8
// floats readable behind the last row); g.snorm holds ||x_t|| of the tile's rows and
// gate_load_tables() has run, both made visible by a __syncthreads() in the caller.  When
// `failed` is set (the producer gave up on a bounded wait) zeros are written instead.
// scan_stage / scan_stage_bytes: shared memory that the last CTA may use to stage the scan
// inputs (may overlap slog).
//
// Thread t serves token t % tok.  Its group g = t / tok splits into the gate it evaluates
// (first half of the groups: off-the-shelf gate; second half: masked gate) and the share of
// the expert range it scans (whole 32-expert chunks, contiguous and ascending per share).
__device__ __forceinline__ void gate_epilogue(const RouterArgs& a, const GateSmem& g, const float* slog,
                                              int tok, int tok0, bool failed, void* scan_stage,
                                              int scan_stage_bytes) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int E = a.E, k = a.k;
  {
    // coalesced copy of the logits: a warp writes a token's row; four rows are in flight
    const int rows = min(tok, a.T - tok0);
    for (int t0 = warp * 4; t0 < rows; t0 += (kGateThreads / 32) * 4) {
      for (int e = lane; e < E; e += 32) {
        float v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = slog[(size_t)min(t0 + q, tok - 1) * (E + 1) + e];
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (t0 + q < rows) a.logits[(size_t)(tok0 + t0 + q) * E + e] = failed ? 0.f : v[q];
      }
    }
  }
  // tok is a power of two (32, 64, 128): shifts, not integer divisions, which cost dozens of
  // dependent instructions each in code that runs once
  const int tok_shift = 31 - __clz(tok);
  const int tl = tid & (tok - 1), grp = tid >> tok_shift;
  const int parts = (kGateThreads >> tok_shift) >> 1;       // threads per token and gate: 1, 2 or 4
  const bool masked = grp >= parts;
  const int part = masked ? grp - parts : grp;
  const int token = tok0 + tl;
  const float* row = slog + (size_t)tl * (E + 1);
  const uint32_t* allow = g.s_mask + (masked ? 8 : 0);
  const int n_chunks = (E + 31) >> 5, cpp = (n_chunks + parts - 1) >> (parts == 4 ? 2 : parts - 1);
  const int e_lo = min(E, part * cpp * 32), e_hi = min(E, (part + 1) * cpp * 32);
  {
    uint32_t* cv = g.cand_v + tid * kMaxTopK;
    int* ce = g.cand_e + tid * kMaxTopK;
    if (k == 1) gate_scan<1>(row, allow, e_lo, e_hi, cv, ce);
    else if (k == 2) gate_scan<2>(row, allow, e_lo, e_hi, cv, ce);
    else gate_scan<kMaxTopK>(row, allow, e_lo, e_hi, cv, ce);
  }
  __syncthreads();
  if (threadIdx.x == 0) SWAPMOE_STAMP(0, 6);
  // merge the shares of one (token, gate) in ascending expert order: a candidate only displaces
  // an entry it strictly beats, so equal logits keep the lowest expert index
  TopK<kMaxTopK> fin;
  fin.init();
  if (part == 0) {
    for (int pp = 0; pp < parts; ++pp) {
      const int src = (((masked ? parts : 0) + pp) * tok + tl) * kMaxTopK;
#pragma unroll
      for (int j = 0; j < kMaxTopK; ++j)
        if (j < k) fin.push(g.cand_v[src + j], g.cand_e[src + j]);      // (key 0, nothing there, displaces nothing)
    }
    g.s_m[tl * 2 + (masked ? 1 : 0)] = gate_entry_value(row, fin.e[0]);
  }
  __syncthreads();
  if (threadIdx.x == 0) SWAPMOE_STAMP(0, 7);
  {
    const float m = g.s_m[tl * 2 + (masked ? 1 : 0)];
    float den = 0.f;
    if (!a.renorm) {
      // eight interleaved partial sums: short dependency chains and a tree-shaped total
      float acc8[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
      for (int e0 = e_lo; e0 < e_hi; e0 += 8) {
        const uint32_t w = allow[e0 >> 5] >> (e0 & 31);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float t = __expf(row[e0 + i] - m);
          acc8[i] += ((w >> i) & 1u) ? t : 0.f;
        }
      }
      den = ((acc8[0] + acc8[1]) + (acc8[2] + acc8[3])) + ((acc8[4] + acc8[5]) + (acc8[6] + acc8[7]));
    }
    g.part_den[tid] = den;
  }
  __syncthreads();
  if (threadIdx.x == 0) SWAPMOE_STAMP(0, 8);
  if (part == 0) {
    const float m = gate_entry_value(row, fin.e[0]);
    float den = 0.f;
    if (a.renorm) {
#pragma unroll
      for (int j = 0; j < kMaxTopK; ++j)
        if (j < k) den += expf(gate_entry_value(row, fin.e[j]) - m);
    } else {
      for (int pp = 0; pp < parts; ++pp) den += g.part_den[((masked ? parts : 0) + pp) * tok + tl];
    }
    const float xn = g.snorm[tl];
#pragma unroll
    for (int j = 0; j < kMaxTopK; ++j) {
      if (j < k) {
        const int pl = tl * k + j;
        const size_t p = (size_t)token * k + j;
        const float gv = failed ? 0.f : expf(gate_entry_value(row, fin.e[j]) - m) / den;
        const int e = fin.e[j];
        if (!masked) {
          if (token < a.T) {
            a.uidx[p] = e; a.ugate[p] = gv;
            g.pe[pl] = e; g.pt[pl] = xn * fabsf(gv) * g.s_enorm[e];   // one term of Eq. (1)
          } else {
            g.pe[pl] = -1; g.pt[pl] = 0.f;
          }
        } else {
          if (token < a.T && e < 0) {
            // fewer resident experts than top_k (a caller-supplied table: the layer API rules it out): the pair
            // is routed nowhere instead of indexing the tables with -1
            a.midx[p] = -1; a.mgate[p] = 0.f; a.slot[p] = -1;
            g.ps[pl] = -1; g.pm[pl] = 0.f;
          } else if (token < a.T) {
            const int sl = g.s_e2s[e];
            a.midx[p] = e; a.mgate[p] = gv; a.slot[p] = sl;
            g.ps[pl] = sl; g.pm[pl] = xn * fabsf(gv) * g.s_enorm[e];
          } else {
            g.ps[pl] = -1; g.pm[pl] = 0.f;
          }
        }
      }
    }
    if (!masked && token < a.T) a.xnorm[token] = xn;
  }
  __syncthreads();
  if (threadIdx.x == 0) SWAPMOE_STAMP(0, 9);
  // Per-CTA partial sums: a thread owns an expert (or a slot) and walks the tile's pairs in order, four per shared-memory
  // load that all threads share - the same association as the small-batch routers, whatever the scheduling.  (A warp per
  // selected expert, lanes over the pairs and a shuffle tree, took 14 us at 256 experts, 64 slots and 256 pairs, this takes 4.3; 3.3 -> 1.0 us at 128, 32 and 64.)
  const int nq = tok * k >> 2;                             // tok is a multiple of 32
  const int n_cols = E + a.K;
  for (int c = tid; c < n_cols; c += kGateThreads) {
    const bool by_slot = c >= E;
    const int id = by_slot ? c - E : c;
    const int4* ids = reinterpret_cast<const int4*>(by_slot ? g.ps : g.pe);
    const float4* terms = reinterpret_cast<const float4*>(by_slot ? g.pm : g.pt);
    float sum = 0.f;
    int n = 0;
#pragma unroll 4
    for (int q = 0; q < nq; ++q) {
      const int4 i4 = ids[q];
      const float4 t4 = terms[q];
      if (i4.x == id) { sum += t4.x; ++n; }
      if (i4.y == id) { sum += t4.y; ++n; }
      if (i4.z == id) { sum += t4.z; ++n; }
      if (i4.w == id) { sum += t4.w; ++n; }
    }
    if (by_slot) {
      a.cta_hist[(size_t)blockIdx.x * a.K + id] = n;
      if (a.cta_mimp) a.cta_mimp[(size_t)blockIdx.x * a.K + id] = sum;
    } else {
      a.cta_imp[(size_t)blockIdx.x * E + id] = sum;
      if (a.cta_cnt) a.cta_cnt[(size_t)blockIdx.x * E + id] = (float)n;
    }
  }
  if (threadIdx.x == 0) SWAPMOE_STAMP(0, 11);
  finish_router_cta(a.scan, scan_stage, scan_stage_bytes);
  if (threadIdx.x == 0) SWAPMOE_STAMP(0, 12);
}

}  // namespace swapmoe
