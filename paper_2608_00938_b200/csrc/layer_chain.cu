// The row-local part of the decoder layers (Section 3.2) as one kernel between two cross-attentions:
//
//   [x += attn Wo_cross, LayerNorm, feed-forward, x += ...]  of the layer whose cross-attention is done    ("post")
//   [LayerNorm, QKV, self-attention over the parent-addressed cache, x += attn Wo, LayerNorm, cross-Q]  of the next one ("pre")
//
// What bounds a decode of a few hundred rows is the number of dependent launches: every product is 1 us of work behind
// 2 to 3 us of launch, first loads and drain, eight to eleven of them per layer.  None of these stages mixes rows, so a
// cluster of C = d_model / 64 CTAs takes 64 rows through all of them and the rows never leave its shared memory:
// CTA i owns columns 64 i .. 64 i + 63 of the residual stream, the heads in them, and 1 / C of the feed-forward's hidden
// columns.  The weights (a C-th of the layer per CTA) stream through a TMA ring that runs ahead of the arithmetic across
// stage boundaries; activations go from CTA to CTA as bulk copies between shared memories, one 64 x 64 tile per CTA
// and exchange, which is a k-block of the next product in the operand layout.
//
// A stage: the operand tile (C k-blocks of up to 64 rows, each with its own barrier, so that the products start with the
// CTA's own k-block) -> tcgen05.mma (M = 64, fp32 in TMEM) -> eight warps, 16 rows and 32 columns each (a row of an M = 64
// accumulator is one of the first 16 lanes of a warp's 32), which keep their part of the residual stream in registers -> next
// tile.  The feed-forward's second product is split along K: a pair of CTAs (2p, 2p + 1) shares its hidden columns, and each
// multiplies them by the weights of the owners of its own parity; the partial sums go to the owners (st.async) and are
// added there in a fixed order.
//
// Every role runs its stages through one loop body: written out one by one they take a launch through far more code, of which
// it executes every line once (a step of 2 layers of 128: 55 us, of 4 layers of 512 at 512 rows: 187; so 47 and 167).  A tile
// has no more rows than it takes to spread them over the clusters that fit, and only rows in use are sent.  What bounds a
// layer is the latency of its stages, one behind the other.  4 x 512, third step, a launch between two cross-attentions, by
// the clock of its first CTA (us; 16 rows in tiles of 8 / 512 in tiles of 40 / 960 in tiles of 64): the rows and their
// parents 1.4 / 1.4 / 1.8; Wo_cross and the first exchange 1.7 / 1.6 / 1.6; hidden columns 4.9 / 6.1 / 6.5; their product, the
// partial sums and the next exchange 5.3 / 5.3 / 6.5; QKV and self-attention 5.5 / 6.8 / 8.9 (16 rows of the first step, without a
// prefix: 4.6); Wo 2.1 / 2.9 / 3.8; the queries 2.0 / 2.8 / 2.9; leaving, up to the next kernel's start 2.3 / 3.5 / 4.0.  No unit is
// busy (512 rows: tensor pipe in 23 % of the cycles of the SMs that have a CTA, L1 22 %).
// Measured and left out: sixteen epilogue warps of 16 columns (167 -> 204 us), a deeper ring (165), all columns of a k-block in
// one MMA (164, d_model 128: 47 -> 50), four chains instead of two for a score (no change), tiles of at least 16 or 32 rows
// (4 x 512, 16 rows 131 -> 132.5 us a step, 32 rows 133 -> 133.5 and 142).
//
// With an fp32 stream the final LayerNorm comes out of the last launch as well (2 x 128, three steps of up to 16 rows: 174 -> 168
// us a search); the bf16 stream's is folded into the output head.
//
// Row statistics travel with the tiles as (mean, sum of squared deviations) per 32 columns and are merged by the reader.
//
// Shared memory that a bulk copy reads may be written again only once the copy is known to have arrived, and that shows at its
// destination alone.  What says so here, for each source: a k-block of the operand tile, a_free, which every CTA gives behind
// the products that read the copy; the hidden k-blocks, over which the cache's prefix comes in, and the row statistics, see
// there.  Every copy, and every arrival on another CTA's barrier, is waited for by its destination in front of the final
// cluster barrier.
#include "common.cuh"
#include "tc.cuh"
#include <initializer_list>

namespace grace {

constexpr int kLcRows = 64;
constexpr int kLcTile = 64 * 64 * 2;                       // 64 rows (of x or of a weight) x 64 columns, 128-byte swizzle
constexpr int kLcStages = 5;                               // ring: two weight tiles each
constexpr int kLcThreads = 320;                            // eight epilogue warps, TMA, MMA
constexpr int kLcMaxHidden = 4;                            // hidden k-blocks of a CTA (d_ffn / C / 64)

struct LayerChainMaps {
  CUtensorMap attn, w_oc, w_1, w_2;                        // post
  CUtensorMap w_qkv, w_o, w_qc;                            // pre
};
struct LayerChainParams {
  int post, pre, embed;
  int R, D, hidden_blocks;                                 // rows; d_model; d_ffn / C / 64
  int t, M_t, d_h, tile_rows;                              // tile_rows: of a cluster, a multiple of 8 up to 64
  int beam[4];
  int64_t R_max, slab_stride;
  float eps, scale;
  const int32_t* token; const uint16_t* embed_rows; const uint16_t* pos; int embed_count;
  uint16_t* x_bf16; float* x_f32;                          // one of them
  uint16_t* q_cross;                                       // [R][D]
  uint16_t* slabs;                                         // [L][R_max][3][D]
  const int32_t* parents;                                  // [L + 1][R_max]
  int32_t* d_status;
  const float *cb_1, *cs_1, *cb_qkv, *cs_qkv, *cb_qc, *cs_qc;              // folded: bias, column sums (or NULL)
  const float *ln1_g, *ln1_b, *ln2_g, *ln2_b, *ln3_g, *ln3_b;              // not folded; behind the last layer ln1 is the final one,
  uint16_t* h_final;                                       //   whose rows go here, [R][D]
};

template <int C>
struct LayerChainSmem {
  static constexpr int kA = 0;                                              // [C] k-blocks of the operand tile
  static constexpr int kH = kA + C * kLcTile;                               // [2][kLcMaxHidden] hidden k-blocks, own and partner's
  static constexpr int kW = kH + 2 * kLcMaxHidden * kLcTile;                // ring
  static constexpr int kStats = kW + kLcStages * 2 * kLcTile;               // [C][2][64] float2
  static constexpr int kVec = kStats + C * 2 * kLcRows * 8;                 // column vectors: [512] + [512] floats
  static constexpr int kScores = kVec + 1024 * 4;                           // [2][64] float4
  static constexpr int kBars = kScores + 2 * kLcRows * 16;
  static constexpr int kTotal = kBars + 512;
  static_assert(kTotal <= 227 * 1024 && kTotal >= tc::kTmemAllSmem, "");
};

__device__ __forceinline__ void dsmem_bulk_copy(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "r"(tc::smem_addr(src)), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void dsmem_st_async(uint32_t dst, uint32_t bar, const uint32_t* v) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
               ::"r"(dst), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(bar) : "memory");
}
// One arrival on the barrier at this offset in every CTA of the mask once the MMAs issued so far by this thread are done.
__device__ __forceinline__ void mma_commit_cluster(uint64_t* bar, uint16_t mask) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(tc::smem_addr(bar)), "h"(mask) : "memory");
}

// F32: fp32 residual stream, LayerNorm applied to the tiles (as the LayerNorm kernel in front of a GEMM does); otherwise bf16
// stream, LayerNorm folded into the products.
template <int C, bool F32>
__global__ void __launch_bounds__(kLcThreads, 1)
layer_chain_kernel(const __grid_constant__ LayerChainMaps maps, const __grid_constant__ LayerChainParams p) {
  using S = LayerChainSmem<C>;
  extern __shared__ __align__(1024) uint8_t smem_chain[];
  if ((tc::smem_addr(smem_chain) & 1023u) != 0) {          // the swizzled tiles need it; same answer in every CTA
    if (threadIdx.x == 0 && blockIdx.x == 0) atomicAdd(&tc::g_tc_timeouts, 1);
    return;
  }
  uint8_t* const tile_a = smem_chain + S::kA;
  uint8_t* const tile_h = smem_chain + S::kH;
  uint8_t* const ring = smem_chain + S::kW;
  float2* const stats = reinterpret_cast<float2*>(smem_chain + S::kStats);
  float* const vec = reinterpret_cast<float*>(smem_chain + S::kVec);
  float* const scores = reinterpret_cast<float*>(smem_chain + S::kScores);       // [2][64][4]
  uint64_t* const w_full = reinterpret_cast<uint64_t*>(smem_chain + S::kBars);
  uint64_t* const w_empty = w_full + kLcStages;
  uint64_t* const a_full = w_empty + kLcStages;            // [C] a k-block of the operand tile has landed
  uint64_t* const a_free = a_full + C;                     // every CTA of the cluster is done with its operand tile
  uint64_t* const acc_full = a_free + 1;                   // [2] alternating accumulators
  uint64_t* const h_full = acc_full + 2;                   // [2][kLcMaxHidden]
  uint64_t* const part_full = h_full + 2 * kLcMaxHidden;   // the other CTAs' partial sums
  uint64_t* const stats_full = part_full + 1;              // the other CTAs' statistics
  uint32_t* const tmem_slot = reinterpret_cast<uint32_t*>(stats_full + 1);
  volatile int* const abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = __shfl_sync(kFullMask, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const int rank = (int)(blockIdx.x % C);                  // in the cluster
  const int row0 = (int)(blockIdx.x / C) * p.tile_rows;
  const int rows = min(p.tile_rows, p.R - row0);           // in use
  const int rows8 = (rows + 7) & ~7;                       // sent: whole groups of eight, 1 KB of a tile each
  const uint32_t tile_bytes = (uint32_t)rows8 * 128u;
  const int n_h = p.hidden_blocks;                         // hidden k-blocks of this CTA
  constexpr int kSources = C / 2 - 1;                      // CTAs that send this one partial sums
  auto kb_of = [&](int j) { return (rank + j) & (C - 1); };    // products start with the CTA's own k-block

  if (threadIdx.x == 0) {
    for (int s = 0; s < kLcStages; ++s) { tc::mbar_init(w_full + s, 1); tc::mbar_init(w_empty + s, 1); }
    for (int k = 0; k < C; ++k) tc::mbar_init(a_full + k, 1);
    tc::mbar_init(a_free, C);
    tc::mbar_init(acc_full, 1);
    tc::mbar_init(acc_full + 1, 1);
    for (int k = 0; k < 2 * kLcMaxHidden; ++k) tc::mbar_init(h_full + k, 1);
    tc::mbar_init(part_full, 1);
    tc::mbar_init(stats_full, 1);
    *abort_flag = 0;
    tc::fence_mbar_init();
  }
  if (warp == 8) tc::tmem_alloc(tmem_slot, 512);
  tc::tc_fence_before();
  __syncthreads();
  // Behind the allocation: no kernel behind this one can take TMEM first.  In front of the wait: the ring fills with weights,
  // and in a later launch of a step the vectors are read, before the kernel in front has completed.  Whoever wrote them has: the
  // step's first launch waits before it reads either, and between two launches lies a cross-attention, which lets the second one
  // start only behind its own wait for the first.
  pdl_trigger();
  tc::cluster_sync_all();                                  // every CTA's barriers exist before the first copy into it
  tc::tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // TMEM columns: [0, 256) hidden columns, QKV; [256, 512) everything else
  constexpr uint32_t kAccLow = 0, kAccHigh = 256;

  // A wait that gives up leaves the roles running, with the abort flag set, so that every barrier is still reached; later
  // waits of the CTA then give up at once.  No address depends on what was waited for.
  // The producer's and the issuer's warp walk their loops whole and one elected lane issues (warp-uniform control flow keeps
  // coordinates and descriptors in uniform registers).
  // The products in order, for the producer and the issuer: Wo_cross; the hidden columns, 128 at a time; the second product,
  // for two owners at a time; Q and K; V; Wo; cross-Q.
  const int n_pass = (n_h + 1) >> 1, n_post = 1 + n_pass + (C >= 4 ? C / 4 : 1);
  const int g_first = p.post ? 0 : n_post, g_last = p.pre ? n_post + 4 : n_post;
  // wide: 128 output columns and a k-block a stage; otherwise 64 output columns and two k-blocks a stage
  auto is_hidden = [&](int g) { return g > n_pass && g < n_post; };
  auto is_wide = [&](int g) { return is_hidden(g) ? C >= 4 : (g == n_post || (g >= 1 && g <= n_pass && 2 * g <= n_h)); };
  auto stages_of = [&](int g) { return (is_hidden(g) ? 2 * n_h : C) >> (is_wide(g) ? 0 : 1); };
  auto owner_of = [&](int i) { return C >= 4 ? 4 * (((rank >> 2) + 1 + i) % (C >= 4 ? C / 4 : 1)) + (rank & 1) : rank; };    // and two further
  if (warp == 8) {
    // ---- weights ----
    int it = 0, slot = 0, lap = 0;
    auto activations = [&]() {                             // the cross-attention's output: the first operand tile
      pdl_wait();
      if (!p.post) return;
#pragma unroll 1
      for (int j = 0; j < C; ++j) {
        const int kb = kb_of(j);
        if (tc::elect_one()) {
          tc::mbar_expect_tx(a_full + kb, kLcTile);
          tc::tma_load_2d(tile_a + kb * kLcTile, &maps.attn, a_full + kb, kb * 64, row0);
        }
        __syncwarp();
      }
    };
    bool waited = false;
    if (p.embed) { pdl_wait(); waited = true; }            // first kernel of a step: its weights may just have been written
#pragma unroll 1
    for (int g = g_first; g < g_last; ++g) {
      const CUtensorMap* map = &maps.w_1;
      int ya = (rank * n_h + 2 * (g - 1)) * 64, yb = ya + 64;
      if (g == 0) { map = &maps.w_oc; ya = rank * 64; }
      if (is_hidden(g)) { map = &maps.w_2; ya = owner_of(g - 1 - n_pass) * 64; yb = ya + 128; }
      if (g >= n_post) {
        map = g < n_post + 2 ? &maps.w_qkv : g == n_post + 2 ? &maps.w_o : &maps.w_qc;
        ya = rank * 64 + (g == n_post + 1 ? 2 * p.D : 0);
        yb = p.D + rank * 64;
      }
      const bool wide = is_wide(g), hid = is_hidden(g);
      const int n = stages_of(g);
      auto x_of = [&](int k) { return (hid ? (k < n_h ? rank : rank ^ 1) * n_h + (k < n_h ? k : k - n_h) : kb_of(k)) * 64; };
#pragma unroll 1
      for (int j = 0; j < n; ++j) {
        if (it == kLcStages && !waited) { activations(); waited = true; }   // the ring is full of weights: now the kernel in front
        if (it >= kLcStages) tc::mbar_wait(w_empty + slot, lap ^ 1, abort_flag);
        __syncwarp();
        const int xa = x_of(wide ? j : 2 * j), xb = wide ? xa : x_of(2 * j + 1);
        if (tc::elect_one()) {
          uint8_t* dst = ring + slot * 2 * kLcTile;
          tc::mbar_expect_tx(w_full + slot, 2 * kLcTile);
          tc::tma_load_2d(dst, map, w_full + slot, xa, ya);
          tc::tma_load_2d(dst + kLcTile, map, w_full + slot, xb, wide ? yb : ya);
        }
        __syncwarp();
        ++it;
        if (++slot == kLcStages) { slot = 0; lap ^= 1; }
      }
    }
    if (!waited) activations();                            // (a chain shorter than the ring)
  } else if (warp == 9) {
    // ---- MMA issuer ----
    constexpr uint32_t kIdesc64 = tc::idesc_bf16(64, 64, 0), kIdesc128 = tc::idesc_bf16(64, 128, 0);
    constexpr uint16_t kAll = (uint16_t)((1u << C) - 1u);
    const uint64_t desc_a = tc::smem_desc_sw128(tc::smem_addr(tile_a), 16, 1024);
    const uint64_t desc_h = tc::smem_desc_sw128(tc::smem_addr(tile_h), 16, 1024);
    const uint64_t desc_w = tc::smem_desc_sw128(tc::smem_addr(ring), 16, 1024);
    constexpr uint64_t kTileStep = kLcTile >> 4;           // a descriptor's start address counts 16 bytes
    int slot = 0, lap = 0, fill = 0, ev = 0;
#pragma unroll 1
    for (int g = g_first; g < g_last; ++g) {
      const bool wide = is_wide(g), hid = is_hidden(g);
      const int n = stages_of(g);
      // a new operand tile from the other CTAs
      if (g == 1 || g == n_post || g >= n_post + 2) {
        if (lane < C && lane != rank)
          tc::mbar_expect_tx(a_full + lane, tile_bytes);
        if (g == 1 && lane < n_h) tc::mbar_expect_tx(h_full + ((rank ^ 1) & 1) * kLcMaxHidden + lane, tile_bytes);
        __syncwarp();
      }
      const uint32_t col = tmem + (g == 0 || g >= n_post + 2 ? kAccHigh
                                   : hid ? kAccHigh + (g - 1 - n_pass) * 128 : g >= n_post ? kAccLow + (g - n_post) * 128 : kAccLow + (g - 1) * 128);
      const uint32_t idesc = wide ? kIdesc128 : kIdesc64;
#pragma unroll 1
      for (int j = 0; j < n; ++j) {
        tc::mbar_wait(w_full + slot, lap, abort_flag);
        __syncwarp();
        uint64_t b = desc_w + (uint64_t)(slot * 2) * kTileStep;
#pragma unroll 1
        for (int i = 0; i < (wide ? 1 : 2); ++i, b += kTileStep) {
          const int k = wide ? j : 2 * j + i;
          uint64_t a;
          if (hid) {
            const int at = (k < n_h ? (rank & 1) : ((rank ^ 1) & 1)) * kLcMaxHidden + (k < n_h ? k : k - n_h);
            tc::mbar_wait_cluster(h_full + at, 0, abort_flag);
            a = desc_h + (uint64_t)at * kTileStep;
          } else {
            const int kb = kb_of(k);
            tc::mbar_wait_cluster(a_full + kb, fill & 1, abort_flag);
            a = desc_a + (uint64_t)kb * kTileStep;
          }
          __syncwarp();
          tc::tc_fence_after();
          if (tc::elect_one()) {
            tc::mma_ss(col, a, b, idesc, k ? 1u : 0u);
#pragma unroll
            for (int m = 1; m < 4; ++m) tc::mma_ss_c<true>(col, a + (uint64_t)(2 * m), b + (uint64_t)(2 * m), idesc);
          }
          __syncwarp();
        }
        if (tc::elect_one()) tc::mma_commit(w_empty + slot);
        __syncwarp();
        if (++slot == kLcStages) { slot = 0; lap ^= 1; }
      }
      // the last product on this tile: the cluster may fill it again.  (Said only where every CTA waits for it before it leaves:
      // with two CTAs and no layer behind, nothing comes after the hidden columns.)
      const bool last = g == 0 || (g == n_pass && (C >= 4 || p.pre)) || g == n_post + 1 || g == n_post + 2;
      if (tc::elect_one()) {
        if (last) mma_commit_cluster(a_free, kAll);
        tc::mma_commit(acc_full + (ev & 1));
      }
      __syncwarp();
      ++ev;
      if (last) ++fill;
    }
  } else {
    // ---- epilogue warps 0 .. 7: rows 16 q .. 16 q + 15 (the first 16 lanes), columns 32 half .. 32 half + 31 of the CTA's 64 ----
    const int q = warp & 3, half = warp >> 2;
    const int row = q * 16 + (lane & 15);
    const bool warp_lives = q * 16 < rows8;                // warps without rows keep to the barriers
    const bool lives = lane < 16 && row < rows8, valid = lane < 16 && row < rows;
    const int64_t mm = row0 + min(row, rows - 1);          // clamped: what is read there is never stored
    const int col0 = rank * 64 + half * 32;                // of the residual stream
    const uint32_t t_lane = tmem + ((uint32_t)(q * 32) << 16);
    int ev = 0, use = 0, ln_count = 0;                     // accumulators; uses of the operand tile; LayerNorms

    // column vectors (weights: at rest, except in front of a step)
    if (p.embed) pdl_wait();
    if (!F32) {
      for (int i = threadIdx.x; i < 512; i += 256) {
        const float* cb = nullptr; const float* cs = nullptr; int n = 0;
        if (i < 192) { if (p.pre) { cb = p.cb_qkv; cs = p.cs_qkv; } n = (i / 64) * p.D + rank * 64 + (i & 63); }
        else if (i < 256) { if (p.pre) { cb = p.cb_qc; cs = p.cs_qc; } n = rank * 64 + (i & 63); }
        else if (i - 256 < n_h * 64) { if (p.post) { cb = p.cb_1; cs = p.cs_1; } n = rank * n_h * 64 + i - 256; }
        vec[i] = cb != nullptr ? __ldg(cb + n) : 0.f;
        vec[512 + i] = cs != nullptr ? __ldg(cs + n) : 0.f;
      }
    } else {
      for (int i = threadIdx.x; i < 384; i += 256) {
        const int which = i >> 6, n = rank * 64 + (i & 63);
        const float* src = which == 0 ? p.ln1_g : which == 1 ? p.ln1_b : which == 2 ? p.ln2_g : which == 3 ? p.ln2_b : which == 4 ? p.ln3_g : p.ln3_b;
        vec[i] = (which < 2 || (which < 4 ? p.pre : p.post)) ? __ldg(src + n) : 0.f;
      }
    }
    if (threadIdx.x == 0) {
      if (kSources > 0 && p.post) tc::mbar_expect_tx(part_full, (uint32_t)(kSources * rows8 * 64 * 4));
    }
    tc::named_bar_sync(1, 256);
    if (!p.embed) pdl_wait();

    // this thread's part of the residual stream
    float x[32];
    if (p.embed) {
      int tok = __ldg(p.token + mm);
      if (tok < 0 || tok >= p.embed_count) {
        if (valid && rank == 0 && half == 0) flag_status(p.d_status, GRACE_DEV_BAD_INDEX);
        tok = 0;
      }
      const uint4* e = reinterpret_cast<const uint4*>(p.embed_rows + (int64_t)tok * p.D + col0);
      const uint4* o = reinterpret_cast<const uint4*>(p.pos + col0);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint4 a = __ldg(e + i), b = __ldg(o + i);
        x[8 * i] = bf16_lo(a.x) + bf16_lo(b.x); x[8 * i + 1] = bf16_hi(a.x) + bf16_hi(b.x);
        x[8 * i + 2] = bf16_lo(a.y) + bf16_lo(b.y); x[8 * i + 3] = bf16_hi(a.y) + bf16_hi(b.y);
        x[8 * i + 4] = bf16_lo(a.z) + bf16_lo(b.z); x[8 * i + 5] = bf16_hi(a.z) + bf16_hi(b.z);
        x[8 * i + 6] = bf16_lo(a.w) + bf16_lo(b.w); x[8 * i + 7] = bf16_hi(a.w) + bf16_hi(b.w);
      }
    } else if (F32) {
      const float4* src = reinterpret_cast<const float4*>(p.x_f32 + mm * p.D + col0);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float4 v = src[i];
        x[4 * i] = v.x; x[4 * i + 1] = v.y; x[4 * i + 2] = v.z; x[4 * i + 3] = v.w;
      }
    } else {
      const uint4* src = reinterpret_cast<const uint4*>(p.x_bf16 + mm * p.D + col0);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint4 v = src[i];
        x[8 * i] = bf16_lo(v.x); x[8 * i + 1] = bf16_hi(v.x); x[8 * i + 2] = bf16_lo(v.y); x[8 * i + 3] = bf16_hi(v.y);
        x[8 * i + 4] = bf16_lo(v.z); x[8 * i + 5] = bf16_hi(v.z); x[8 * i + 6] = bf16_lo(v.w); x[8 * i + 7] = bf16_hi(v.w);
      }
    }
    // rows of the earlier steps that hold this row's prefix
    int64_t anc[3] = {0, 0, 0};
    if (p.pre && p.t > 0) {
      const int b = (int)(mm / p.M_t);
      int64_t at = mm;
      bool bad = false;
#pragma unroll
      for (int j = 3; j >= 1; --j) {
        if (j <= p.t) {
          int par = __ldg(p.parents + (int64_t)j * p.R_max + at);
          if (par < 0 || par >= p.beam[j - 1]) { bad = true; par = 0; }
          at = (int64_t)b * p.beam[j - 1] + par;
          anc[j - 1] = at;
        }
      }
      if (bad && valid && rank == 0 && half == 0) flag_status(p.d_status, GRACE_DEV_BAD_INDEX);
    }
    const int D3 = 3 * p.D;
    // keys and values of the prefix wait where the hidden columns were: [position][K, V][eight pieces of 16 bytes][row]
    auto prefix_at = [&](int j, int kv, int i) { return tile_h + (((j * 2 + kv) * 8 + half * 4 + i) * kLcRows + row) * 16; };

    auto accumulated = [&]() {
      tc::mbar_wait(acc_full + (ev & 1), (ev >> 1) & 1, abort_flag);
      ++ev;
      __syncwarp();
      tc::tc_fence_after();
    };
    // (mean, 1 / deviation) of the whole row from the cluster's 2 C parts of it
    // (Statistics have a barrier of their own: a CTA may fill its k-block of the operand tile again, with its self-attention's
    // output, while a warp here has yet to look at what the block held before.  The next statistics come after this CTA's own.)
    auto row_norm = [&]() -> float2 {
      tc::mbar_wait_cluster(stats_full, ln_count & 1, abort_flag);
      ++ln_count;
      __syncwarp();
      float mean = 0.f, var = 0.f;
      float2 part[2 * C];
#pragma unroll
      for (int i = 0; i < 2 * C; ++i) { part[i] = stats[i * kLcRows + row]; mean += part[i].x; }
      mean *= 1.f / (float)(2 * C);
#pragma unroll
      for (int i = 0; i < 2 * C; ++i) { const float d = part[i].x - mean; var += fmaf(32.f * d, d, part[i].y); }
      return make_float2(mean, rsqrtf(var / (float)(64 * C) + p.eps));
    };

    if (p.post) ++use;                                     // the tile that TMA fills
    // 0: x += attn Wo_cross   1: hidden = relu(LN(x) W1)   2: x += hidden W2 (or the embedded rows)
    // 3: q, k, v, self-attention   4: x += attn Wo   5: the cross-attention's queries
#pragma unroll 1
    for (int step = p.post ? 0 : 2; step < (p.pre ? 6 : 3); ++step) {
      uint32_t r[32], w[16];                               // a row's 32 columns: accumulator; bf16 pairs
      if (step & 1) {
        float2 ar = make_float2(1.f, 0.f);                 // folded: y = rstd acc + (-rstd mean) col_sum + col_bias
        uint32_t qw[16];
        auto fetch_prefix = [&]() {
          if (step != 3 || !lives) return;
#pragma unroll 1
          for (int j = 0; j < p.t; ++j) {
            const int64_t a = j == 0 ? anc[0] : j == 1 ? anc[1] : anc[2];
            const uint16_t* src = p.slabs + (int64_t)j * p.slab_stride + a * D3 + p.D + col0;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(tc::smem_addr(prefix_at(j, 0, i))), "l"(src + 8 * i) : "memory");
              asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(tc::smem_addr(prefix_at(j, 1, i))), "l"(src + p.D + 8 * i) : "memory");
            }
          }
        };
        // The prefix overwrites the CTA's hidden k-blocks, the source of the copies to the pair's other CTA.  That they have
        // arrived there is known from what the other CTA does behind its second product: its arrival after the partial sums
        // (C >= 4), or its statistics of step 2, which an fp32 stream has waited for and a bf16 one waits for here.
        constexpr bool kPrefixFirst = F32 || C >= 4;
        if (kPrefixFirst) fetch_prefix();
        if constexpr (!F32) {
          const float2 nm = row_norm();
          ar = make_float2(nm.y, -nm.y * nm.x);
        }
        if (!kPrefixFirst) fetch_prefix();
        const int chunks = step == 1 ? n_h : step == 3 ? 3 : 1;
#pragma unroll 1
        for (int c = 0; c < chunks; ++c) {
          const bool two = step == 1 && (c | 1) < n_h;     // 128 hidden columns: a k-block per half; or one k-block, 32 columns per half
          if (step == 1 ? !(c & 1) : c != 1) accumulated();
          const int at = two ? (c & ~1) * 64 + half * 64 + (c & 1) * 32 : c * 64 + half * 32;
          const float* v = vec + (step == 1 ? 256 : step == 3 ? 0 : 192) + at;
          if (warp_lives) {
            float y[32];
            tc::tmem_ld32(t_lane + (step == 5 ? kAccHigh : kAccLow) + at, r);
            tc::tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 32; i += 4) {
              if (F32) {
#pragma unroll
                for (int k = 0; k < 4; ++k) y[i + k] = __uint_as_float(r[i + k]);
              } else {
                const float4 cb = *reinterpret_cast<const float4*>(v + i), cs = *reinterpret_cast<const float4*>(v + 512 + i);
                y[i] = fmaf(ar.x, __uint_as_float(r[i]), fmaf(ar.y, cs.x, cb.x));
                y[i + 1] = fmaf(ar.x, __uint_as_float(r[i + 1]), fmaf(ar.y, cs.y, cb.y));
                y[i + 2] = fmaf(ar.x, __uint_as_float(r[i + 2]), fmaf(ar.y, cs.z, cb.z));
                y[i + 3] = fmaf(ar.x, __uint_as_float(r[i + 3]), fmaf(ar.y, cs.w, cb.w));
              }
            }
            if (step == 1) {
#pragma unroll
              for (int i = 0; i < 32; ++i) y[i] = fmaxf(y[i], 0.f);
            }
#pragma unroll
            for (int i = 0; i < 16; ++i) w[i] = pack_bf16x2(y[2 * i], y[2 * i + 1]);
            if (step == 1) {
              if (lives) {
                uint8_t* tile = tile_h + ((rank & 1) * kLcMaxHidden + (two ? (c & ~1) + half : c)) * kLcTile + row * 128;
                const int piece0 = two ? (c & 1) * 4 : half * 4;
#pragma unroll
                for (int j = 0; j < 4; ++j)
                  *reinterpret_cast<uint4*>(tile + (((piece0 + j) ^ (row & 7)) << 4)) = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
              }
            } else if (valid) {
              uint4* dst = reinterpret_cast<uint4*>(step == 3 ? p.slabs + (int64_t)p.t * p.slab_stride + mm * D3 + c * p.D + col0
                                                              : p.q_cross + mm * p.D + col0);
#pragma unroll
              for (int j = 0; j < 4; ++j) dst[j] = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
            }
            if (step == 3) {
              if (c == 0) {
#pragma unroll
                for (int i = 0; i < 16; ++i) qw[i] = w[i];
              } else if (c == 1) {                         // scores of the row's own position (3) and of its prefix, over 32 columns
                asm volatile("cp.async.wait_all;" ::: "memory");
#pragma unroll 1
                for (int n = 0; n <= p.t; ++n) {
                  const int j = n == 0 ? 3 : n - 1;
                  if (n != 0) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                      const uint4 k4 = *reinterpret_cast<const uint4*>(prefix_at(j, 0, i));
                      w[4 * i] = k4.x; w[4 * i + 1] = k4.y; w[4 * i + 2] = k4.z; w[4 * i + 3] = k4.w;
                    }
                  }
                  float s0 = 0.f, s1 = 0.f;
#pragma unroll
                  for (int i = 0; i < 16; ++i) {
                    s0 = fmaf(bf16_lo(qw[i]), bf16_lo(w[i]), s0);
                    s1 = fmaf(bf16_hi(qw[i]), bf16_hi(w[i]), s1);
                  }
                  if (lives) scores[(half * kLcRows + row) * 4 + j] = s0 + s1;
                }
              } else {
                // softmax over the prefix and the row's own position, weighted sum of the values
                float s[4];
                const float* sa = scores + (half * kLcRows + row) * 4;
#pragma unroll
                for (int j = 0; j < 4; ++j) s[j] = j < p.t || j == 3 ? sa[j] : 0.f;
                if (p.d_h == 64) {                         // a head's other 32 columns are another warp's
                  const float* sb = scores + ((half ^ 1) * kLcRows + row) * 4;
#pragma unroll
                  for (int j = 0; j < 4; ++j) if (j < p.t || j == 3) s[j] += sb[j];
                }
                float mx = s[3] * p.scale;
#pragma unroll
                for (int j = 0; j < 3; ++j) { s[j] = j < p.t ? s[j] * p.scale : -INFINITY; mx = fmaxf(mx, s[j]); }
                s[3] *= p.scale;
                float den = 0.f;
#pragma unroll
                for (int j = 0; j < 4; ++j) { s[j] = __expf(s[j] - mx); den += s[j]; }
                const float inv = 1.f / den;
#pragma unroll
                for (int i = 0; i < 32; ++i) y[i] = 0.f;
#pragma unroll 1
                for (int j = 0; j <= p.t; ++j) {
                  const float f = (j == p.t ? s[3] : j == 0 ? s[0] : j == 1 ? s[1] : s[2]) * inv;
                  if (j != p.t) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                      const uint4 v4 = *reinterpret_cast<const uint4*>(prefix_at(j, 1, i));
                      r[4 * i] = v4.x; r[4 * i + 1] = v4.y; r[4 * i + 2] = v4.z; r[4 * i + 3] = v4.w;
                    }
                  } else {
#pragma unroll
                    for (int i = 0; i < 16; ++i) r[i] = w[i];
                  }
#pragma unroll
                  for (int i = 0; i < 16; ++i) { y[2 * i] = fmaf(f, bf16_lo(r[i]), y[2 * i]); y[2 * i + 1] = fmaf(f, bf16_hi(r[i]), y[2 * i + 1]); }
                }
#pragma unroll
                for (int i = 0; i < 16; ++i) w[i] = pack_bf16x2(y[2 * i], y[2 * i + 1]);
              }
            }
          }
          tc::tc_fence_before();
          if (step == 3 && c == 1 && p.d_h == 64) tc::named_bar_sync(1, 256);          // the scores of both halves
          if (step == 1 && ((c & 1) || !two)) {            // the k-blocks of this accumulator: to the issuer and to the pair's other CTA
            tc::fence_proxy_async_smem();
            tc::named_bar_sync(1, 256);
            if (warp < (two ? 2 : 1) && tc::elect_one()) {
              const int kb = (rank & 1) * kLcMaxHidden + (two ? (c & ~1) + warp : c);
              tc::mbar_arrive(h_full + kb);
              dsmem_bulk_copy(tc::cluster_addr_of(tile_h + kb * kLcTile, (uint32_t)(rank ^ 1)), tile_h + kb * kLcTile, tile_bytes,
                              tc::cluster_addr_of(h_full + kb, (uint32_t)(rank ^ 1)));
            }
            __syncwarp();
          }
        }
        if (step != 3) continue;
      } else {
        bool add = true;
        if (step == 2 && !p.post) {
          add = false;                                     // the embedded rows
        } else if (step == 2 && C >= 4) {
          // partial sums to the owners of the columns, this CTA's own ones from them
          tc::mbar_wait_cluster(a_free, (use - 1) & 1, abort_flag);      // no CTA reads its operand tile any more: partial sums go there
          ++use;
          float own[32];
#pragma unroll 1
          for (int i = 0; i < C / 2; ++i) {
            const int o = owner_of(i >> 1) + 2 * (i & 1);
            if (!(i & 1)) accumulated();
            if (!warp_lives) continue;
            tc::tmem_ld32(t_lane + kAccHigh + i * 64 + half * 32, r);
            tc::tmem_ld_wait();
            if (o == rank) {
#pragma unroll
              for (int k = 0; k < 32; ++k) own[k] = __uint_as_float(r[k]);
            } else if (lives) {
              const int slot = (rank >> 1) < (o >> 1) ? (rank >> 1) : (rank >> 1) - 1;
              const uint32_t dst = tc::cluster_addr_of(tile_a + slot * (kLcRows * 64 * 4) + (half * 8 * kLcRows + row) * 16, (uint32_t)o);
              const uint32_t bar = tc::cluster_addr_of(part_full, (uint32_t)o);
#pragma unroll
              for (int k = 0; k < 8; ++k) dsmem_st_async(dst + k * kLcRows * 16, bar, r + 4 * k);
            }
            __syncwarp();
          }
          tc::tc_fence_before();
          tc::mbar_wait_cluster(part_full, 0, abort_flag);
          __syncwarp();
          // in the order of the sources, the CTA itself among them
#pragma unroll
          for (int i = 0; i < 32; ++i) r[i] = 0u;
#pragma unroll 1
          for (int sc = 0; sc < C / 2; ++sc) {
            const float4* src = reinterpret_cast<const float4*>(tile_a + (sc < (rank >> 1) ? sc : sc - 1) * (kLcRows * 64 * 4)) + half * 8 * kLcRows + row;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
              float4 v = make_float4(own[4 * k], own[4 * k + 1], own[4 * k + 2], own[4 * k + 3]);
              if (sc != (rank >> 1)) v = src[k * kLcRows];
              r[4 * k] = __float_as_uint(__uint_as_float(r[4 * k]) + v.x); r[4 * k + 1] = __float_as_uint(__uint_as_float(r[4 * k + 1]) + v.y);
              r[4 * k + 2] = __float_as_uint(__uint_as_float(r[4 * k + 2]) + v.z); r[4 * k + 3] = __float_as_uint(__uint_as_float(r[4 * k + 3]) + v.w);
            }
          }
          tc::named_bar_sync(1, 256);                      // all of them read: the cluster may fill this CTA's tile again
          if (warp < C && tc::elect_one()) {
            if (warp == rank) tc::mbar_arrive(a_free);
            else tc::mbar_arrive_remote(a_free, (uint32_t)warp);
          }
          __syncwarp();
        } else {
          accumulated();
          tc::tmem_ld32(t_lane + kAccHigh + half * 32, r);
          tc::tmem_ld_wait();
          tc::tc_fence_before();
        }
        if (add) {
#pragma unroll
          for (int i = 0; i < 32; ++i) x[i] += __uint_as_float(r[i]);
        }
        if (!F32) {                                        // the stream's values are bf16
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            w[i] = pack_bf16x2(x[2 * i], x[2 * i + 1]);
            x[2 * i] = bf16_lo(w[i]);
            x[2 * i + 1] = bf16_hi(w[i]);
          }
        }
      }
      // The CTA's 64 columns become k-block `rank` of every CTA's operand tile: x for a LayerNorm (the raw bf16 rows with
      // their statistics, or, F32, the normalised rows), or the self-attention's output.
      // a warp per destination: copies that eight lanes of one warp send are issued one after the other
      auto send_stats = [&]() {
        const float2* mine = stats + rank * 2 * kLcRows;
        if (warp == rank) tc::mbar_expect_tx(stats_full, (C - 1) * 2 * kLcRows * 8);
        else dsmem_bulk_copy(tc::cluster_addr_of(mine, (uint32_t)warp), mine, 2 * kLcRows * 8, tc::cluster_addr_of(stats_full, (uint32_t)warp));
      };
      // (F32 behind the last layer: the final LayerNorm's rows go to memory, for the output head.)
      const bool next = step != 2 || p.pre;
      auto tile_free = [&]() {                             // every CTA is done with its operand tile
        if (use > 0) tc::mbar_wait_cluster(a_free, (use - 1) & 1, abort_flag);
        ++use;
      };
      float2 mine32 = make_float2(0.f, 0.f);
      if ((next || F32) && step != 3 && warp_lives) {      // mean and sum of squared deviations of the thread's 32 columns
        float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
#pragma unroll
        for (int i = 0; i < 32; i += 4) { s0 += x[i]; s1 += x[i + 1]; s2 += x[i + 2]; s3 += x[i + 3]; }
        const float mean = ((s0 + s1) + (s2 + s3)) * (1.f / 32.f);
        s0 = s1 = s2 = s3 = 0.f;
#pragma unroll
        for (int i = 0; i < 32; i += 4) {
          const float a = x[i] - mean, b = x[i + 1] - mean, c = x[i + 2] - mean, d = x[i + 3] - mean;
          s0 = fmaf(a, a, s0); s1 = fmaf(b, b, s1); s2 = fmaf(c, c, s2); s3 = fmaf(d, d, s3);
        }
        mine32 = make_float2(mean, (s0 + s1) + (s2 + s3));
        if (F32 && lives) stats[(rank * 2 + half) * kLcRows + row] = mine32;
      }
      // The statistics before these were the source of copies.  That they have arrived: an fp32 stream's last tiles came
      // behind every CTA's wait for them; for a bf16 stream, whose tiles travel beside them, a free tile says it (step 2: all
      // CTAs have added their partial sums or, with two, the other one's hidden columns have come; step 4: all are through
      // the self-attention).
      if constexpr (!F32) {
        if (next) {
          tile_free();
          if (step != 3 && lives) stats[(rank * 2 + half) * kLcRows + row] = mine32;
        }
      } else if (step != 3) {
        tc::fence_proxy_async_smem();
        tc::named_bar_sync(1, 256);
        if (warp < C && tc::elect_one()) send_stats();
        __syncwarp();
        const float2 nm = row_norm();
        const float* g = vec + (step == 0 ? 256 : step == 2 ? 0 : 128) + half * 32;
#pragma unroll
        for (int i = 0; i < 32; i += 2)
          w[i >> 1] = pack_bf16x2((x[i] - nm.x) * nm.y * g[i] + g[64 + i], (x[i + 1] - nm.x) * nm.y * g[i + 1] + g[65 + i]);
      }
      if (next) {
        if (F32) tile_free();
        if (lives) {
          uint8_t* tile = tile_a + rank * kLcTile + row * 128;
#pragma unroll
          for (int j = 0; j < 4; ++j)
            *reinterpret_cast<uint4*>(tile + (((half * 4 + j) ^ (row & 7)) << 4)) = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
        }
        tc::fence_proxy_async_smem();
        tc::named_bar_sync(1, 256);
        if (warp < C && tc::elect_one()) {
          uint8_t* mine = tile_a + rank * kLcTile;
          if (warp == rank) tc::mbar_arrive(a_full + rank);
          else dsmem_bulk_copy(tc::cluster_addr_of(mine, (uint32_t)warp), mine, tile_bytes, tc::cluster_addr_of(a_full + rank, (uint32_t)warp));
          if (!F32 && step != 3) send_stats();
        }
        __syncwarp();
      } else if (F32 && valid) {
        uint4* dst = reinterpret_cast<uint4*>(p.h_final + mm * p.D + col0);
#pragma unroll
        for (int j = 0; j < 4; ++j) dst[j] = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
      }
      if (step == 4 || (step == 2 && !p.pre)) {            // the stream as the next kernel finds it
        if (valid) {
          if (F32) {
            float4* dst = reinterpret_cast<float4*>(p.x_f32 + mm * p.D + col0);
#pragma unroll
            for (int i = 0; i < 8; ++i) dst[i] = make_float4(x[4 * i], x[4 * i + 1], x[4 * i + 2], x[4 * i + 3]);
          } else {
            uint4* dst = reinterpret_cast<uint4*>(p.x_bf16 + mm * p.D + col0);
#pragma unroll
            for (int j = 0; j < 4; ++j) dst[j] = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
          }
        }
      }
    }
  }
  // no CTA may leave while copies into it or arrivals on its barriers can be under way
  if (*abort_flag) __nanosleep(100000);
  tc::tc_fence_before();
  __syncthreads();
  tc::cluster_sync_all();
  if (warp == 8) tc::tmem_dealloc(tmem, 512);
}

int layer_chain_timeouts() { return tc::tc_timeouts_read_and_clear(); }

// Clusters of two, four and eight CTAs, one to an SM, that a B200 holds at once.
static int layer_chain_clusters(int C) { return C == 2 ? kSmsInTwos / 2 : C == 4 ? kSmsInFours / 4 : kSmsInEights / 8; }

// Whether grace_decode_step runs the layers of step t through the kernel above: where its clusters take all rows at once (a
// second wave costs as much again).  A step replayed from a graph, 3 tokens, selection included, launches / so (us).  2 x 128: 16
// rows 56 / 48, 256 rows 76 / 65, 4096 rows 139 / 119, 4736 rows 138 / 114 (8192 rows, two waves, 184 / 207); fp32 stream 64 / 50,
// 84 / 66, 147 / 118, 146 / 114.  2 x 256: 1 row 59 / 55, 16 rows 65 / 65, 256 rows 92 / 82, 2112 rows 112 / 98; fp32 67 / 57, 74 / 68,
// 98 / 84, 123 / 99.  4 x 512: 1 row 116 / 116, 16 rows 127 / 132, 32 rows 130 / 133, 64 rows 136 / 137, 128 rows 155 / 145, 512 rows
// 193 / 175, 960 rows 221 / 200; fp32 137 / 122, 151 / 137, 151 / 138, 157 / 143, 174 / 151, 213 / 183, 245 / 207.
// So up to 64 rows of a bf16 stream with 4 d_model hidden columns can take the GPU longer, by what the prefix costs inside the
// kernel: 4 x 512, steps 1 and 3, 1 row 113 / 116 and 113 / 120, 8 rows 117 / 117 and 119 / 121, 64 rows 135 / 136 and 137 / 140; 2 x 256, 16
// rows 63.5 / 65 and 64 / 67; a search's first step loses nothing (1 request 115 / 115, 32 requests 121 / 121).  They are taken all
// the same, for what the host has to launch (2 kernels a layer instead of 8).  A search of one request, projection included, 4 x 512
// bf16, beam 1, 4, 16, 64, 512: as calls 587 -> 555 us, 596 -> 557, 627 -> 594, 689 -> 649, 859 -> 818, each waited for 641 -> 606,
// 650 -> 610, 680 -> 649, 742 -> 702, 914 -> 874, and from a graph 529 -> 533, 543 -> 539, 570 -> 569, 628 -> 623, 801 -> 791; 2 x 256, beam 16:
// 305 -> 288, 349 -> 331, 275 -> 272.
bool layer_chain_takes(const grace_decoder_t* d, int t) {
  const int D = d->d_model;
  if ((D != 128 && D != 256 && D != 512) || d->H * d->d_h != D || (d->d_h != 32 && d->d_h != 64)) return false;
  const int C = D / 64;
  if (d->d_ffn <= 0 || d->d_ffn % (64 * C) != 0 || d->d_ffn / (64 * C) > kLcMaxHidden) return false;
  if (d->x == nullptr && d->row_affine == nullptr) return false;       // bf16 stream with LayerNorm kernels of its own
  auto aligned = [](std::initializer_list<const void*> ps) {
    for (const void* q : ps)
      if (!grace_aligned16(q)) return false;
    return true;
  };
  // (what the launches refuse for its alignment is left to them)
  if (!aligned({d->x, d->x_bf16, d->attn, d->qkv, d->h, d->embed, d->pos, d->lnf_g, d->lnf_b})) return false;
  for (int l = 0; l < d->n_layers; ++l) {
    const grace_layer_t& w = d->layers[l];
    if (w.qkv_slabs == nullptr || !aligned({w.qkv_slabs, w.w_qkv, w.w_o, w.w_qc, w.w_oc, w.w_1, w.w_2, w.ln1_g, w.ln1_b, w.ln2_g,
                                             w.ln2_b, w.ln3_g, w.ln3_b}))
      return false;
    if (d->x == nullptr && !aligned({w.cb_qkv, w.cs_qkv, w.cb_qc, w.cs_qc, w.cb_1, w.cs_1})) return false;
  }
  const int64_t R = (int64_t)d->B * d->beam_sizes[t];
  return t <= 3 && R <= (int64_t)layer_chain_clusters(C) * kLcRows;
}

template <int C, bool F32>
static grace_status_t launch_chain(const LayerChainMaps& maps, const LayerChainParams& p, cudaStream_t s) {
  using S = LayerChainSmem<C>;
  static unsigned long long attr_set_devices = 0;
  DeviceSetup su(&attr_set_devices);
  if (su) {
    GRACE_CUDA_TRY(cudaFuncSetAttribute(layer_chain_kernel<C, F32>, cudaFuncAttributeMaxDynamicSharedMemorySize, S::kTotal));
    su.done();
  }
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = C; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.gridDim = dim3((unsigned)((p.R + p.tile_rows - 1) / p.tile_rows * C));
  cfg.blockDim = dim3(kLcThreads); cfg.dynamicSmemBytes = S::kTotal; cfg.stream = s;
  cfg.attrs = attr; cfg.numAttrs = 2;
  cudaLaunchKernelEx(&cfg, layer_chain_kernel<C, F32>, maps, p);
  GRACE_LAUNCH_CHECK();
  return GRACE_OK;
}

// The part of layer `post` behind its cross-attention (post < 0: none; then the rows are embedded first) and the part of
// layer post + 1 in front of its own; behind the last layer, with an fp32 stream, the final LayerNorm into d->h.
grace_status_t layer_chain(const grace_decoder_t* d, int t, int post, void* stream) {
  const int D = d->d_model, C = D / 64, R = d->B * d->beam_sizes[t], pre = post + 1;
  LayerChainMaps maps;
  LayerChainParams p = {};
  auto weight = [](CUtensorMap* map, const uint16_t* w, int rows, int cols) {
    const uint64_t dims[2] = {(uint64_t)cols, (uint64_t)rows}, str[1] = {(uint64_t)cols};
    const uint32_t box[2] = {64u, 64u};
    return tc::make_tmap_bf16(map, w, 2, dims, str, box);
  };
  p.post = post >= 0; p.pre = pre < d->n_layers; p.embed = post < 0;
  // rows of a tile: as few as spread them over the clusters that fit at once
  const int fit = layer_chain_clusters(C), spread = ((R + fit - 1) / fit + 7) & ~7;
  p.tile_rows = spread < kLcRows ? spread : kLcRows;
  p.R = R; p.D = D; p.hidden_blocks = d->d_ffn / (64 * C); p.t = t; p.M_t = d->beam_sizes[t]; p.d_h = d->d_h;
  for (int j = 0; j < 4; ++j) p.beam[j] = j <= t ? d->beam_sizes[j] : 1;
  p.R_max = d->R_max; p.slab_stride = d->R_max * 3 * (int64_t)D;
  p.eps = d->ln_eps; p.scale = 1.0f / sqrtf((float)d->d_h);
  p.token = d->token[t & 1]; p.embed_rows = d->embed; p.pos = d->pos + (int64_t)t * D; p.embed_count = d->V + 1;
  p.x_bf16 = d->x_bf16; p.x_f32 = d->x; p.q_cross = d->qkv; p.parents = d->parents; p.d_status = d->d_status;
  bool ok = true;
  if (p.post) {
    const grace_layer_t& w = d->layers[post];
    ok = ok && weight(&maps.attn, d->attn, R, D) && weight(&maps.w_oc, w.w_oc, D, D) && weight(&maps.w_1, w.w_1, d->d_ffn, D) &&
         weight(&maps.w_2, w.w_2, D, d->d_ffn);
    p.cb_1 = w.cb_1; p.cs_1 = w.cs_1; p.ln3_g = w.ln3_g; p.ln3_b = w.ln3_b;
  }
  if (p.pre) {
    const grace_layer_t& w = d->layers[pre];
    ok = ok && weight(&maps.w_qkv, w.w_qkv, 3 * D, D) && weight(&maps.w_o, w.w_o, D, D) && weight(&maps.w_qc, w.w_qc, D, D);
    p.cb_qkv = w.cb_qkv; p.cs_qkv = w.cs_qkv; p.cb_qc = w.cb_qc; p.cs_qc = w.cs_qc;
    p.ln1_g = w.ln1_g; p.ln1_b = w.ln1_b; p.ln2_g = w.ln2_g; p.ln2_b = w.ln2_b;
    p.slabs = w.qkv_slabs;
  } else {
    p.ln1_g = d->lnf_g; p.ln1_b = d->lnf_b; p.h_final = d->h;
  }
  if (!ok) return GRACE_CUDA_ERROR;
  cudaStream_t s = (cudaStream_t)stream;
  const bool f32 = d->x != nullptr;
  switch (C) {
    case 2: return f32 ? launch_chain<2, true>(maps, p, s) : launch_chain<2, false>(maps, p, s);
    case 4: return f32 ? launch_chain<4, true>(maps, p, s) : launch_chain<4, false>(maps, p, s);
    case 8: return f32 ? launch_chain<8, true>(maps, p, s) : launch_chain<8, false>(maps, p, s);
  }
  return GRACE_UNSUPPORTED_SHAPE;
}

}  // namespace grace
