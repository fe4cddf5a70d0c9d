// Cross-attention on tcgen05 tensor cores (Section 5.1: beams of a request are the M dimension of
// a dense contraction against that request's shared K/V): head size 128, and head size 64 with at most one
// 128-row tile per SM or with lengths and few rows per request (otherwise the four-stream kernel of cross_attn_ms.cuh).
//
// A work item is 128 query rows of one (request, head); its encoder positions are streamed in
// blocks of 128:
//   S   = Q K_blk^T        tcgen05.mma, A = Q (shared, K-major), B = K_blk (shared, K-major),
//                          fp32 S[128 x 128] in TMEM
//   P   = exp2(S*c - max)  softmax threads: TMEM lane = query row; two threads per row, half of the block's
//                          columns each (256 threads); P goes to its own TMEM columns as packed bf16
//   O  += P V_blk          tcgen05.mma, A = P (TMEM), B = V_blk (shared, read MN-major, so V is
//                          used as stored: no transpose anywhere); O stays in TMEM for the whole
//                          row tile and is rescaled lazily, only when a row maximum grows by > 2^8
// K and V blocks arrive by TMA through two separate two-slot rings; Q, K and V are addressed with 4-D tensor
// maps over the caller's strides, so the beam-major Q / O layout is never permuted (the view /
// permute / reshape chain of Section 5.1 costs nothing).  Ragged M and T are zero-filled by TMA
// and masked in the softmax; K and V past a request's length have no influence whatever they hold.  Warp roles: softmax + epilogue warps first, then the TMA producer warp, then
// the MMA issuer warp.
// The kernel is persistent (each CTA loops over work items; Q is double-buffered), one CTA per SM with all
// 512 TMEM columns: S (128), O twice (by item parity) and P twice (by block parity).  The softmax threads
// therefore never wait for P V: they hand P of a block over and go on to the next block (whose S the tensor
// core produced under their exponentials), and an item's output is read from TMEM and stored one block later.
// A 128-wide tile is held as two 64-wide halves (the 128-byte swizzle spans 64 bf16), each with its own TMA
// box and its own MMA k-steps (Q, K) or half of the output columns (V: one MMA spans both).
#pragma once
#include "common.cuh"
#include "tc.cuh"

namespace grace {

constexpr int kCaBM = 128;        // query rows per work item
constexpr int kCaBN = 128;        // encoder positions per block
constexpr int kCaStages = 2;
constexpr int kCaHalfBytes = 128 * 64 * 2;                       // 16 KB: 128 rows x 64 bf16, one swizzle span wide
constexpr int kCaSoftmaxWarps = 8;   // two threads per query row: each half of a block's score columns and of the output columns
constexpr int kCaThreads = (kCaSoftmaxWarps + 2) * 32;
constexpr int kCaBarBytes = 256;
// SPLIT > 1: a cluster of SPLIT CTAs shares one work item, each taking a contiguous range of its K / V blocks; the
// partial results (unnormalised output, maximum and sum per row) are merged through distributed shared memory:
// every CTA owns DH / SPLIT of the output columns and receives the others' partial sums of them.
template <int DH, int SPLIT> struct CaCfg {
  static constexpr int kHalves = DH / 64;
  static constexpr int kTileBytes = kCaHalfBytes * kHalves;      // Q, K_blk or V_blk
  static constexpr int kQBufs = SPLIT > 1 ? 1 : 2;
  static constexpr int kSlice = DH / SPLIT;                      // output columns a CTA finishes
  static constexpr int kXBytes = SPLIT > 1 ? (SPLIT - 1) * 128 * kSlice * 4 + SPLIT * 128 * 8 : 0;
  static constexpr int kUsedBytes = kTileBytes * (kQBufs + 2 * kCaStages) + 1024 + kCaBarBytes + 2 * 2 * 128 * 4 + 2 * 2 * 128 * 4 + kXBytes;
  // (at head size 64 less than the SM has twice, and a CTA takes all of TMEM)
  static constexpr int kSmemBytes = kUsedBytes > tc::kTmemAllSmem ? kUsedBytes : tc::kTmemAllSmem;
  static_assert(kSmemBytes <= 227 * 1024, "");
  static constexpr uint32_t kTmemCols = 512;                     // S: 0..127, O: 2 x DH (by item parity), P: 2 x 64 (by block parity)
};

struct CrossTcParams {
  uint16_t* out;
  float* lse;
  const int32_t* enc_len;       // LENGTHS: valid encoder positions per request (<= T)
  int64_t out_row_stride;
  int B, M, H, T;
  int tiles_m, total_items;
  float scale_log2;             // scale * log2(e)
};

// One work item: request, head, 128-row tile, encoder positions and the K / V blocks they take.  Every role of a
// CTA walks the same sequence of items; those without any encoder position (nb == 0) are passed over by the loads
// and the MMAs and written as zeros by the epilogue warps.
// With SPLIT > 1 an item is a CTA's share of one: nb blocks from position t0 on (T counts from there).
struct CaItem { int b, h, tile, t0, T, nb; };
template <int SPLIT, bool LENGTHS>
__device__ __forceinline__ CaItem ca_item(const CrossTcParams& p, int item) {
  CaItem it;
  const int part = item % SPLIT;
  item /= SPLIT;
  const int bh = item / p.tiles_m;
  it.tile = item - bh * p.tiles_m;
  it.b = bh / p.H;
  it.h = bh - it.b * p.H;
  it.T = p.T;
  if (LENGTHS) { const int e = __ldg(p.enc_len + it.b); it.T = e < 0 ? 0 : (e < p.T ? e : p.T); }
  it.nb = (it.T + kCaBN - 1) / kCaBN;
  it.t0 = 0;
  if (SPLIT > 1) {
    const int first = it.nb * part / SPLIT;
    it.nb = it.nb * (part + 1) / SPLIT - first;
    it.t0 = first * kCaBN;
    it.T -= it.t0;
  }
  return it;
}
// A position in that sequence: item, its place among the CTA's non-empty items (li), block inside the item.
template <int SPLIT, bool LENGTHS>
struct CaCursor {
  int item, li, j;
  CaItem it;
  __device__ __forceinline__ bool live(const CrossTcParams& p) const { return item < p.total_items; }
  __device__ __forceinline__ void seek(const CrossTcParams& p) {       // to the first non-empty item from here on
    for (; item < p.total_items; item += (int)gridDim.x) {
      it = ca_item<SPLIT, LENGTHS>(p, item);
      if (it.nb > 0) return;
    }
  }
  __device__ __forceinline__ void start(const CrossTcParams& p) { item = (int)blockIdx.x; li = 0; j = 0; seek(p); }
  __device__ __forceinline__ void next(const CrossTcParams& p) {       // one block on
    if (++j == it.nb) { j = 0; ++li; item += (int)gridDim.x; seek(p); }
  }
};

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ float max3(float a, float b, float c) {
  float m;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(m) : "f"(a), "f"(b), "f"(c));
  return m;
}

// Persistent kernel: a flat grid of one CTA per SM; CTA g takes the work items g, g + gridDim.x,
// ...  An item is one (request, head, 128-row tile); consecutive items are the tiles of the same
// (request, head), so the CTAs running at the same time read the same K/V from L2.
// P32: the probabilities keep (at least) sixteen bits of their fp32 mantissa: P is stored as the sum of two bf16 values
// and multiplied with V twice.  The two take the P columns of both block parities, so P of a block is stored
// once P V of the block before it is complete.  Calls with per-request lengths run this form: they were computed with
// fp32 probabilities before the tensor cores took them over, and one bf16 rounding of P shows in the result
// (relative error against 64 bits 2.2e-3 instead of the output rounding's 1.66e-3).  What is left of the difference to
// fp32, 16 x 100 x 16 x 128 x 200: 1.660216e-3 against 1.660215e-3, log-sum-exp 4.8e-8 against 3.6e-8.  The second value of a
// probability may be zero or negative: an infinite value of V inside the length gives NaN, not the infinity.
// LENGTHS: per-request lengths are given (without them no code for them: it costs a split call 2 to 3 %).
template <int DH, int SPLIT, bool P32, bool LENGTHS>
__global__ void __launch_bounds__(kCaThreads, 1)
cross_attn_tc_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                     const __grid_constant__ CUtensorMap map_v, const CrossTcParams p) {
  constexpr int kCols = kCaBN / 2;                         // score columns per softmax thread and block
  constexpr int kCaTileBytes = CaCfg<DH, SPLIT>::kTileBytes, kHalves = CaCfg<DH, SPLIT>::kHalves;
  constexpr uint32_t kCaTmemCols = CaCfg<DH, SPLIT>::kTmemCols;
  constexpr int kQBufs = CaCfg<DH, SPLIT>::kQBufs, kSlice = CaCfg<DH, SPLIT>::kSlice;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t* q_tiles = tiles;                                      // two Q buffers (one if an item is all a CTA does)
  uint8_t* kv_tiles = tiles + kQBufs * kCaTileBytes;             // stage s: K at 2s, V at 2s+1
  uint64_t* bars = reinterpret_cast<uint64_t*>(tiles + kCaTileBytes * (kQBufs + 2 * kCaStages));
  uint64_t* q_full = bars;                    // [2]
  uint64_t* q_empty = bars + 2;               // [2]
  uint64_t* k_full = bars + 4;                // [stages]  K and V have separate rings: a K slot is
  uint64_t* k_empty = k_full + kCaStages;     // [stages]  free once S of its block has run, a V
  uint64_t* v_full = k_empty + kCaStages;     // [stages]  slot only after P V of its block
  uint64_t* v_empty = v_full + kCaStages;     // [stages]
  uint64_t* s_full = v_empty + kCaStages;
  // [2] by block parity.  The softmax threads hand P of block g + 1 over without waiting for anything the issuer does
  // after its wait for P of block g, so with a single barrier an issuer that comes late to that wait could find the
  // phase after it complete as well and wait for good; with two, P of block g + 2 comes after P V of block g.
  uint64_t* p_full = s_full + 1;
  uint64_t* o_full = p_full + 2;              // [2] by block parity: P V of the block is complete
  uint64_t* s_free = o_full + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(s_free + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  float* half_max = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(bars) + kCaBarBytes);   // [2][2][128]
  float* half_sum = half_max + 2 * 2 * 128;                                                     // [2][128]

  float4* xbuf = reinterpret_cast<float4*>(half_sum + 2 * 2 * 128);                             // SPLIT: [SPLIT - 1][kSlice / 4][128]
  float2* mlbuf = reinterpret_cast<float2*>(xbuf + (SPLIT - 1) * (kSlice / 4) * 128);           // SPLIT: [SPLIT][128] (maximum, sum)

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (SPLIT > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");   // "this CTA has started"
  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) { tc::mbar_init(q_full + i, 1); tc::mbar_init(q_empty + i, 1); }
    for (int s = 0; s < kCaStages; ++s) {
      tc::mbar_init(k_full + s, 1); tc::mbar_init(k_empty + s, 1);
      tc::mbar_init(v_full + s, 1); tc::mbar_init(v_empty + s, 1);
    }
    tc::mbar_init(s_full, 1);
    tc::mbar_init(p_full, kCaSoftmaxWarps);    // one arrival per softmax warp
    tc::mbar_init(p_full + 1, kCaSoftmaxWarps);
    tc::mbar_init(o_full, 1);
    tc::mbar_init(o_full + 1, 1);
    tc::mbar_init(s_free, kCaSoftmaxWarps);
    *abort_flag = 0;
    tc::fence_mbar_init();
  }
  if (warp == kCaSoftmaxWarps) tc::tmem_alloc(tmem_slot, kCaTmemCols);
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  pdl_wait();                                  // barrier set-up and TMEM allocation overlapped the previous kernel's tail
  pdl_trigger();                               // not before the wait: layer_chain_kernel reads weights before its own
  const uint32_t tmem_s = tmem_base;           // S fp32, 128 columns
  // O of an item lives in one of two accumulators (item parity) and P of a block in one of two column sets (block
  // parity), so the softmax threads hand P(g) over and go straight on to block g + 1 (whose S is already there)
  // while the tensor core runs P V of block g; an item's output is read and stored one block later, when its last
  // P V has long finished.  With one K/V block per item (128 encoder positions) that takes the wait for P V and
  // most of the output path out of the per-item chain.
  static_assert(128 + 2 * DH + 2 * 64 <= 512, "TMEM columns");
  const uint32_t tmem_o = tmem_base + 128;             // O fp32, 2 x DH columns
  const uint32_t tmem_p = tmem_base + 128 + 2 * DH;    // P bf16 pairs, 2 x 64 columns

  if (warp == kCaSoftmaxWarps) {
    // ---------------- TMA producer ----------------
    if (tc::elect_one()) {
      tc::tma_prefetch_desc(&map_q); tc::tma_prefetch_desc(&map_k); tc::tma_prefetch_desc(&map_v);
      // One thread feeds three queues (Q per item, K and V per block).  K of block g+2 can be
      // requested as soon as S of block g has run, long before the V slot of block g frees, so the
      // thread polls: whichever slot is free next gets its load, neither queue blocks the other.
      int gk = 0, gv = 0;                                    // next K block, next V block (counted over the CTA's items)
      CaCursor<SPLIT, LENGTHS> ck, cv;
      ck.start(p);
      cv = ck;
      int idle = 0;
      while ((ck.live(p) || cv.live(p)) && !*abort_flag) {
        bool progressed = false;
        if (ck.live(p)) {
          const int s = gk % kCaStages;
          const bool need_q = (ck.j == 0);
          const int qb = ck.li & 1;
          if (tc::mbar_try_wait_now(k_empty + s, ((gk / kCaStages) & 1) ^ 1) &&
              (!need_q || tc::mbar_try_wait_now(q_empty + qb, ((ck.li >> 1) & 1) ^ 1))) {
            if (need_q) {
              tc::mbar_expect_tx(q_full + qb, kCaTileBytes);
#pragma unroll
              for (int hf = 0; hf < kHalves; ++hf)
                tc::tma_load_4d(q_tiles + qb * kCaTileBytes + hf * kCaHalfBytes, &map_q, q_full + qb, 64 * hf, ck.it.h,
                                ck.it.tile * kCaBM, ck.it.b);
            }
            tc::mbar_expect_tx(k_full + s, kCaTileBytes);
#pragma unroll
            for (int hf = 0; hf < kHalves; ++hf)
              tc::tma_load_4d(kv_tiles + (2 * s) * kCaTileBytes + hf * kCaHalfBytes, &map_k, k_full + s, 64 * hf, ck.it.t0 + ck.j * kCaBN, ck.it.h, ck.it.b);
            ++gk;
            ck.next(p);
            progressed = true;
          }
        }
        if (cv.live(p) && gv < gk) {
          const int s = gv % kCaStages;
          if (tc::mbar_try_wait_now(v_empty + s, ((gv / kCaStages) & 1) ^ 1)) {
            tc::mbar_expect_tx(v_full + s, kCaTileBytes);
#pragma unroll
            for (int hf = 0; hf < kHalves; ++hf)
              tc::tma_load_4d(kv_tiles + (2 * s + 1) * kCaTileBytes + hf * kCaHalfBytes, &map_v, v_full + s, 64 * hf, cv.it.t0 + cv.j * kCaBN, cv.it.h, cv.it.b);
            ++gv;
            cv.next(p);
            progressed = true;
          }
        }
        if (progressed) {
          idle = 0;
        } else {
          __nanosleep(512);                                 // polling costs issue slots the softmax warps of this scheduler need
          if (++idle > (1 << 24)) {                          // bounded: about a second of nothing to do
            if (*abort_flag == 0) atomicAdd(&tc::g_tc_timeouts, 1);
            *abort_flag = 1;
          }
        }
      }
    }
  } else if (warp == kCaSoftmaxWarps + 1) {
    // ---------------- MMA issuer ----------------
    // (An elected lane, not a branch on the lane number: the compiler then knows that one thread is left and takes operands
    // straight to the registers that tcgen05.mma and TMA read.  What the issuing warps save, the softmax warps of their
    // schedulers gain: 16 x 1000 x 16 x 128 x 50..200 62.5 -> 59.5 us, 4 x 700 x 16 x 128 x 256..1024 42.4 -> 35.7,
    // 40 x 6 x 16 x 128 x 100..600 42.6 -> 35.9, 1 x 300 x 16 x 128 x 1024 11.05 -> 10.45, 1 x 512 x 8 x 64 x 1024 7.1 -> 6.85.)
    if (tc::elect_one()) {
      constexpr uint32_t idesc_s = tc::idesc_bf16(kCaBM, kCaBN, 0);     // Q K^T : B K-major
      constexpr uint32_t idesc_o = tc::idesc_bf16(kCaBM, DH, 1);        // P V   : B MN-major, all output columns at once
      // Every operand descriptor is fixed by (Q buffer, ring slot, k-step): build them once.  The
      // issuing thread shares its scheduler with busy softmax warps, so each instruction it does not
      // execute per block shortens the hand-off to the tensor core.
      // k-step k of Q or K: 16 of the DH columns = 32 bytes inside the 64-wide half (k / 4)
      uint64_t q_desc[kQBufs][DH / 16], k_desc[kCaStages][DH / 16], v_desc[kCaStages][kCaBN / 16];
#pragma unroll
      for (int i = 0; i < kQBufs; ++i)
#pragma unroll
        for (int k = 0; k < DH / 16; ++k)
          q_desc[i][k] = tc::smem_desc_sw128(tc::smem_addr(q_tiles + i * kCaTileBytes) + (k / 4) * kCaHalfBytes + 32 * (k % 4), 16, 1024);
#pragma unroll
      for (int st = 0; st < kCaStages; ++st) {
#pragma unroll
        for (int k = 0; k < DH / 16; ++k)
          k_desc[st][k] = tc::smem_desc_sw128(tc::smem_addr(kv_tiles + (2 * st) * kCaTileBytes) + (k / 4) * kCaHalfBytes + 32 * (k % 4), 16, 1024);
        // (the second 64-wide half of V's columns lies kCaHalfBytes further)
#pragma unroll
        for (int k = 0; k < kCaBN / 16; ++k)
          v_desc[st][k] = tc::smem_desc_sw128(tc::smem_addr(kv_tiles + (2 * st + 1) * kCaTileBytes) + 2048 * k, kHalves > 1 ? kCaHalfBytes : 1024, 1024);
      }
      // S of global block g: Q buffer of its item, K of ring slot g % stages
      auto issue_s = [&](int g, const CaCursor<SPLIT, LENGTHS>& c) -> bool {
        const int qb = c.li & 1, s = g % kCaStages;
        if (c.j == 0 && !tc::mbar_wait(q_full + qb, (c.li >> 1) & 1, abort_flag)) return false;
        if (!tc::mbar_wait(k_full + s, (g / kCaStages) & 1, abort_flag)) return false;
        tc::tc_fence_after();
        if (kQBufs == 1 || qb == 0) {
          if (s == 0) {
#pragma unroll
            for (int k = 0; k < DH / 16; ++k) tc::mma_ss(tmem_s, q_desc[0][k], k_desc[0][k], idesc_s, k ? 1u : 0u);
          } else {
#pragma unroll
            for (int k = 0; k < DH / 16; ++k) tc::mma_ss(tmem_s, q_desc[0][k], k_desc[1][k], idesc_s, k ? 1u : 0u);
          }
        } else {
          if (s == 0) {
#pragma unroll
            for (int k = 0; k < DH / 16; ++k) tc::mma_ss(tmem_s, q_desc[kQBufs - 1][k], k_desc[0][k], idesc_s, k ? 1u : 0u);
          } else {
#pragma unroll
            for (int k = 0; k < DH / 16; ++k) tc::mma_ss(tmem_s, q_desc[kQBufs - 1][k], k_desc[1][k], idesc_s, k ? 1u : 0u);
          }
        }
        tc::mma_commit(s_full);
        tc::mma_commit(k_empty + s);                         // K of block g is consumed
        if (c.j == c.it.nb - 1) tc::mma_commit(q_empty + qb);       // last use of this item's Q tile
        return true;
      };
      static_assert(kCaStages == 2, "descriptor selection below is written for two ring slots");
      CaCursor<SPLIT, LENGTHS> cs;                                           // the block whose S is issued next; (j, li): the one whose P V is
      cs.start(p);
      bool ok = cs.live(p) && issue_s(0, cs);
      for (int g = 0; ok; ++g) {
        const int s = g & 1, j = cs.j, li = cs.li;
        const int left = cs.it.T - j * kCaBN;                // positions of the request from this block on
        cs.next(p);
        const bool more = cs.live(p);
        // s_free(g): every softmax thread holds its scores of block g in registers, so the S
        // columns can be overwritten: S of block g+1 (possibly the next item's first block) runs
        // on the tensor core while the exponentials of block g are computed.
        if (!tc::mbar_wait(s_free, g & 1, abort_flag)) break;
        if (more && !issue_s(g + 1, cs)) break;
        // p_full(g): P of block g is in its TMEM columns (and, on an item's first block, the
        // previous item's epilogue has read O).
        if (!tc::mbar_wait(p_full + (g & 1), (g >> 1) & 1, abort_flag)) break;
        if (!tc::mbar_wait(v_full + s, (g >> 1) & 1, abort_flag)) break;
        tc::tc_fence_after();
        const uint32_t o_acc = tmem_o + (uint32_t)((li & 1) * DH), p_cols = tmem_p + (uint32_t)(P32 ? 0 : (g & 1) * 64);
        if (left <= kCaBN - 16) {                            // (on its own: a test per k-step slows the full blocks)
          const uint64_t v0 = s == 0 ? v_desc[0][0] : v_desc[1][0];
#pragma unroll 1
          for (int k = 0; 16 * k < left; ++k) {
            tc::mma_ts(o_acc, p_cols + 8 * k, v0 + (uint64_t)(k * 2048 / 16), idesc_o, (j | k) ? 1u : 0u);
            if (P32) tc::mma_ts(o_acc, p_cols + 64 + 8 * k, v0 + (uint64_t)(k * 2048 / 16), idesc_o, 1u);
          }
        } else if (s == 0) {
#pragma unroll
          for (int k = 0; k < kCaBN / 16; ++k) {
            tc::mma_ts(o_acc, p_cols + 8 * k, v_desc[0][k], idesc_o, (j | k) ? 1u : 0u);
            if (P32) tc::mma_ts(o_acc, p_cols + 64 + 8 * k, v_desc[0][k], idesc_o, 1u);
          }
        } else {
#pragma unroll
          for (int k = 0; k < kCaBN / 16; ++k) {
            tc::mma_ts(o_acc, p_cols + 8 * k, v_desc[1][k], idesc_o, (j | k) ? 1u : 0u);
            if (P32) tc::mma_ts(o_acc, p_cols + 64 + 8 * k, v_desc[1][k], idesc_o, 1u);
          }
        }
        tc::mma_commit(v_empty + s);                         // V of block g is consumed
        tc::mma_commit(o_full + (g & 1));                    // O includes block g
        ok = more;
      }
    }
  } else {
    // ---------------- softmax + epilogue ----------------
    // Warps w and w+4 share the TMEM lanes (= query rows) 32*(w&3)..+31; each takes one half of the
    // 128 score columns and one half of the DH output columns of those rows.  O stays in TMEM and
    // accumulates across blocks; it is rescaled only when a row's maximum grows by more than 2^8
    // (probabilities may then reach 256, which bf16 and the fp32 sums hold without loss).
    const int quarter = warp & 3, half = warp >> 2;
    const int row = quarter * 32 + lane;
    const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
    const int col_base = kCols * half;
    constexpr int kOutCols = DH / 2;                       // output columns per thread
    bool ok = true;
    int g = 0, n_done = 0, li = 0;
    // the item whose output is still to be read from TMEM and stored (after the next block's P hand-over)
    int pend_g = -1, pend_li = 0;
    CaItem pend_it = {0, 0, 0, 0, 0, 0};
    float pend_m = 0.f, pend_l = 0.f;
    // wait for P V of global block gb (completion gb >> 1 of the barrier of its parity)
    auto wait_pv = [&](int gb) -> bool {
      bool w = tc::mbar_wait(o_full + (gb & 1), (gb >> 1) & 1, abort_flag);
      return __all_sync(kFullMask, w);
    };
    auto store_item = [&](const CaItem& it_e, int g_last, int li_e, float m_e, float l_e) -> bool {
      const int tile = it_e.tile, h = it_e.h, b = it_e.b;
      if (!wait_pv(g_last)) return false;
      tc::tc_fence_after();
      const uint32_t o_acc = tmem_o + (uint32_t)((li_e & 1) * DH);
      uint32_t o[kOutCols];
#pragma unroll
      for (int c = 0; c < kOutCols; c += 32)
        tc::tmem_ld32(o_acc + lane_addr + kOutCols * half + c, *reinterpret_cast<uint32_t(*)[32]>(&o[c]));
      tc::tmem_ld_wait();
      float* hs = half_sum + (n_done & 1) * 256;              // double-buffered by item parity
      hs[half * 128 + row] = l_e;
      tc::named_bar_sync(2 + quarter, 64);
      const float l_tot = l_e + hs[(half ^ 1) * 128 + row];
      ++n_done;
      const int m = tile * kCaBM + row;
      if (m < p.M) {
        const float inv = 1.f / l_tot;
        const int64_t r_out = (int64_t)b * p.M + m;
        uint4* dst = reinterpret_cast<uint4*>(p.out + r_out * p.out_row_stride + h * DH + kOutCols * half);
        auto piece = [&](int i) {
          return make_uint4(
              pack_bf16x2(__uint_as_float(o[8 * i]) * inv, __uint_as_float(o[8 * i + 1]) * inv),
              pack_bf16x2(__uint_as_float(o[8 * i + 2]) * inv, __uint_as_float(o[8 * i + 3]) * inv),
              pack_bf16x2(__uint_as_float(o[8 * i + 4]) * inv, __uint_as_float(o[8 * i + 5]) * inv),
              pack_bf16x2(__uint_as_float(o[8 * i + 6]) * inv, __uint_as_float(o[8 * i + 7]) * inv));
        };
        // a thread owns a row: its stores are pieces at a row stride, so whole 32-byte sectors where the
        // output's alignment allows (half the store transactions of 16-byte pieces)
        if ((reinterpret_cast<uintptr_t>(dst) & 31) == 0) {
#pragma unroll
          for (int i = 0; i < kOutCols / 8; i += 2) st_global_32B(dst + i, piece(i), piece(i + 1));
        } else {
#pragma unroll
          for (int i = 0; i < kOutCols / 8; ++i) dst[i] = piece(i);
        }
        if (p.lse != nullptr && half == 0) p.lse[r_out * p.H + h] = (m_e + log2f(l_tot)) * 0.6931471805599453f;
      }
      // the accumulator is free for the item after next: its first P V is issued only after these threads have
      // arrived on p_full for that item's first block, which comes after this read in program order
      tc::tc_fence_before();
      return true;
    };
    for (int item = blockIdx.x; ok && item < p.total_items; item += gridDim.x) {
      const CaItem it = ca_item<SPLIT, LENGTHS>(p, item);
      if (SPLIT > 1) pend_it = it;
      if (it.nb == 0) {
        if (SPLIT > 1) continue;                              // nothing of this item falls to this CTA
        // no encoder position: the attention output is defined as zero
        const int m = it.tile * kCaBM + row;
        if (m < p.M) {
          const int64_t r_out = (int64_t)it.b * p.M + m;
          uint4* dst = reinterpret_cast<uint4*>(p.out + r_out * p.out_row_stride + it.h * DH + kOutCols * half);
#pragma unroll
          for (int i = 0; i < kOutCols / 8; ++i) dst[i] = make_uint4(0u, 0u, 0u, 0u);
          if (p.lse != nullptr && half == 0) p.lse[r_out * p.H + it.h] = -INFINITY;
        }
        continue;
      }
      const uint32_t o_acc = tmem_o + (uint32_t)((li & 1) * DH);
      float m_run = -INFINITY, l_run = 0.f;
      for (int j = 0; j < it.nb; ++j, ++g) {
        ok = ok && tc::mbar_wait(s_full, g & 1, abort_flag);
        ok = __all_sync(kFullMask, ok);
        if (!ok) break;
        tc::tc_fence_after();
        uint32_t r[kCols];
        {
#pragma unroll
          for (int c = 0; c < kCols; c += 32)
            tc::tmem_ld32(tmem_s + lane_addr + col_base + c, *reinterpret_cast<uint32_t(*)[32]>(&r[c]));
          tc::tmem_ld_wait();
        }
        tc::tc_fence_before();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(s_free);              // the scores now live in registers
        const int valid = min(kCaBN, it.T - j * kCaBN) - col_base;   // this thread's columns that exist
        if (valid < kCols) {
#pragma unroll
          for (int i = 0; i < kCols; ++i)
            if (i >= valid) r[i] = 0xff800000u;                     // -inf: no weight, no influence on the max
        }
        // four independent chains instead of one 32-deep one
        float mx0 = max3(__uint_as_float(r[0]), __uint_as_float(r[1]), __uint_as_float(r[2]));
        float mx1 = max3(__uint_as_float(r[3]), __uint_as_float(r[4]), __uint_as_float(r[5]));
        float mx2 = max3(__uint_as_float(r[6]), __uint_as_float(r[7]), __uint_as_float(r[8]));
        float mx3 = max3(__uint_as_float(r[9]), __uint_as_float(r[10]), __uint_as_float(r[11]));
#pragma unroll
        for (int i = 12; i + 7 < kCols; i += 8) {
          mx0 = max3(mx0, __uint_as_float(r[i]), __uint_as_float(r[i + 1]));
          mx1 = max3(mx1, __uint_as_float(r[i + 2]), __uint_as_float(r[i + 3]));
          mx2 = max3(mx2, __uint_as_float(r[i + 4]), __uint_as_float(r[i + 5]));
          mx3 = max3(mx3, __uint_as_float(r[i + 6]), __uint_as_float(r[i + 7]));
        }
        mx0 = max3(mx0, __uint_as_float(r[kCols - 4]), __uint_as_float(r[kCols - 3]));
        mx1 = max3(mx1, __uint_as_float(r[kCols - 2]), __uint_as_float(r[kCols - 1]));
        float mx = fmaxf(max3(mx0, mx1, mx2), mx3);
        float* hm = half_max + (g & 1) * 256;
        hm[half * 128 + row] = mx;
        tc::named_bar_sync(2 + quarter, 64);                  // the two warps of this row quarter
        mx = fmaxf(mx, hm[(half ^ 1) * 128 + row]);
        const float m_blk = mx * p.scale_log2;
        const bool grow = m_blk > m_run + 8.0f;               // always true on an item's first block
        const float m_new = grow ? m_blk : m_run;
        const float alpha = grow ? ex2(m_run - m_new) : 1.0f; // 0 on the first block
        m_run = m_new;
        // probabilities -> packed bf16 in the P columns; row sum in four independent accumulators
        const float neg_m = -m_new;
        float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
        uint32_t lo[P32 ? kCols / 2 : 1];
#pragma unroll
        for (int i = 0; i < kCols / 4; ++i) {
          const float e0 = ex2(fmaf(__uint_as_float(r[4 * i]), p.scale_log2, neg_m));
          const float e1 = ex2(fmaf(__uint_as_float(r[4 * i + 1]), p.scale_log2, neg_m));
          const float e2 = ex2(fmaf(__uint_as_float(r[4 * i + 2]), p.scale_log2, neg_m));
          const float e3 = ex2(fmaf(__uint_as_float(r[4 * i + 3]), p.scale_log2, neg_m));
          s0 += e0; s1 += e1; s2 += e2; s3 += e3;
          const uint32_t h0 = pack_bf16x2(e0, e1), h1 = pack_bf16x2(e2, e3);
          r[2 * i] = h0;
          r[2 * i + 1] = h1;
          if (P32) {
            lo[2 * i] = pack_bf16x2(e0 - bf16_lo(h0), e1 - bf16_hi(h0));
            lo[2 * i + 1] = pack_bf16x2(e2 - bf16_lo(h1), e3 - bf16_hi(h1));
          }
        }
        l_run = fmaf(l_run, alpha, (s0 + s1) + (s2 + s3));
        constexpr int kPBack = P32 ? 1 : 2;                   // the P columns were last read by P V of block g - kPBack
        if (g >= kPBack) {
          ok = wait_pv(g - kPBack);                           // (two blocks back: long finished, but it must be)
          if (!ok) break;
          tc::tc_fence_after();
        }
        {
          const uint32_t p_cols = tmem_p + (uint32_t)(P32 ? 0 : (g & 1) * 64) + lane_addr + (kCols / 2) * half;
#pragma unroll
          for (int c = 0; c < kCols / 2; c += 16) {
            tc::tmem_st16(p_cols + c, *reinterpret_cast<uint32_t(*)[16]>(&r[c]));
            if (P32) tc::tmem_st16(p_cols + 64 + c, *reinterpret_cast<uint32_t(*)[16]>(&lo[P32 ? c : 0]));
          }
        }
        if (j > 0 && __any_sync(kFullMask, grow)) {           // rare after the first blocks
          // O changes under the tensor core only here: P V of block g - 1 (the same item) must be complete
          ok = wait_pv(g - 1);
          if (!ok) break;
          tc::tc_fence_after();
#pragma unroll
          for (int c = 0; c < kOutCols; c += 32) {
            uint32_t o[32];
            tc::tmem_ld32(o_acc + lane_addr + kOutCols * half + c, o);
            tc::tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
            uint32_t (&o0)[16] = *reinterpret_cast<uint32_t(*)[16]>(&o[0]);
            uint32_t (&o1)[16] = *reinterpret_cast<uint32_t(*)[16]>(&o[16]);
            tc::tmem_st16(o_acc + lane_addr + kOutCols * half + c, o0);
            tc::tmem_st16(o_acc + lane_addr + kOutCols * half + c + 16, o1);
          }
        }
        // Positions past the request's length: their probabilities are 0, but 0 times what the padding holds (NaN, Inf) is
        // not.  P V leaves out whole k-steps of them; the rest of a k-step's rows of V is cleared here.  (Past p.T the
        // loads left zeros.)  16 x 1000 x 16 x 128 x 50..200: 57.5 us without, 59.2 so; cleared by the issuing thread
        // 62, by a warp of its own 64, not loaded at all (boxes of 64, 32 .. 1 rows) 65; without leaving k-steps out 61.
        const int left = it.T - j * kCaBN;
        if (LENGTHS && left < kCaBN && it.t0 + it.T < p.T && (left & 15) != 0) {
          ok = tc::mbar_wait(v_full + (g & 1), (g >> 1) & 1, abort_flag);
          ok = __all_sync(kFullMask, ok);
          if (!ok) break;
          const int i = left * 8 + (int)threadIdx.x;          // 16-byte pieces of the half's 128-byte rows
          if (i < ((left + 15) & ~15) * 8) {
#pragma unroll
            for (int hf = 0; hf < kHalves; ++hf)
              reinterpret_cast<uint4*>(kv_tiles + (2 * (g & 1) + 1) * kCaTileBytes + hf * kCaHalfBytes)[i] = make_uint4(0u, 0u, 0u, 0u);
            tc::fence_proxy_async_smem();
          }
        }
        tc::tmem_st_wait();
        tc::tc_fence_before();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(p_full + (g & 1));
        // the previous item's output, now that this block is with the tensor core
        if (SPLIT == 1 && pend_g >= 0) {
          ok = store_item(pend_it, pend_g, pend_li, pend_m, pend_l);
          pend_g = -1;
          if (!ok) break;
        }
      }
      if (!ok) break;
      pend_it = it; pend_g = g - 1; pend_li = li; pend_m = m_run; pend_l = l_run;
      ++li;
    }
    if (SPLIT == 1) {
      if (ok && pend_g >= 0) store_item(pend_it, pend_g, pend_li, pend_m, pend_l);
    } else {
      // ---- merge of the cluster's partial results ----
      const int rank = (int)tc::cluster_cta_rank();
      const bool have = pend_g >= 0;                          // this CTA had blocks of the item
      if (have) { ok = wait_pv(pend_g) && ok; tc::tc_fence_after(); }
      half_sum[half * 128 + row] = pend_l;
      tc::named_bar_sync(2 + quarter, 64);
      const float l_tot = pend_l + half_sum[(half ^ 1) * 128 + row];
      const float2 ml = make_float2(have ? pend_m : -INFINITY, have ? l_tot : 0.f);
      __syncwarp();
      asm volatile("barrier.cluster.wait.aligned;" ::: "memory");        // the other CTAs have started
      // A slice of kSlice columns goes to its owner (16 at a time; the two threads of a row take every second piece)
      auto read_o = [&](int col, uint32_t (&o)[16]) {
        if (have) {
          tc::tmem_ld16(tmem_o + lane_addr + (uint32_t)col, o);
          tc::tmem_ld_wait();
        } else {
#pragma unroll
          for (int i = 0; i < 16; ++i) o[i] = 0u;
        }
      };
      constexpr int kPieces = kSlice / 16;
#pragma unroll 1
      for (int o = 1; o < SPLIT; ++o) {
        const int dst = (rank + o) % SPLIT, slot = rank < dst ? rank : rank - 1;
#pragma unroll 1
        for (int c = 0; c < kPieces; ++c) {
          if (((c + o) & 1) != half) continue;
          uint32_t v[16];
          read_o(dst * kSlice + 16 * c, v);
          const uint32_t remote = tc::cluster_addr_of(xbuf + (slot * (kSlice / 4) + 4 * c) * 128 + row, (uint32_t)dst);
#pragma unroll
          for (int j = 0; j < 4; ++j)
            asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};"
                         ::"r"(remote + (uint32_t)(j * 128 * 16)), "r"(v[4 * j]), "r"(v[4 * j + 1]), "r"(v[4 * j + 2]),
                           "r"(v[4 * j + 3]) : "memory");
        }
        if (half == 0)
          asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};"
                       ::"r"(tc::cluster_addr_of(mlbuf + rank * 128 + row, (uint32_t)dst)), "f"(ml.x), "f"(ml.y) : "memory");
      }
      if (half == 0) mlbuf[rank * 128 + row] = ml;
      tc::cluster_sync_all();
      float m_all = -INFINITY, l_all = 0.f, w[SPLIT];
#pragma unroll
      for (int s = 0; s < SPLIT; ++s) { w[s] = mlbuf[s * 128 + row].x; m_all = fmaxf(m_all, w[s]); }
#pragma unroll
      for (int s = 0; s < SPLIT; ++s) {
        w[s] = w[s] == -INFINITY ? 0.f : ex2(w[s] - m_all);
        l_all = fmaf(mlbuf[s * 128 + row].y, w[s], l_all);
      }
      const float inv = l_all == 0.f ? 0.f : 1.f / l_all;      // no encoder position: the output is defined as zero (NaN stays)
      const int m = pend_it.tile * kCaBM + row;
      const int64_t r_out = (int64_t)pend_it.b * p.M + m;
      const bool live = ok && m < p.M;
#pragma unroll 1
      for (int c = 0; c < kPieces; ++c) {
        if ((c & 1) != half) continue;
        uint32_t own[16];
        read_o(rank * kSlice + 16 * c, own);
        float v[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = 0.f;
#pragma unroll
        for (int s = 0; s < SPLIT; ++s) {                      // in rank order, whoever owns the columns
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            float4 t = make_float4(__uint_as_float(own[4 * j]), __uint_as_float(own[4 * j + 1]),
                                   __uint_as_float(own[4 * j + 2]), __uint_as_float(own[4 * j + 3]));
            if (s != rank) t = xbuf[((s < rank ? s : s - 1) * (kSlice / 4) + 4 * c + j) * 128 + row];
            v[4 * j] = fmaf(t.x, w[s], v[4 * j]); v[4 * j + 1] = fmaf(t.y, w[s], v[4 * j + 1]);
            v[4 * j + 2] = fmaf(t.z, w[s], v[4 * j + 2]); v[4 * j + 3] = fmaf(t.w, w[s], v[4 * j + 3]);
          }
        }
        if (live) {
          uint4* dst = reinterpret_cast<uint4*>(p.out + r_out * p.out_row_stride + pend_it.h * DH + rank * kSlice + 16 * c);
#pragma unroll
          for (int j = 0; j < 2; ++j)
            dst[j] = make_uint4(pack_bf16x2(v[8 * j] * inv, v[8 * j + 1] * inv), pack_bf16x2(v[8 * j + 2] * inv, v[8 * j + 3] * inv),
                                pack_bf16x2(v[8 * j + 4] * inv, v[8 * j + 5] * inv), pack_bf16x2(v[8 * j + 6] * inv, v[8 * j + 7] * inv));
        }
      }
      if (live && p.lse != nullptr && rank == 0 && half == 0)
        p.lse[r_out * p.H + pend_it.h] = l_all == 0.f ? -INFINITY : (m_all + log2f(l_all)) * 0.6931471805599453f;
      tc::tc_fence_before();
    }
  }
  if (SPLIT > 1 && warp >= kCaSoftmaxWarps) {                  // the producer's and the issuer's part in the two cluster barriers
    __syncwarp();
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
    tc::cluster_sync_all();
  }
  tc::tc_fence_before();
  __syncthreads();
  if (warp == kCaSoftmaxWarps) tc::tmem_dealloc(tmem_base, kCaTmemCols);
}

inline bool cross_attn_tc_supported(int B, int M, int H, int d_h, int T_ctx) {
  return (d_h == 64 || d_h == 128) && H <= 65535 && B <= 65535 && T_ctx >= 1 && M >= 1;
}

template <int DH, int SPLIT, bool P32, bool LENGTHS>
inline grace_status_t launch_cross_attn_tc_form(const CUtensorMap& mq, const CUtensorMap& mk, const CUtensorMap& mv,
                                                const CrossTcParams& p, int items, cudaStream_t s) {
  constexpr int kCaSmemBytes = CaCfg<DH, SPLIT>::kSmemBytes;
  static unsigned long long attr_set_devices = 0;
  static int n_sm_of[kMaxDevices] = {0};
  DeviceSetup su(&attr_set_devices);
  if (su) {
    GRACE_CUDA_TRY(cudaFuncSetAttribute(cross_attn_tc_kernel<DH, SPLIT, P32, LENGTHS>, cudaFuncAttributeMaxDynamicSharedMemorySize, kCaSmemBytes));
    GRACE_CUDA_TRY(cudaDeviceGetAttribute(&n_sm_of[su.dev], cudaDevAttrMultiProcessorCount, su.dev));
    su.done();
  }
  const int n_sm = n_sm_of[su.dev];
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = SPLIT; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.gridDim = dim3(SPLIT > 1 ? items * SPLIT : (items < n_sm ? items : n_sm));
  cfg.blockDim = dim3(kCaThreads); cfg.dynamicSmemBytes = kCaSmemBytes; cfg.stream = s;
  cfg.attrs = attr; cfg.numAttrs = SPLIT > 1 ? 2 : 1;
  cudaLaunchKernelEx(&cfg, cross_attn_tc_kernel<DH, SPLIT, P32, LENGTHS>, mq, mk, mv, p);
  GRACE_LAUNCH_CHECK();
  return GRACE_OK;
}

// split: how many CTAs share a work item (1, 2 or 4); p32: fp32-like probabilities (above).  GRACE_UNSUPPORTED_SHAPE, with
// nothing launched: too many items, or (p32) strides that a tensor map cannot express.
template <int DH>
inline grace_status_t launch_cross_attn_tc(const uint16_t* q, int64_t q_row_stride, const uint16_t* k,
                                           const uint16_t* v, int64_t kv_stride_b, int64_t kv_stride_h,
                                           int64_t kv_stride_t, uint16_t* out, int64_t out_row_stride, float* lse,
                                           const int32_t* enc_len, int B, int M, int H, int T_ctx, float scale, int split, bool p32,
                                           cudaStream_t s) {
  CUtensorMap mq, mk, mv;
  const grace_status_t no_map = p32 ? GRACE_UNSUPPORTED_SHAPE : GRACE_CUDA_ERROR;
  {
    const uint64_t dims[4] = {(uint64_t)DH, (uint64_t)H, (uint64_t)M, (uint64_t)B};
    const uint64_t str[3] = {(uint64_t)DH, (uint64_t)q_row_stride, (uint64_t)M * (uint64_t)q_row_stride};
    const uint32_t box[4] = {64u, 1u, (uint32_t)kCaBM, 1u};
    if (!tc::make_tmap_bf16(&mq, q, 4, dims, str, box)) return no_map;
  }
  {
    const uint64_t dims[4] = {(uint64_t)DH, (uint64_t)T_ctx, (uint64_t)H, (uint64_t)B};
    const uint64_t str[3] = {(uint64_t)kv_stride_t, (uint64_t)kv_stride_h, (uint64_t)kv_stride_b};
    const uint32_t box[4] = {64u, (uint32_t)kCaBN, 1u, 1u};
    if (!tc::make_tmap_bf16(&mk, k, 4, dims, str, box)) return no_map;
    if (!tc::make_tmap_bf16(&mv, v, 4, dims, str, box)) return no_map;
  }
  CrossTcParams p;
  p.out = out; p.lse = lse; p.enc_len = enc_len; p.out_row_stride = out_row_stride; p.B = B; p.M = M; p.H = H; p.T = T_ctx;
  p.tiles_m = (M + kCaBM - 1) / kCaBM;
  const int64_t items = (int64_t)p.tiles_m * H * B;
  if (items * split > 0x7fffffff) return GRACE_UNSUPPORTED_SHAPE;
  p.total_items = (int)items * split;
  p.scale_log2 = scale * 1.4426950408889634f;
  const int n = (int)items;
  if (enc_len != nullptr) {
    if (p32) {
      if constexpr (DH == 128) {                             // (at head size 64 these are more items than SMs)
        if (split == 4) return launch_cross_attn_tc_form<DH, 4, true, true>(mq, mk, mv, p, n, s);
        if (split == 2) return launch_cross_attn_tc_form<DH, 2, true, true>(mq, mk, mv, p, n, s);
      }
      return launch_cross_attn_tc_form<DH, 1, true, true>(mq, mk, mv, p, n, s);
    }
    if constexpr (DH == 64) {                                // (at head size 128 lengths mean p32)
      if (split == 4) return launch_cross_attn_tc_form<DH, 4, false, true>(mq, mk, mv, p, n, s);
      if (split == 2) return launch_cross_attn_tc_form<DH, 2, false, true>(mq, mk, mv, p, n, s);
      return launch_cross_attn_tc_form<DH, 1, false, true>(mq, mk, mv, p, n, s);
    }
  }
  if (split == 4) return launch_cross_attn_tc_form<DH, 4, false, false>(mq, mk, mv, p, n, s);
  if (split == 2) return launch_cross_attn_tc_form<DH, 2, false, false>(mq, mk, mv, p, n, s);
  return launch_cross_attn_tc_form<DH, 1, false, false>(mq, mk, mv, p, n, s);
}

}  // namespace grace
