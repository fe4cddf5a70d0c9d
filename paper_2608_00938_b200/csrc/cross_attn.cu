// Cross-attention in the beam-as-query layout (Section 5.1, Appendix B): the M beams of a request
// are M query rows against that request's one copy of K and V.
//
// Three kernels behind one entry point:
//   * cross_attn_ms_kernel (cross_attn_ms.cuh): tcgen05 / TMEM / TMA, four softmax streams per SM,
//     head size 64: the serving shapes.
//   * cross_attn_tc_kernel (cross_attn_tc.cuh): tcgen05 / TMEM / TMA flash attention, head size 128, and head size 64
//     with few tiles.
//   * cross_attn_row_kernel (below): a (row, head) pair on its own: step 0 of a decode, the smallest searches, head
//     size 32, and more than 65535 requests or heads.
// Per-request encoder lengths take the same routes as full-length requests.  (Head size 128 with lengths ran the
// CUDA-core kernel before: 16 x 1000 x 16 x 128, lengths 50..200: 7700 us; on the tensor cores 72.)
#include "common.cuh"
#include "cross_attn_tc.cuh"
#include "cross_attn_ms.cuh"


namespace grace {

struct CrossRowParams {
  const uint16_t* q; const uint16_t* k; const uint16_t* v; uint16_t* out; float* lse;
  int64_t q_row_stride, out_row_stride, kv_stride_b, kv_stride_h, kv_stride_t;
  int R, M, H, T_ctx; float scale;
  const int32_t* enc_len;        // nullable: valid encoder positions per request
};

__device__ __forceinline__ float max_nan(float a, float b) {       // NaN if one of them is
  float m;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(m) : "f"(a), "f"(b));
  return m;
}

// A (row, head) pair on its own: a handful of query rows (step 0 of a decode: one beam per request; the smallest
// searches), where the tensor-core kernels would run one 128-row tile with a few live rows through all K/V blocks in
// sequence, and head size 32.  WARPS warps split the encoder positions of a pair (PAIRS pairs per CTA); inside a warp
// DH/8 lanes share a position (16 bytes of the K / V row each, so a row is one coalesced run), every lane group keeps an
// online-softmax state (running maximum, sum, its slice of the weighted sum) over four positions at a time; the groups of
// a warp are merged by shuffles, the warps through shared memory.  All arithmetic in fp32.
// Up to eight warps per pair request the pieces of the next four passes before the current four are used; 32 warps per
// pair, for so few pairs that the SMs have room, hide each other's loads and make the chain of passes a fourth as long.
template <int DH, int WARPS, int PAIRS>
__global__ void __launch_bounds__(WARPS * PAIRS * 32)
cross_attn_row_kernel(const CrossRowParams p) {
  pdl_wait();
  pdl_trigger();                              // not before the wait: layer_chain_kernel reads weights before its own
  constexpr int G = DH / 8;                   // lanes per encoder position
  constexpr int RP = 32 / G;                  // positions per warp pass
  constexpr bool kAhead = WARPS <= 8;
  static_assert(WARPS == 1 || PAIRS == 1, "");
  __shared__ float st_m[WARPS], st_l[WARPS], st_acc[WARPS][DH];
  const int lane = threadIdx.x & 31, warp = WARPS == 1 ? 0 : (int)(threadIdx.x >> 5);
  const int piece = lane % G, grp = lane / G;
  const int64_t pair = PAIRS == 1 ? (int64_t)blockIdx.x : (int64_t)blockIdx.x * PAIRS + (threadIdx.x >> 5);
  if (PAIRS > 1 && pair >= (int64_t)p.R * p.H) return;
  const int r = (int)(pair / p.H), h = (int)(pair - (int64_t)r * p.H);
  const int b = r / p.M;
  const uint16_t* kb = p.k + (int64_t)b * p.kv_stride_b + (int64_t)h * p.kv_stride_h + piece * 8;
  const uint16_t* vb = p.v + (int64_t)b * p.kv_stride_b + (int64_t)h * p.kv_stride_h + piece * 8;
  float q[8];
  {
    const uint4 t4 = __ldg(reinterpret_cast<const uint4*>(p.q + (int64_t)r * p.q_row_stride + h * DH) + piece);
    q[0] = bf16_lo(t4.x) * p.scale; q[1] = bf16_hi(t4.x) * p.scale; q[2] = bf16_lo(t4.y) * p.scale; q[3] = bf16_hi(t4.y) * p.scale;
    q[4] = bf16_lo(t4.z) * p.scale; q[5] = bf16_hi(t4.z) * p.scale; q[6] = bf16_lo(t4.w) * p.scale; q[7] = bf16_hi(t4.w) * p.scale;
  }
  int T = p.T_ctx;                             // valid encoder positions of this request
  if (p.enc_len != nullptr) { const int e = __ldg(p.enc_len + b); T = e < 0 ? 0 : (e < T ? e : T); }
  // this warp's contiguous slice of the encoder positions, RP at a time
  const int per_warp = (T + WARPS - 1) / WARPS;
  const int t_begin = warp * per_warp, t_end = min(T, t_begin + per_warp);
  float m_run = -INFINITY, l_run = 0.f;
  float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  constexpr int U = 4;
  uint4 kk[U], vv[U], kn[kAhead ? U : 1], vn[kAhead ? U : 1];
  auto fetch = [&](int t0, uint4* kd, uint4* vd) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int t = t0 + u * RP + grp;
      const int64_t off = (int64_t)(t < t_end ? t : t_begin) * p.kv_stride_t;
      kd[u] = __ldg(reinterpret_cast<const uint4*>(kb + off));
      vd[u] = __ldg(reinterpret_cast<const uint4*>(vb + off));
    }
  };
  if (kAhead && t_begin < t_end) fetch(t_begin, kk, vv);
  for (int t0 = t_begin; t0 < t_end; t0 += U * RP) {
    if (!kAhead) fetch(t0, kk, vv);
    else if (t0 + U * RP < t_end) fetch(t0 + U * RP, kn, vn);
    float d[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      d[u] = q[0] * bf16_lo(kk[u].x);
      d[u] = fmaf(q[1], bf16_hi(kk[u].x), d[u]); d[u] = fmaf(q[2], bf16_lo(kk[u].y), d[u]); d[u] = fmaf(q[3], bf16_hi(kk[u].y), d[u]);
      d[u] = fmaf(q[4], bf16_lo(kk[u].z), d[u]); d[u] = fmaf(q[5], bf16_hi(kk[u].z), d[u]); d[u] = fmaf(q[6], bf16_lo(kk[u].w), d[u]);
      d[u] = fmaf(q[7], bf16_hi(kk[u].w), d[u]);
    }
#pragma unroll
    for (int o = 1; o < G; o <<= 1)
#pragma unroll
      for (int u = 0; u < U; ++u) d[u] += __shfl_xor_sync(kFullMask, d[u], o);
    float m_new = m_run;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (t0 + u * RP + grp >= t_end) d[u] = -INFINITY;
      m_new = max_nan(m_new, d[u]);
    }
    if (m_new != -INFINITY) {                               // (a group past the slice's end has seen nothing yet)
      // Past the slice's end some other position was read, with a weight of 0; 0 times an infinite value is NaN.  (Cleared in
      // the last pass only: loads that depend on the position, or a test per position in every pass, cost 1 x 1 x 8 x 64 x 1024
      // 5.2 -> 6.6 and 5.9 us; so 5.3.)
      if (t0 + U * RP > t_end) {
#pragma unroll
        for (int u = 0; u < U; ++u) if (t0 + u * RP + grp >= t_end) vv[u] = make_uint4(0u, 0u, 0u, 0u);
      }
      const float corr = __expf(m_run - m_new);              // 0 the first time (m_run = -inf)
      l_run *= corr;
#pragma unroll
      for (int i = 0; i < 8; ++i) acc[i] *= corr;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const float w = __expf(d[u] - m_new);                // 0 past the end
        l_run += w;
        acc[0] = fmaf(w, bf16_lo(vv[u].x), acc[0]); acc[1] = fmaf(w, bf16_hi(vv[u].x), acc[1]);
        acc[2] = fmaf(w, bf16_lo(vv[u].y), acc[2]); acc[3] = fmaf(w, bf16_hi(vv[u].y), acc[3]);
        acc[4] = fmaf(w, bf16_lo(vv[u].z), acc[4]); acc[5] = fmaf(w, bf16_hi(vv[u].z), acc[5]);
        acc[6] = fmaf(w, bf16_lo(vv[u].w), acc[6]); acc[7] = fmaf(w, bf16_hi(vv[u].w), acc[7]);
      }
      m_run = m_new;
    }
    if (kAhead) {
#pragma unroll
      for (int u = 0; u < U; ++u) { kk[u] = kn[kAhead ? u : 0]; vv[u] = vn[kAhead ? u : 0]; }
    }
  }
  // the lane groups of the warp: a common maximum, then plain sums
  float m_w = m_run;
#pragma unroll
  for (int o = G; o < 32; o <<= 1) m_w = fmaxf(m_w, __shfl_xor_sync(kFullMask, m_w, o));
  const float f_w = m_run == -INFINITY ? 0.f : __expf(m_run - m_w);
  l_run *= f_w;
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i] *= f_w;
#pragma unroll
  for (int o = G; o < 32; o <<= 1) {
    l_run += __shfl_xor_sync(kFullMask, l_run, o);
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i] += __shfl_xor_sync(kFullMask, acc[i], o);
  }
  if (WARPS == 1) {
    const float inv = T > 0 ? 1.f / l_run : 0.f;            // no encoder position: the output is defined as zero
    if (grp == 0)
      *reinterpret_cast<uint4*>(p.out + (int64_t)r * p.out_row_stride + h * DH + piece * 8) =
          make_uint4(pack_bf16x2(acc[0] * inv, acc[1] * inv), pack_bf16x2(acc[2] * inv, acc[3] * inv),
                     pack_bf16x2(acc[4] * inv, acc[5] * inv), pack_bf16x2(acc[6] * inv, acc[7] * inv));
    if (p.lse != nullptr && lane == 0) p.lse[(int64_t)r * p.H + h] = T > 0 ? m_w + logf(l_run) : -INFINITY;
    return;
  }
  if (grp == 0) {
#pragma unroll
    for (int i = 0; i < 8; ++i) st_acc[warp][piece * 8 + i] = acc[i];
    if (piece == 0) { st_m[warp] = m_w; st_l[warp] = l_run; }
  }
  __syncthreads();
  // the warps: every warp of the first DH threads forms the common factor of each state once (a lane per state)
  if (threadIdx.x < DH) {
    const float m_s = lane < WARPS ? st_m[lane] : -INFINITY;
    float m_all = m_s;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m_all = fmaxf(m_all, __shfl_xor_sync(kFullMask, m_all, o));
    const float f = m_s == -INFINITY ? 0.f : __expf(m_s - m_all);    // a warp that saw no position
    float l_all = lane < WARPS ? st_l[lane] * f : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) l_all += __shfl_xor_sync(kFullMask, l_all, o);
    float o = 0.f;
#pragma unroll
    for (int s2 = 0; s2 < WARPS; ++s2) o = fmaf(st_acc[s2][threadIdx.x], __shfl_sync(kFullMask, f, s2), o);
    __nv_bfloat16 ob = __float2bfloat16_rn(T > 0 ? o / l_all : 0.f);    // no encoder position: zero by definition
    p.out[(int64_t)r * p.out_row_stride + h * DH + threadIdx.x] = *reinterpret_cast<uint16_t*>(&ob);
    if (p.lse != nullptr && threadIdx.x == 0) p.lse[(int64_t)r * p.H + h] = T > 0 ? m_all + logf(l_all) : -INFINITY;
  }
}

}  // namespace grace

namespace grace {
// Which kernel and, for cross_attn_tc_kernel, how many CTAs share a work item (0: cross_attn_ms_kernel).  With at most
// one 128-row tile per SM the GPU is idle beside them and an item's chain over its K / V blocks is what a call takes,
// so the blocks are split as far as SMs and blocks go (d 64: 32 tiles, 8 blocks: ms 20.9 us, split 1 14.4, 2 9.2,
// 4 7.6; 64 tiles, 4 blocks: 12.5 / 9.1 / 7.3; 128 tiles, 8 blocks: 21.2 / 15.1, 64 tiles, 1 block: 4.9 / 5.1);
// clusters that do not all fit at once cost more than they give (64 tiles, 4 blocks, split 4: 12.4).  At head size 128 a
// CTA keeps two blocks (16 tiles, 2 blocks: 6.2 / 6.7; 16 tiles, 8 blocks: 16.7 / 11.6 / 8.8).  Beyond one tile per SM
// head size 64 takes the four-stream kernel (256 tiles, 8 blocks: ms 25.0 us, tc 27.6; 512 tiles: 36.6 / 50.6).
static int cross_attn_form(int B, int M, int H, int d_h, int T_ctx, bool p32) {
  const int64_t tiles = (int64_t)((M + kCaBM - 1) / kCaBM) * H * B;
  const int blocks = (T_ctx + kCaBN - 1) / kCaBN, least = d_h == 128 ? 2 : 1;
  if (tiles > kSms) return d_h == 64 && !p32 ? 0 : 1;
  if (tiles * 4 <= kSmsInFours && blocks >= 4 * least) return 4;
  if (tiles * 2 <= kSmsInTwos && blocks >= 2 * least) return 2;
  return 1;
}
int cross_attn_tc_timeouts() { return tc::tc_timeouts_read_and_clear(); }
}  // namespace grace

extern "C" grace_status_t grace_cross_attn_varlen(const uint16_t* q, int64_t q_row_stride,
                                                  const uint16_t* k, const uint16_t* v,
                                                  int64_t kv_stride_b, int64_t kv_stride_h, int64_t kv_stride_t,
                                                  uint16_t* out, int64_t out_row_stride, float* lse,
                                                  const int32_t* enc_len,
                                                  int B, int M, int H, int d_h, int T_ctx, float scale,
                                                  int32_t* d_status, void* stream) {
  using namespace grace;
  (void)d_status;
  if (!q || !k || !v || !out) return GRACE_INVALID_ARG;
  if (B <= 0 || M <= 0 || H <= 0 || T_ctx <= 0 || (int64_t)B * M > 0x7fffffff) return GRACE_INVALID_ARG;
  if (d_h != 32 && d_h != 64 && d_h != 128) return GRACE_UNSUPPORTED_SHAPE;
  if (!grace_aligned16(q) || !grace_aligned16(k) || !grace_aligned16(v) || !grace_aligned16(out) ||
      (q_row_stride & 7) || (out_row_stride & 7) || (kv_stride_b & 7) || (kv_stride_h & 7) || (kv_stride_t & 7) ||
      q_row_stride < (int64_t)H * d_h || out_row_stride < (int64_t)H * d_h || kv_stride_t < d_h)
    return GRACE_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  CrossRowParams p;
  p.q = q; p.k = k; p.v = v; p.out = out; p.lse = lse;
  p.q_row_stride = q_row_stride; p.out_row_stride = out_row_stride;
  p.kv_stride_b = kv_stride_b; p.kv_stride_h = kv_stride_h; p.kv_stride_t = kv_stride_t;
  p.R = B * M; p.M = M; p.H = H; p.T_ctx = T_ctx; p.scale = scale; p.enc_len = enc_len;
  const int64_t pairs = (int64_t)B * M * H;
  auto run_pairs = [&](bool few) -> grace_status_t {
#define GRACE_PAIR_LAUNCH(D)                                                                                              \
  do {                                                                                                                  \
    if (few && pairs <= kSms && T_ctx >= 512)                                                                            \
      launch_pdl(cross_attn_row_kernel<D, 32, 1>, dim3((unsigned)pairs), dim3(1024), 0, s, p);                          \
    else if (few) launch_pdl(cross_attn_row_kernel<D, 8, 1>, dim3((unsigned)pairs), dim3(256), 0, s, p);                \
    else launch_pdl(cross_attn_row_kernel<D, 1, 8>, dim3((unsigned)((pairs + 7) / 8)), dim3(256), 0, s, p);             \
  } while (0)
    if (d_h == 32) GRACE_PAIR_LAUNCH(32);
    else if (d_h == 64) GRACE_PAIR_LAUNCH(64);
    else GRACE_PAIR_LAUNCH(128);
#undef GRACE_PAIR_LAUNCH
    GRACE_LAUNCH_CHECK();
    return GRACE_OK;
  };
  // Few pairs, or long ones: a CTA each, all resident at once; 32 warps each while there is one pair
  // per SM (32 x 1 x 8 x 64 x 1024: 8 warps 15.9 us, 32 warps 16.4).  A warp each when there are more and they are short:
  // eight warps win from T = pairs / 3 on at head size 64 (512 x 511 positions: 18.3 us with one warp, 11 with eight;
  // 1184: 200 positions 10 / 14, 333 23 / 22, 511 38 / 32), pairs / 2 at 32 (592 x 256: 6.6 / 5.6), pairs / 9 at 128, where a
  // warp has two lane groups only (592 x 64: 7 / 5; 1184 x 128: 12 / 15).  (1 x 1 x 8 x 64 x 1024: 8.8 us with 8 warps and states merged one by one, 5.3 now;
  // head size 32 against the kernel before, which read K and V two bytes at a time: 1 x 16 x 4 x 64: 6.0 -> 2.3 us,
  // 1 x 16 x 4 x 1024: 66 -> 4.4, 8 x 200 x 4 x 128: 31 -> 13.8, 64 x 16 x 4 x 512: 78 -> 30.)
  if ((M <= 8 || d_h == 32) && pairs <= 8 * kSms)
    return run_pairs(pairs <= 2 * kSms || (int64_t)T_ctx * (d_h == 128 ? 9 : d_h == 64 ? 3 : 2) >= pairs);
  if (cross_attn_tc_supported(B, M, H, d_h, T_ctx)) {
    // probabilities as before the tensor cores took these over: fp32 (see cross_attn_tc_kernel)
    const bool p32 = enc_len != nullptr && (d_h == 128 || M <= 8);
    // ... and any stride and any scale: what a tensor map cannot say (negative and huge strides) and scales that are not
    // positive (the softmax threads take the maximum before they scale) still run on the CUDA cores.
    if (p32 && !(scale >= 1e-30f)) return run_pairs(false);
    // A 128-row tile with a few live rows is no faster than a warp per pair while rows x positions are few (with lengths,
    // one / the tensor cores: 1 row, head size 64: 2400 pairs x 33 positions 5 / 42 us, x 1024 94 / 204; head size 128: 2368 x 33
    // 7 / 45, x 511 80 / 109; 2 rows, 64: 4800 x 1024 131 / 205, 128: 2368 x 256 36 / 38, x 511 68 / 58; 8 rows, 64: 4736 x 64
    // 10 / 12, x 128 17 / 13, 128: 2432 x 64 10 / 10).
    if (p32 && M <= 8 && ((d_h == 64 && M <= 2) || M * (int64_t)T_ctx <= 512)) return run_pairs(false);
    const int form = cross_attn_form(B, M, H, d_h, T_ctx, p32);
    if (form == 0)
      return launch_cross_attn_ms(q, q_row_stride, k, v, kv_stride_b, kv_stride_h, kv_stride_t, out,
                                  out_row_stride, lse, enc_len, B, M, H, T_ctx, scale, s);
    const grace_status_t st = (d_h == 64 ? launch_cross_attn_tc<64> : launch_cross_attn_tc<128>)(
        q, q_row_stride, k, v, kv_stride_b, kv_stride_h, kv_stride_t, out, out_row_stride, lse, enc_len, B, M, H, T_ctx,
        scale, form, p32, s);
    if (p32 && st == GRACE_UNSUPPORTED_SHAPE) return run_pairs(false);
    return st;
  }
  return run_pairs(false);
}

extern "C" grace_status_t grace_cross_attn(const uint16_t* q, int64_t q_row_stride,
                                           const uint16_t* k, const uint16_t* v,
                                           int64_t kv_stride_b, int64_t kv_stride_h, int64_t kv_stride_t,
                                           uint16_t* out, int64_t out_row_stride, float* lse,
                                           int B, int M, int H, int d_h, int T_ctx, float scale,
                                           int32_t* d_status, void* stream) {
  return grace_cross_attn_varlen(q, q_row_stride, k, v, kv_stride_b, kv_stride_h, kv_stride_t, out, out_row_stride, lse,
                                 nullptr, B, M, H, d_h, T_ctx, scale, d_status, stream);
}
