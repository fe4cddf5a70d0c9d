"""GPU parity at the sizes where a kernel or a dispatch rule can go wrong: tile edges, remainders, the smallest and the
largest of its range, against the oracle (fp64) on the same seeded inputs."""
import numpy as np
import pytest
import torch

import synth
from oracle import attention as OA
from oracle import topk as OT

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    from paper_2608_00938_b200 import api as _api
    return _api


from gpu_util import DEV, assert_attention_close, dev, dev_bf16, f64  # noqa: E402


# head size 128 with lengths: one block and several, several items per CTA with empty ones among them (more items than
# SMs), few rows per request (a CTA per row and head) at every head size it serves, and too many pairs for that
@pytest.mark.parametrize("B,M,H,d,T", [(7, 130, 16, 128, 260), (3, 257, 4, 128, 129), (40, 20, 9, 128, 130), (5, 8, 4, 64, 90),
                                       (5, 1, 2, 128, 33), (6, 8, 30, 64, 70)])
def test_cross_attn_lengths_on_every_route(api, B, M, H, d, T):
    rng = synth.rng_for(2, 1300 + M + T)
    q, k, v = (synth.normal_bf16(rng, s) for s in ((B, M, H, d), (B, H, T, d), (B, H, T, d)))
    enc_len = np.array(([T, 0, 1, 128, T - 1, 64, 0] * B)[:B], dtype=np.int32)
    enc_len = np.minimum(enc_len, T).astype(np.int32)
    ref, lse_ref = OA.cross_attn_varlen(f64(q), f64(k), f64(v), enc_len, d ** -0.5)
    kf, vf = synth.bf16_bits_to_f32(k).copy(), synth.bf16_bits_to_f32(v).copy()
    for b in range(B):                                       # what lies past a request's length has no influence
        kf[b, :, enc_len[b]:], vf[b, :, enc_len[b]:] = 50.0, -1000.0
    out = torch.full((B * M, H, d), 7.0, dtype=torch.bfloat16, device=DEV)
    lse = torch.zeros((B * M, H), dtype=torch.float32, device=DEV)
    api.grace_cross_attn_varlen(dev_bf16(q).reshape(B * M, H, d), dev(kf).to(torch.bfloat16), dev(vf).to(torch.bfloat16),
                                out, dev(enc_len), d ** -0.5, lse)
    torch.cuda.synchronize()
    got, got_lse = out.float().cpu().numpy().reshape(B, M, H, d), lse.cpu().numpy().reshape(B, M, H)
    assert_attention_close(got, ref, "cross-attn lengths")
    empty = enc_len == 0
    assert (got[empty] == 0).all() and np.isneginf(got_lse[empty]).all()
    np.testing.assert_allclose(got_lse[~empty], lse_ref[~empty], atol=2e-3, rtol=0)


@pytest.mark.parametrize("B,M,H,T", [(16, 1000, 16, 200), (20, 300, 8, 640)])
def test_cross_attn_waits_never_give_up_back_to_back(api, B, M, H, T):
    """Head size 128, launches queued without a gap, with and without lengths: no bounded wait runs out (the issuing
    thread may come arbitrarily late to its wait for a block's probabilities), and the last output is the first's."""
    d = 128
    g = torch.Generator(device=DEV)
    g.manual_seed(5)
    q, k, v = (torch.randn(*s, device=DEV, generator=g).to(torch.bfloat16) for s in ((B * M, H, d), (B, H, T, d), (B, H, T, d)))
    lengths = torch.from_numpy(np.linspace(T // 4, T, B).astype(np.int32)).to(DEV)
    first, last = torch.empty_like(q), torch.empty_like(q)
    api.grace_wait_timeouts()
    for enc_len in (None, lengths):
        def call(out):
            if enc_len is None:
                api.grace_cross_attn(q, k, v, out, d ** -0.5)
            else:
                api.grace_cross_attn_varlen(q, k, v, out, enc_len, d ** -0.5)
        call(first)
        for _ in range(4000):
            call(last)
        torch.cuda.synchronize()
        assert api.grace_wait_timeouts() == 0
        assert torch.equal(first, last)


@pytest.mark.parametrize("N,V,K", [(64, 64, 16), (8192, 64, 4096), (8196, 4, 512), (32768, 2048, 1000), (32772, 4, 64),
                                   (40960, 64, 300), (65536, 1024, 4096), (100000, 1000, 700)])
@pytest.mark.parametrize("finite", [0.0, 0.001, 0.2, 1.0])
def test_topk_between_its_paths(api, N, V, K, finite):
    """Sizes around the limits of the one-kernel selection and of the sampled one, with few, some and all candidates
    finite (more than fit in shared memory among them), ties included: exact against the oracle."""
    rng = np.random.default_rng(N + K + int(1000 * finite))
    B = 3
    cand = np.where(rng.random((B, N)) < finite, np.round(rng.standard_normal((B, N)) * 50) / 16, -np.inf).astype(np.float32)
    sc, flat, par, tok = OT.beam_topk(cand, K, V)
    out = [torch.zeros(B, K, device=DEV), *(torch.zeros(B, K, device=DEV, dtype=torch.int32) for _ in range(3))]
    ws = torch.full((api.grace_beam_topk_workspace_bytes(B, N, K),), 255, device=DEV, dtype=torch.uint8)
    api.grace_beam_topk(dev(cand), K, V, *out, ws)
    torch.cuda.synchronize()
    for got, want in zip(out, (sc, flat, par, tok)):
        assert np.array_equal(got.cpu().numpy(), want)


# the forms of linear_kernel (columns / split): 32/1, 32/1, 32/2, 64/4, 64/1, 32/1, 128/1, 128/2, 64/1, 64/4, 128/1, 128/4, 64/2, 128/1
# two CTAs per SM (centred and the additions: the pair kernel), 128/1, 128/1 two per SM, 64/1 two per SM; the pair kernel
# with the statistics kernel in front
@pytest.mark.parametrize("M,N,K", [(1, 64, 64), (17, 96, 128), (130, 512, 512), (129, 528, 2048), (512, 1536, 512), (1025, 512, 512),
                                   (1030, 2048, 512), (300, 2048, 1088), (2049, 272, 320), (5, 2048, 2048), (513, 2064, 1088),
                                   (5, 4096, 1088), (513, 528, 1088), (5001, 528, 320), (1500, 1040, 512), (700, 6160, 1088),
                                   (1025, 1040, 128), (5001, 1040, 64)])
@pytest.mark.parametrize("centred", [True, False])
def test_layer_norm_gemm_in_every_form(api, M, N, K, centred):
    """grace_linear_layer_norm (statistics inside the GEMM, K shared by the CTAs of a cluster) and the additions into
    both residual streams, at tile edges and remainders, against fp64 on the same bf16 operands.

    Bounds: LayerNorm: one rounding of the result to bf16 (2^-9 relative) and fp32 sums (a few 2^-24 of the row's absolute
    sum, scaled by rstd); additions likewise."""
    g = torch.Generator(device=DEV)
    g.manual_seed(M + N + K)
    x = torch.randn(M, K, device=DEV, generator=g)
    x = (x - x.mean(1, keepdim=True) + (0.0 if centred else 0.7)).to(torch.bfloat16)
    w = (torch.randn(N, K, device=DEV, generator=g) * 0.05).to(torch.bfloat16)
    cs, cb = w.double().sum(1).float(), torch.randn(N, device=DEV, generator=g)
    x64, w64 = x.double(), w.double()
    mean, var = x64.mean(1, keepdim=True), x64.var(1, unbiased=False, keepdim=True)
    rstd = (var + 1e-5).rsqrt()
    prod, absolute = x64 @ w64.T, x64.abs() @ w64.abs().T
    shift = 0.0 if centred else -rstd * mean * cs.double()
    want = torch.relu(rstd * prod + shift + cb.double())
    y, aff = torch.empty(M, N, device=DEV, dtype=torch.bfloat16), torch.empty(M, 2, device=DEV)
    api.grace_linear_layer_norm(x, w, 1e-5, aff, None if centred else cs, cb, y, relu=True)
    bound = 2.0 ** -8 * want.abs() + 2.0 ** -17 * (rstd * absolute + (0 if centred else (rstd * mean * cs.double()).abs())) + 1e-5
    assert ((y.double() - want).abs() <= bound).all()
    for dtype in (torch.bfloat16, torch.float32):
        r = torch.randn(M, N, device=DEV, generator=g).to(dtype)
        want = r.double() + prod
        if dtype == torch.bfloat16:
            api.grace_linear_add_bf16(x, w, r)
            bound = 2.0 ** -8 * (want.abs() + prod.abs()) + 2.0 ** -19 * absolute
        else:
            api.grace_linear(x, w, r, residual=r)
            bound = 2.0 ** -19 * absolute + 2.0 ** -22 * want.abs()
        assert ((r.double() - want).abs() <= bound + 1e-30).all()


# 32/1, 32/1, the pair kernel twice (the ninth: 64/1), 32/1, the pair kernel, 128/4, 64/4, 128/1, 64/2, 32/2, 128/4, 128/1 two CTAs per SM
@pytest.mark.parametrize("M,N,K,count", [(1, 64, 64, 2), (129, 512, 128, 4), (1024, 512, 512, 8), (2000, 512, 512, 9), (33, 528, 320, 17),
                                         (9000, 256, 192, 8), (1, 512, 512, 8), (130, 512, 1088, 2), (500, 512, 512, 8),
                                         (40, 528, 1088, 8), (130, 128, 512, 3), (700, 144, 2048, 2), (900, 272, 512, 8)])
def test_linear_multi_is_the_single_products(api, M, N, K, count):
    """Every product of grace_linear_multi against fp64 (fp32 sums, one rounding to bf16), with more products than a
    launch takes, tiles that cut the last rows and columns, and neighbours' outputs that must stay apart."""
    g = torch.Generator(device=DEV)
    g.manual_seed(M + N + K)
    x = torch.randn(M, K, device=DEV, generator=g).to(torch.bfloat16)
    ws = [(torch.randn(N, K, device=DEV, generator=g) * 0.1).to(torch.bfloat16) for _ in range(count)]
    ys = [torch.full((M, N), float("nan"), device=DEV, dtype=torch.bfloat16) for _ in range(count)]
    api.grace_linear_multi(x, ws, ys)
    for w, y in zip(ws, ys):
        want, absolute = x.double() @ w.double().T, x.double().abs() @ w.double().abs().T
        assert ((y.double() - want).abs() <= 2.0 ** -8 * want.abs() + 2.0 ** -19 * absolute + 1e-30).all()


# a (row, head) pair on its own: 32, 8 and 1 warps per pair at every head size that takes them; slices of the positions that
# some warps or lane groups have none of; a last CTA with fewer pairs than it has warps
@pytest.mark.parametrize("B,M,H,d,T", [(1, 1, 8, 64, 1030), (2, 3, 5, 128, 513), (1, 16, 4, 32, 700), (1, 8, 8, 64, 5), (3, 2, 2, 128, 1),
                                       (2, 100, 3, 32, 37), (7, 61, 3, 32, 129), (4, 300, 1, 32, 1)])
def test_cross_attn_pairs(api, B, M, H, d, T):
    rng = synth.rng_for(2, 1400 + M + T)
    q, k, v = (synth.normal_bf16(rng, s) for s in ((B, M, H, d), (B, H, T, d), (B, H, T, d)))
    ref, lse_ref = OA.cross_attn(f64(q), f64(k), f64(v), d ** -0.5)
    out = torch.full((B * M, H, d), 7.0, dtype=torch.bfloat16, device=DEV)
    lse = torch.zeros((B * M, H), dtype=torch.float32, device=DEV)
    api.grace_cross_attn(dev_bf16(q).reshape(B * M, H, d), dev_bf16(k), dev_bf16(v), out, d ** -0.5, lse)
    torch.cuda.synchronize()
    # fp32 throughout: the output's rounding to bf16 alone
    got = out.double().cpu().numpy().reshape(B, M, H, d)
    assert (np.abs(got - ref) <= 2.0 ** -8 * np.abs(ref) + 1e-5).all()
    np.testing.assert_allclose(lse.cpu().numpy().reshape(B, M, H), lse_ref, atol=1e-4, rtol=0)


# head size 64 beyond one tile per SM (the four-stream kernel), several items per half, the last rows of a request in one
# tile of two: items with one live tile and with two in the same half
@pytest.mark.parametrize("B,M,H,T", [(16, 600, 8, 130), (20, 300, 8, 200), (13, 1100, 5, 70), (30, 100, 10, 65)])
@pytest.mark.parametrize("lengths", [False, True])
def test_cross_attn_items_with_one_tile_and_with_two(api, B, M, H, T, lengths):
    d = 64
    rng = synth.rng_for(2, 1500 + M + T)
    q, k, v = (synth.normal_bf16(rng, s) for s in ((B, M, H, d), (B, H, T, d), (B, H, T, d)))
    enc_len = np.minimum(np.array([T, 0, 1, 64, T - 1, 65, 0, 63] * B)[:B], T).astype(np.int32)
    out = torch.full((B * M, H, d), 7.0, dtype=torch.bfloat16, device=DEV)
    lse = torch.zeros((B * M, H), dtype=torch.float32, device=DEV)
    args = dev_bf16(q).reshape(B * M, H, d), dev_bf16(k), dev_bf16(v), out
    if lengths:
        ref, lse_ref = OA.cross_attn_varlen(f64(q), f64(k), f64(v), enc_len, d ** -0.5)
        api.grace_cross_attn_varlen(*args, dev(enc_len), d ** -0.5, lse)
    else:
        ref, lse_ref = OA.cross_attn(f64(q), f64(k), f64(v), d ** -0.5)
        api.grace_cross_attn(*args, d ** -0.5, lse)
    torch.cuda.synchronize()
    assert api.grace_wait_timeouts() == 0
    got, got_lse = out.float().cpu().numpy().reshape(B, M, H, d), lse.cpu().numpy().reshape(B, M, H)
    assert_attention_close(got, ref, "one tile and two")
    some = enc_len > 0 if lengths else np.ones(B, bool)
    assert (got[~some] == 0).all() and np.isneginf(got_lse[~some]).all()
    np.testing.assert_allclose(got_lse[some], lse_ref[some], atol=2e-3, rtol=0)


# the four-stream kernel (head size 64, more than one tile per SM); the one-stream kernel: head size 128, items of a CTA
# alone and shared by clusters of two and four (CTAs of them without any block), head size 64 shared by two and four, few
# rows per request with more pairs than the pair kernel takes; a (row, head) pair per CTA and per warp
PADDED = [(20, 300, 8, 64, 200), (16, 600, 8, 64, 130), (10, 257, 8, 128, 300), (10, 20, 7, 128, 700), (10, 130, 1, 128, 1100),
          (10, 130, 3, 64, 300), (10, 40, 3, 64, 600), (20, 8, 8, 64, 200), (20, 8, 8, 128, 200), (10, 2, 3, 64, 200),
          (10, 5, 3, 32, 200), (10, 200, 3, 32, 130), (10, 1, 3, 128, 530)]


@pytest.mark.parametrize("B,M,H,d,T", PADDED)
@pytest.mark.parametrize("padding", [float("nan"), float("inf")])
def test_cross_attn_padding_has_no_influence_whatever_it_holds(api, B, M, H, d, T, padding):
    """K and V past a request's length: NaN or infinities there give the bits that zeros give."""
    rng = synth.rng_for(2, 1600 + M + T)
    q, k, v = (dev_bf16(synth.normal_bf16(rng, s)) for s in ((B * M, H, d), (B, H, T, d), (B, H, T, d)))
    enc_len = np.minimum(np.array([T, 0, 1, 64, T - 1, 65, 17, 127, 128, 15] * B)[:B], T).astype(np.int32)
    past = torch.arange(T, device=DEV)[None, None, :, None] >= dev(enc_len)[:, None, None, None]
    results = []
    for fill in (0.0, padding):
        out, lse = torch.empty_like(q), torch.empty(B * M, H, device=DEV)
        api.grace_cross_attn_varlen(q, k.masked_fill(past, fill), v.masked_fill(past, fill), out, dev(enc_len), d ** -0.5, lse)
        results.append((out, lse))
    assert not results[0][0].isnan().any()
    assert torch.equal(results[0][0], results[1][0]) and torch.equal(results[0][1], results[1][1])


# a (row, head) pair on 32, 8 and 1 warps; lane groups whose positions are all NaN, and others that saw none; the
# one-stream kernel alone and in clusters of two and four at both head sizes; the four-stream kernel
NAN_SHAPES = [(1, 2, 3, 64, 700), (2, 3, 2, 128, 20), (5, 100, 3, 32, 40), (64, 5, 3, 64, 9), (2, 130, 3, 128, 130),
              (2, 130, 3, 128, 600), (2, 130, 3, 128, 1100), (2, 40, 3, 64, 100), (30, 40, 2, 64, 200), (2, 40, 3, 64, 600),
              (20, 300, 8, 64, 100)]


@pytest.mark.parametrize("B,M,H,d,T", NAN_SHAPES)
@pytest.mark.parametrize("lengths", [False, True])
def test_cross_attn_does_not_hide_nan(api, B, M, H, d, T, lengths):
    """A NaN in a query row, a NaN key and a score that overflows to +inf leave NaN in the outputs and the log-sum-exp they
    have a part in, whichever kernel runs, and nothing in the others: not the zeros of a request without positions."""
    rng = synth.rng_for(2, 1700 + M + T)
    q, k, v = (dev_bf16(synth.normal_bf16(rng, s)) for s in ((B * M, H, d), (B, H, T, d), (B, H, T, d)))
    enc_len = torch.full((B,), T, device=DEV, dtype=torch.int32)

    def run(q, k):
        out, lse = torch.zeros_like(q), torch.zeros(B * M, H, device=DEV)
        if lengths:
            api.grace_cross_attn_varlen(q, k, v, out, enc_len, d ** -0.5, lse)
        else:
            api.grace_cross_attn(q, k, v, out, d ** -0.5, lse)
        return out, lse

    good, good_lse = run(q, k)
    assert good.isfinite().all() and good_lse.isfinite().all()
    bad_q = q.clone()
    bad_q[M - 1, 0, 3] = float("nan")                                    # one row of request 0, one head
    bad_k = k.clone()
    bad_k[0, 0, T - 1, 5] = float("nan")
    big_q, big_k = q.clone(), k.clone()
    big_q[:M, 0, 1], big_k[0, 0, T // 2, :], big_k[0, 0, T // 2, 1] = 64.0, 0.0, 3e38
    for case, (out, lse), rows in (("query", run(bad_q, k), slice(M - 1, M)), ("key", run(q, bad_k), slice(0, M)),
                                   ("overflow", run(big_q, big_k), slice(0, M))):
        hit = torch.zeros(B * M, H, dtype=torch.bool, device=DEV)
        hit[rows, 0] = True
        assert out[hit].isnan().all() and lse[hit].isnan().all(), case
        assert torch.equal(out[~hit], good[~hit]) and torch.equal(lse[~hit], good_lse[~hit]), case


@pytest.mark.parametrize("B,M,H,d,T", [(1, 2, 3, 64, 5), (2, 3, 2, 128, 21), (5, 100, 3, 32, 7), (1, 1, 2, 64, 515)])
def test_cross_attn_pairs_with_an_infinite_value(api, B, M, H, d, T):
    """An infinite value at any one position gives the infinity in its column and leaves the other columns alone: no lane
    that has run out of positions multiplies it with a weight of zero."""
    rng = synth.rng_for(2, 1800 + M + T)
    q, k, v = (dev_bf16(synth.normal_bf16(rng, s)) for s in ((B * M, H, d), (B, H, T, d), (B, H, T, d)))
    good, out = torch.zeros_like(q), torch.zeros_like(q)
    api.grace_cross_attn(q, k, v, good, d ** -0.5)
    for t in sorted({0, 1, T // 2, T - 1}):
        w = v.clone()
        w[:, :, t, 2] = float("inf")
        api.grace_cross_attn(q, k, w, out, d ** -0.5)
        assert (out[:, :, 2] == float("inf")).all()
        assert torch.equal(out[:, :, 3:], good[:, :, 3:]) and torch.equal(out[:, :, :2], good[:, :, :2])


@pytest.mark.parametrize("B,M,H,d,T", [(3, 40, 2, 128, 150), (4, 20, 9, 128, 300), (20, 8, 8, 64, 70)])
@pytest.mark.parametrize("form", ["shared context", "shared heads", "heads backwards", "no scale", "negative scale"])
def test_cross_attn_lengths_with_any_strides_and_scale(api, B, M, H, d, T, form):
    """Calls with lengths take strides of zero, negative strides (which no tensor map can express) and scales that are not
    positive."""
    rng = synth.rng_for(2, 1900 + M + T)
    kvB, kvH = 1 if form == "shared context" else B, 1 if form == "shared heads" else H
    q, k, v = (synth.normal_bf16(rng, s) for s in ((B, M, H, d), (kvB, kvH, T, d), (kvB, kvH, T, d)))
    enc_len = np.minimum(np.array([T, 0, 1, 128, T - 1, 65] * B)[:B], T).astype(np.int32)
    scale = {"no scale": 0.0, "negative scale": -(d ** -0.5)}.get(form, d ** -0.5)
    kr, vr = (np.broadcast_to(f64(a), (B, H, T, d)) for a in (k, v))
    if form == "heads backwards":
        kr, vr = kr[:, ::-1], vr[:, ::-1]
    ref, lse_ref = OA.cross_attn_varlen(f64(q), kr, vr, enc_len, scale)
    qd, kd, vd, lens = dev_bf16(q).reshape(B * M, H, d), dev_bf16(k), dev_bf16(v), dev(enc_len)
    out, lse = torch.full_like(qd, 7.0), torch.zeros(B * M, H, device=DEV)
    if form == "heads backwards":
        last = [a[0, H - 1].data_ptr() for a in (kd, vd)]
        st = api._cross_attn_varlen(qd.data_ptr(), H * d, *last, H * T * d, -T * d, d, out.data_ptr(), H * d, lse.data_ptr(),
                                    lens.data_ptr(), B, M, H, d, T, scale, None, torch.cuda.current_stream().cuda_stream)
        assert st == api.GRACE_OK
    else:
        api.grace_cross_attn_varlen(qd, kd.expand(B, H, T, d), vd.expand(B, H, T, d), out, lens, scale, lse)
    torch.cuda.synchronize()
    some = enc_len > 0
    got, got_lse = out.float().cpu().numpy().reshape(B, M, H, d), lse.cpu().numpy().reshape(B, M, H)
    assert_attention_close(got, ref, form)
    assert (got[~some] == 0).all()
    np.testing.assert_allclose(got_lse[some], lse_ref[some], atol=2e-3, rtol=0)


@pytest.mark.parametrize("N,K,M", [(1008, 512, 16), (1024, 512, 1024), (512, 512, 2048), (64, 1024, 300)])
def test_linear_reads_weights_that_the_call_before_wrote(api, N, K, M):
    """w of one product is the output of the product in front of it on the stream, long in its K loop when the second call
    is launched: whatever the form, the second reads what the first left."""
    g = torch.Generator(device=DEV)
    g.manual_seed(N + K + M)
    a = torch.randn(N, 8192, device=DEV, generator=g).to(torch.bfloat16)
    b = (torch.randn(K, 8192, device=DEV, generator=g) * 0.02).to(torch.bfloat16)
    x = torch.randn(M, K, device=DEV, generator=g).to(torch.bfloat16)
    w = torch.empty(N, K, device=DEV, dtype=torch.bfloat16)
    want, y = torch.empty(M, N, device=DEV, dtype=torch.bfloat16), torch.empty(M, N, device=DEV, dtype=torch.bfloat16)
    aff, cb = torch.empty(M, 2, device=DEV), torch.zeros(N, device=DEV)
    calls = (lambda out: api.grace_linear(x, w, out), lambda out: api.grace_linear_multi(x, [w, w], [out, torch.empty_like(out)]),
             lambda out: api.grace_linear_layer_norm(x, w, 1e-5, aff, None, cb, out),
             lambda out: api.grace_linear_add_bf16(x, w, out.zero_()))
    for call in calls:
        api.grace_linear(a, b, w)
        torch.cuda.synchronize()
        call(want)
        for _ in range(20):
            w.fill_(float("nan"))
            api.grace_linear(a, b, w)
            call(y)
            assert torch.equal(y, want)


def test_layer_norm_gemm_of_more_row_tiles_than_a_grid_is_high(api):
    """65536 x 128 rows and one more: the form whose row tiles are gridDim.y cannot run them."""
    M, N, K = 65536 * 128 + 1, 256, 1024
    g = torch.Generator(device=DEV)
    g.manual_seed(3)
    some = torch.tensor([0, 1, 128 * 65535 - 1, 128 * 65535, M - 2, M - 1], device=DEV)
    x = torch.zeros(M, K, device=DEV, dtype=torch.bfloat16)
    x[some] = torch.randn(some.numel(), K, device=DEV, generator=g).to(torch.bfloat16)
    w = (torch.randn(N, K, device=DEV, generator=g) * 0.05).to(torch.bfloat16)
    cs, cb = w.double().sum(1).float(), torch.randn(N, device=DEV, generator=g)
    y, aff = torch.empty(M, N, device=DEV, dtype=torch.bfloat16), torch.empty(M, 2, device=DEV)
    api.grace_linear_layer_norm(x, w, 1e-5, aff, cs, cb, y)
    x64 = x[some].double()
    mean, rstd = x64.mean(1, keepdim=True), (x64.var(1, unbiased=False, keepdim=True) + 1e-5).rsqrt()
    prod, absolute = x64 @ w.double().T, x64.abs() @ w.double().abs().T
    want = rstd * (prod - mean * cs.double()) + cb.double()
    bound = 2.0 ** -8 * want.abs() + 2.0 ** -17 * rstd * (absolute + (mean * cs.double()).abs()) + 1e-5
    assert ((y[some].double() - want).abs() <= bound).all()
    assert (y[2].double() - cb.double()).abs().max() <= 2.0 ** -8 * cb.abs().max()        # a row of zeros: the bias


@pytest.mark.parametrize("M,K", [(4, 512), (1000, 512), (1024, 2048), (3000, 1088), (70, 128)])
@pytest.mark.parametrize("mean", [0.0, 0.7, 10.0])
def test_row_statistics_of_a_gemm_that_forms_them(api, M, K, mean):
    """row_affine as the GEMM leaves it against 64 bits.  Bound: (rstd, -rstd mean) are rounded to fp32 a few times each
    (2^-25 rms a rounding) and E[x^2] - mean^2 enlarges the error of the two sums by 1 + mean^2 / var; the sums themselves may
    add no more than that.  rms over the rows, three such roundings."""
    g = torch.Generator(device=DEV)
    g.manual_seed(M + K)
    x = (torch.randn(M, K, device=DEV, generator=g) + mean).to(torch.bfloat16)
    w = (torch.randn(256, K, device=DEV, generator=g) * 0.05).to(torch.bfloat16)
    cs, cb = w.double().sum(1).float(), torch.zeros(256, device=DEV)
    y, aff = torch.empty(M, 256, device=DEV), torch.zeros(M, 2, device=DEV)
    api.grace_linear_layer_norm(x, w, 1e-5, aff, cs, cb, y)
    mu, var = x.double().mean(1), x.double().var(1, unbiased=False)
    rstd = (var + 1e-5).rsqrt()
    bound = 3 * 2.0 ** -25 * (1 + (mu * mu / var).mean().item())
    assert (((aff[:, 0].double() - rstd) / rstd) ** 2).mean().sqrt() <= bound
    assert ((aff[:, 1].double() + rstd * mu).norm() / (rstd * mu).norm().clamp_min(1e-30)) <= 2 * bound


# an item shared by a cluster of two and of four CTAs at both head sizes, ragged, with and without lengths (CTAs of a cluster
# that have no block of a short request)
@pytest.mark.parametrize("B,M,H,d,T", [(1, 130, 4, 128, 600), (1, 130, 4, 128, 1100), (7, 20, 2, 128, 1030), (7, 20, 5, 128, 520),
                                       (3, 70, 2, 64, 600), (7, 130, 4, 64, 300)])
@pytest.mark.parametrize("lengths", [False, True])
def test_cross_attn_items_shared_by_clusters(api, B, M, H, d, T, lengths):
    rng = synth.rng_for(2, 2000 + M + T)
    q, k, v = (synth.normal_bf16(rng, s) for s in ((B, M, H, d), (B, H, T, d), (B, H, T, d)))
    enc_len = np.minimum(np.array([T - 3, 0, 1, 128, T, 257, 130]), T).astype(np.int32)[:B]
    out, lse = torch.full((B * M, H, d), 7.0, dtype=torch.bfloat16, device=DEV), torch.zeros((B * M, H), device=DEV)
    args = dev_bf16(q).reshape(B * M, H, d), dev_bf16(k), dev_bf16(v), out
    if lengths:
        ref, lse_ref = OA.cross_attn_varlen(f64(q), f64(k), f64(v), enc_len, d ** -0.5)
        api.grace_cross_attn_varlen(*args, dev(enc_len), d ** -0.5, lse)
    else:
        ref, lse_ref = OA.cross_attn(f64(q), f64(k), f64(v), d ** -0.5)
        api.grace_cross_attn(*args, d ** -0.5, lse)
    torch.cuda.synchronize()
    got, got_lse = out.float().cpu().numpy().reshape(B, M, H, d), lse.cpu().numpy().reshape(B, M, H)
    assert_attention_close(got, ref, "shared by clusters")
    some = enc_len > 0 if lengths else np.ones(B, bool)
    assert (got[~some] == 0).all() and np.isneginf(got_lse[~some]).all()
    np.testing.assert_allclose(got_lse[some], lse_ref[some], atol=2e-3, rtol=0)


# the four-stream kernel, and items shared by clusters of two and four at both head sizes
@pytest.mark.parametrize("B,M,H,d,T", [(20, 300, 4, 64, 640), (1, 130, 2, 128, 640), (1, 130, 2, 128, 1152), (2, 130, 2, 64, 640),
                                       (2, 130, 12, 64, 300)])
@pytest.mark.parametrize("lengths", [False, True])
def test_cross_attn_growing_scores_on_the_other_routes(api, B, M, H, d, T, lengths):
    """Scores that rise along the positions by more than the lazy-rescaling threshold, and rows where they fall: the
    accumulator is rescaled under way, and CTAs that share an item merge very different maxima."""
    rng = synth.rng_for(2, 2100 + M + T)
    q = np.abs(synth.bf16_bits_to_f32(synth.normal_bf16(rng, (B, M, H, d)))) + 0.5
    q[:, ::2] *= -1.0
    k = synth.bf16_bits_to_f32(synth.normal_bf16(rng, (B, H, T, d))) * 0.1 + np.linspace(0.0, 9.0, T, dtype=np.float32)[None, None, :, None]
    qb, kb, vb = synth.f32_to_bf16_bits(q), synth.f32_to_bf16_bits(k), synth.normal_bf16(rng, (B, H, T, d))
    scale = 0.125 if d == 64 else 0.0625
    enc_len = np.full(B, T - 5, np.int32) if lengths else np.full(B, T, np.int32)
    ref, _ = OA.cross_attn_varlen(f64(qb), f64(kb), f64(vb), enc_len, scale)
    out = torch.zeros((B * M, H, d), dtype=torch.bfloat16, device=DEV)
    args = dev_bf16(qb).reshape(B * M, H, d), dev_bf16(kb), dev_bf16(vb), out
    if lengths:
        api.grace_cross_attn_varlen(*args, dev(enc_len), scale)
    else:
        api.grace_cross_attn(*args, scale)
    torch.cuda.synchronize()
    assert_attention_close(out.float().cpu().numpy().reshape(B, M, H, d), ref, "growing scores")


# a few survivors of the attributes share the locations among the lanes of a warp: fewer locations than lanes that share
# them, counts that no share divides, one past a whole group of eight; a request that every entry's attributes let through
@pytest.mark.parametrize("n_loc", [1, 3, 9, 33])
def test_gtm_lookup_with_any_number_of_locations(api, n_loc):
    from test_gpu_ops import test_gtm_lookup_paper_form_matches_oracle as paper_form
    paper_form(api, 256, 4, 9000, 3, 21, 1, n_loc)
