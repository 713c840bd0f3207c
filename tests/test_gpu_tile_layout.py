"""GPU parity at the edges of the tile layout and of the kernels that write and read it: every mix of widths in a tile, lists
and groups that end anywhere, tiles with more outliers than are listed on chip, thresholds and ranges that are not ordinary
numbers, runs of tiles cut anywhere, several queries in one launch.  Bit-exact against the CPU oracle where it is a matter of
stored bytes; attention within the tolerance of the other parity tests (ATOL + RTOL * |ref|)."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2403_04643_b200 import qaq, synth

from gpu_helpers import assert_attention_close, compare_export, gpu_pipeline, make_inputs, oracle_batch, u16

pytestmark = pytest.mark.gpu

HYPER = (0.002, 0.01, 128.0)


def _widths(wl, T, mix, seed):
    g = torch.Generator().manual_seed(seed)
    if mix == "any":                         # every width, sections of a few rows
        return torch.randint(1, 9, (wl.bh, T), generator=g, dtype=torch.uint8)
    if mix == "one odd":                     # one wide token among narrow ones: a group of values at the width of one of its tokens
        b = torch.full((wl.bh, T), 2, dtype=torch.uint8)
        b[:, 5::64] = 7
        return b
    lo, hi = mix                             # sections of lo rows, the rest: remainders of 16 rows (keys) and 4 groups (values)
    t = torch.arange(T) % 64
    return torch.where(t < lo, hi, 11 - hi).to(torch.uint8).expand(wl.bh, T).contiguous()


@pytest.mark.parametrize("D", [32, 64, 128])
@pytest.mark.parametrize("mix", ["any", "one odd", (1, 8), (15, 3), (17, 5), (49, 4), (63, 6)])
def test_every_mix_of_widths(D, mix):
    # 128 tokens in whole tiles, 37 in an open one; 5 % outliers
    wl = synth.scaled(synth.CONFIGS["C2"], heads=2, head_dim=D, tokens=165, alpha=0.05, bits_min=1, seed=D)
    K, V, q, ring, nv = make_inputs(wl)
    bK, bV = _widths(wl, 165, mix, 3), _widths(wl, 165, mix, 4)
    pol = qaq.qaq_policy_from_hyper(*HYPER, 165)
    cfg, cache, thr, out, scores, dev = gpu_pipeline(wl, K, V, q, ring, nv, pol, bits=(bK, bV))
    ref = oracle_batch(wl, K, V, q, ring, nv, pol.cK, pol.cV, bitsK=bK.numpy(), bitsV=bV.numpy())
    compare_export(cache, ref)
    assert_attention_close(out.cpu().numpy(), ref.X)


def _same_cache(a, b):
    for x in (0, 1):
        ea, eb = qaq.qaq_cache_export(a, x), qaq.qaq_cache_export(b, x)
        for k in ("bits", "off", "rowptr", "codes", "ch"):
            assert torch.equal(ea[k], eb[k]), (x, k)
        for k in ("mn", "step", "val"):
            ua, ub = (e[k].contiguous().view(torch.int16 if e[k].dtype == torch.float16 else torch.int32) for e in (ea, eb))
            assert torch.equal(ua, ub), (x, k)


@pytest.mark.parametrize("D", [32, 64, 128])
@pytest.mark.parametrize("bounds", ["most are outliers", "crossed", "not a number", "none, with infinities", "all equal"])
def test_whole_tiles_equal_tiles_filled_in_pieces(D, bounds):
    # whole tiles (one kernel) against the same tokens appended 40 + 24 + 50 + 14 (the other one), at thresholds and data at
    # which the two could part
    T, BH = 128, 3
    g = torch.Generator().manual_seed(D)
    K = torch.randn((1, BH, T, D), generator=g).half()
    V = torch.randn((1, BH, T, D), generator=g).half()
    thr = torch.tensor([-0.2, 0.2] * 2)
    if bounds == "crossed": thr = torch.tensor([0.5, -0.5] * 2)
    if bounds == "not a number": thr = torch.tensor([math.nan, 1.0] * 2)
    if bounds == "none, with infinities":
        thr = torch.tensor([-math.inf, math.inf] * 2)
        for X in (K, V):
            X[:, :, 3, 5] = math.inf; X[:, :, 70, D - 1] = -math.inf
            X[:, 1, 9, 0] = math.inf; X[:, 1, 9, 7] = -math.inf; X[:, 2, 100, 31] = math.nan
    if bounds == "all equal":
        K[:], V[:] = 0.75, -0.0
        thr = torch.tensor([-1.0, 1.0] * 2)
    thr = thr.repeat(BH, 1).cuda().contiguous()
    bK = torch.randint(1, 9, (BH, T), generator=g, dtype=torch.uint8).cuda()
    bV = torch.randint(1, 9, (BH, T), generator=g, dtype=torch.uint8).cuda()
    cfg = qaq.make_config(1, BH, D, T, 1, 8, 4, 0.01, 2 * T * D)
    Kd, Vd = K.cuda(), V.cuda()
    whole, pieces = qaq.Cache(cfg), qaq.Cache(cfg)
    qaq.qaq_quantize_append(whole, Kd, Vd, thr, bitsK=bK, bitsV=bV)
    for a, b in ((0, 40), (40, 64), (64, 114), (114, 128)):
        qaq.qaq_quantize_append(pieces, Kd[:, :, a:b], Vd[:, :, a:b], thr, bitsK=bK[:, a:b].contiguous(), bitsV=bV[:, a:b].contiguous())
    assert qaq.qaq_cache_stats(whole).device_status == 0 and qaq.qaq_cache_stats(pieces).device_status == 0
    _same_cache(whole, pieces)


@pytest.mark.parametrize("window", [1, 15, 16, 33, 64, 71, 255])
def test_windows_of_any_number_of_rows_choose_the_oracles_widths(window):
    wl = synth.scaled(synth.CONFIGS["C2"], heads=2, tokens=192, window=window)
    K, V, q, ring, nv = make_inputs(wl, ragged=True)
    pol = qaq.qaq_policy_from_hyper(*HYPER, 192)
    cfg, cache, thr, out, scores, dev = gpu_pipeline(wl, K, V, q, ring, nv, pol)
    compare_export(cache, oracle_batch(wl, K, V, q, ring, nv, pol.cK, pol.cV))


@pytest.mark.parametrize("D,alpha,scale", [(128, 0.3, 1.0), (128, 0.05, 300.0), (64, 0.45, 1.0), (32, 0.05, 300.0)])
def test_outlier_lists_longer_than_the_buffer_and_values_too_large_for_one_word(D, alpha, scale):
    # 8-bit tiles fill the staging buffer; 0.3 * 64 * 128 = 2457 entries per tile lie beyond what is staged (and beyond what
    # the quantizer lists on chip); values above 128 take the sums of two words
    wl = synth.scaled(synth.CONFIGS["C2"], heads=2, head_dim=D, tokens=200, alpha=alpha)
    K, V, q, ring, nv = make_inputs(wl)
    K, V = (K * scale).half(), (V * scale).half()
    q = (q / scale).half()
    b = torch.full((wl.bh, 200), 8, dtype=torch.uint8)
    pol = qaq.qaq_policy_from_hyper(*HYPER, 200)
    cfg, cache, thr, out, scores, dev = gpu_pipeline(wl, K, V, q, ring, nv, pol, bits=(b, b), max_outliers=200 * D)
    ref = oracle_batch(wl, K, V, q, ring, nv, pol.cK, pol.cV, bitsK=b.numpy(), bitsV=b.numpy())
    compare_export(cache, ref)
    # the tolerance is absolute for values of order one
    assert_attention_close(out.cpu().numpy() / scale, ref.X / scale)
    q4 = torch.stack([dev[2].view(wl.bh, D)] * 3, dim=1).contiguous()
    out4 = qaq.qaq_decode_attention_multi(cache, q4, 1 / math.sqrt(D))
    for j in range(3): assert_attention_close(out4[:, j].cpu().numpy() / scale, ref.X / scale)


@pytest.mark.parametrize("n_q", [2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("heads,tokens", [(3, 65), (40, 700), (230, 130)])
def test_several_queries_in_one_launch_or_in_turn(n_q, heads, tokens):
    # groups side by side while half of the chip has a place for every (b,h) and the tiles per warp do not double; 230 (b,h)
    # have more than half of the places.  Row by row the result of a call with one query.
    D = 64
    wl = synth.scaled(synth.CONFIGS["C2"], heads=heads, head_dim=D, tokens=tokens)
    K, V, q, ring, nv = make_inputs(wl)
    pol = qaq.qaq_policy_from_hyper(*HYPER, tokens)
    cfg, cache, thr, out, scores, dev = gpu_pipeline(wl, K, V, q, ring, nv, pol)
    qs = torch.stack([synth.make_query(wl, step=i).view(wl.bh, D) for i in range(n_q)], dim=1).cuda().contiguous()
    got = qaq.qaq_decode_attention_multi(cache, qs, 1 / math.sqrt(D))
    for j in range(n_q):
        one = qaq.qaq_decode_attention(cache, qs[:, j].contiguous(), 1 / math.sqrt(D))
        # Both take the same integer products; key corrections are summed in units of 2^-24 of at most twice the query's own bound
        # 2 max|q| max|x| (of the power of two above max|q| where several share a pass), so a token's few terms (at most 4
        # here) move a logit by at most 4 * 2^-24 * 4 max|q| max|x| / sqrt(D), and its weight relatively by as much.  (The same
        # bound pays for binary32 sums in another order.)
        bound = 4 * 2.0 ** -22 * 2 * qs.abs().max().item() * K.abs().max().item() / math.sqrt(D)
        assert (got[:, j] - one).abs().max().item() <= 2 * bound * V.abs().max().item()


@pytest.mark.parametrize("tokens", [1, 64, 8192, 8193])
def test_score_rows_at_the_length_where_a_kernel_of_their_own_normalises_them(tokens):
    wl = synth.scaled(synth.CONFIGS["C2"], heads=2, head_dim=32, tokens=tokens)
    K, V, q, ring, nv = make_inputs(wl)
    pol = qaq.qaq_policy_from_hyper(*HYPER, tokens)
    cfg, cache, thr, out, scores, dev = gpu_pipeline(wl, K, V, q, ring, nv, pol)
    ref = oracle_batch(wl, K, V, q, ring, nv, pol.cK, pol.cV)
    assert_attention_close(out.cpu().numpy(), ref.X)
    S = scores.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(S - ref.S) <= 1e-6 + 1e-2 * ref.S) and np.allclose(S.sum(1), 1.0, atol=1e-3)


def test_query_rows_at_any_address():
    D = 128
    wl = synth.scaled(synth.CONFIGS["C2"], heads=5, tokens=300)
    K, V, q, ring, nv = make_inputs(wl)
    pol = qaq.qaq_policy_from_hyper(*HYPER, 300)
    cfg, cache, thr, out, scores, dev = gpu_pipeline(wl, K, V, q, ring, nv, pol)
    shifted = torch.zeros(wl.bh * D + 1, dtype=torch.float16, device="cuda")[1:]
    shifted.copy_(dev[2].reshape(-1))
    got = qaq.qaq_decode_attention(cache, shifted.view(wl.bh, D), 1 / math.sqrt(D))
    assert torch.equal(got, out)


@pytest.mark.parametrize("D,window,tokens", [(128, 64, 4097), (64, 5, 4161), (32, 64, 4500), (64, 64, 8257)])
def test_long_windows_of_any_length_and_number_of_rows(D, window, tokens):
    # above 4096 tokens: one pass with the logits in tensor memory (64 rows), two tiles to a group of warps (5 rows), two passes (8257)
    wl = synth.scaled(synth.CONFIGS["C1"], batch=1, heads=2, head_dim=D, tokens=tokens, window=window, seed=D)
    K, _ = synth.make_kv(wl)
    Q = torch.randn((wl.bh, window, D), generator=torch.Generator().manual_seed(D)).to(torch.float16)
    cfg = qaq.make_config(1, 2, D, tokens, 2, 8, window, wl.alpha)
    ring, nvalid = qaq.qaq_prefill_window(cfg, Q.cuda(), K.cuda(), 1 / math.sqrt(D))
    ring = ring.cpu().numpy().reshape(wl.bh, window, tokens).astype(np.float64)
    ku, qu = u16(K).reshape(wl.bh, tokens, D), u16(Q)
    for bh in range(wl.bh):
        want, nv, _ = oracle.prefill_window(qu[bh], ku[bh], 1 / math.sqrt(D))
        assert np.array_equal(nvalid.cpu().numpy().reshape(wl.bh, tokens)[bh], nv)
        assert np.all(ring[bh][want == 0] == 0)
        assert np.all(np.abs(ring[bh] - want) <= 1e-6 + 1e-2 * want)


@pytest.mark.parametrize("D,tokens", [(128, 65), (128, 128), (128, 129), (32, 512), (32, 513), (64, 255)])
@pytest.mark.parametrize("alpha,kind", [(0.01, "normal"), (1.0, "normal"), (0.0, "normal"), (0.3, "sorted"), (0.02, "nan"), (0.5, "few values")])
def test_thresholds_of_short_sequences(D, tokens, alpha, kind):
    # up to 16384 entries one kernel, beyond three; a bracket that misses, lists that overflow, NaNs of both signs
    g = torch.Generator().manual_seed(tokens)
    K, V = (torch.randn((1, 3, tokens, D), generator=g).half() for _ in range(2))
    if kind == "sorted": K = K.reshape(3, -1).sort(dim=1).values.reshape(1, 3, tokens, D).contiguous()      # the sample is off
    if kind == "nan":
        K[0, 0, 1::3] = math.nan; K[0, 1, 5] = -math.nan; V[:] = math.nan; V[0, 2, 0, 0] = 1.0
    if kind == "few values": K = (K * 2).round().half(); V[:] = 0.0
    cfg = qaq.make_config(1, 3, D, tokens, 2, 8, 4, alpha)
    thr = qaq.qaq_outlier_thresholds(cfg, K.cuda(), V.cuda()).cpu().numpy()
    ku, vu = u16(K).reshape(3, tokens, D), u16(V).reshape(3, tokens, D)
    want = np.array([[*oracle.thresholds(ku[b], alpha), *oracle.thresholds(vu[b], alpha)] for b in range(3)], dtype=np.float32)
    assert np.array_equal(thr, want)


@pytest.mark.parametrize("D,tokens", [(128, 513), (64, 576), (128, 1025), (32, 3650), (128, 4096)])
def test_sequences_split_over_a_cluster(D, tokens):
    # 9, 9, 17, 58 and 64 tiles: clusters of 2, 2, 3, 8 and 8 CTAs; then the same query with the token count in device memory, in
    # clusters of the size that the capacity of 4160 tokens asks for, most of whose CTAs find nothing at 70 tokens
    wl = synth.scaled(synth.CONFIGS["C2"], heads=2, head_dim=D, tokens=tokens)
    K, V, q, ring, nv = make_inputs(wl, ragged=True)
    pol = qaq.qaq_policy_from_hyper(*HYPER, tokens)
    cfg, cache, thr, out, scores, dev = gpu_pipeline(wl, K, V, q, ring, nv, pol, max_tokens=4160)
    ref = oracle_batch(wl, K, V, q, ring, nv, pol.cK, pol.cV)
    assert_attention_close(out.cpu().numpy(), ref.X)
    S = scores.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(S - ref.S) <= 1e-6 + 1e-2 * ref.S) and np.allclose(S.sum(1), 1.0, atol=1e-3)
    for n in (tokens, 70):
        if n != tokens:
            cache.reset()
            qaq.qaq_quantize_append(cache, dev[0][:, :, :n], dev[1][:, :, :n], thr, policy=pol, ring=dev[3][..., :n].contiguous(), nvalid=dev[4][..., :n].contiguous())
        want = qaq.qaq_decode_attention(cache, dev[2], 1 / math.sqrt(D))
        got, row = torch.empty_like(want), torch.empty((wl.bh, 4160), dtype=torch.float32, device="cuda")
        qaq.qaq_stream_begin(cache)
        qaq.qaq_stream_decode(cache, dev[2], 1 / math.sqrt(D), got, row)
        qaq.qaq_stream_end(cache)
        # the same tiles, summed in another order: binary32 rounding of at most 65 partial sums and weights
        assert (got - want).abs().max().item() <= 65 * 2.0 ** -23 * 4 * V.abs().max().item()
        assert torch.allclose(row[:, :n].sum(1), torch.ones(wl.bh, device="cuda"), atol=1e-3)


@pytest.mark.parametrize("heads,tokens", [(37, 1100), (49, 1600), (73, 1025), (74, 1025), (96, 2000), (98, 2000), (148, 1100)])
def test_sequences_of_many_heads_whose_clusters_may_not_all_run_at_once(heads, tokens):
    # near the largest number of (b,h) for clusters of 8, 6, 4, 3 and 2 CTAs: smaller clusters or the flattened sequence, same result
    D = 32
    wl = synth.scaled(synth.CONFIGS["C2"], heads=heads, head_dim=D, tokens=tokens)
    K, V, q, ring, nv = make_inputs(wl)
    pol = qaq.qaq_policy_from_hyper(*HYPER, tokens)
    cfg, cache, thr, out, scores, dev = gpu_pipeline(wl, K, V, q, ring, nv, pol)
    ref = oracle_batch(wl, K, V, q, ring, nv, pol.cK, pol.cV)
    assert_attention_close(out.cpu().numpy(), ref.X)
    S = scores.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(S - ref.S) <= 1e-6 + 1e-2 * ref.S) and np.allclose(S.sum(1), 1.0, atol=1e-3)


@pytest.mark.parametrize("D", [32, 64, 128])
@pytest.mark.parametrize("heads", [148, 149])
def test_open_tiles_of_many_heads(D, heads):
    # one-token and longer appends by CTAs of eight warps (148) and of four (149): the cache equals the oracle's, and one filled at once
    T = 150
    g = torch.Generator().manual_seed(heads + D)
    K, V = (torch.randn((1, heads, T, D), generator=g).half() for _ in range(2))
    bits = torch.randint(1, 9, (heads, T), generator=g).to(torch.uint8).cuda()
    cfg = qaq.make_config(1, heads, D, T, 1, 8, 1, 0.02)
    Kd, Vd = K.cuda(), V.cuda()
    thr = qaq.qaq_outlier_thresholds(cfg, Kd, Vd)
    caches = []
    for cuts in ((0, T), (0, 20, 21, 63, 64, 65, 129, 130, T)):
        cache = qaq.Cache(cfg)
        for a, b in zip(cuts, cuts[1:]):
            w = bits[:, a:b].contiguous()
            qaq.qaq_quantize_append(cache, Kd[:, :, a:b], Vd[:, :, a:b], thr, bitsK=w, bitsV=w)
        caches.append([qaq.qaq_cache_export(cache, x) for x in (0, 1)])
    th = thr.cpu().numpy()
    for x, X in enumerate((K, V)):
        a, b = caches[0][x], caches[1][x]
        assert b["stats"].device_status == 0
        assert all(torch.equal(a[k], b[k]) for k in ("bits", "mn", "step", "off", "codes", "rowptr"))
        for bh in (0, 77, heads - 1):
            want = oracle.quantize(X[0, bh].numpy().view("uint16"), th[bh, 2 * x], th[bh, 2 * x + 1], bits[bh].cpu().numpy())
            nb = int(want.off[T])
            assert (b["codes"][bh, :nb].cpu().numpy() == want.stream).all() and (b["rowptr"][bh].cpu().numpy() == want.rowptr).all()
