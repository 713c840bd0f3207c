"""GPU checks of what the decode kernels sum in integers: that long pieces of equal weights stay inside the 32-bit
accumulators, and that the unit of the outlier sums follows from what is cached and from the query itself, not from what a
cache held before or from the queries beside it."""
import math

import pytest
import torch

import oracle
from paper_2403_04643_b200 import qaq, synth

from gpu_helpers import assert_attention_close, gpu_pipeline, make_inputs, u16

pytestmark = pytest.mark.gpu

HYPER = (0.002, 0.01, 128.0)


def test_value_sums_of_long_pieces_of_equal_weights():
    # A warp gets 296 tiles of a (b,h) in a row with one query and 395 with four, all weights equal (zero query, one value row
    # throughout), 8-bit codes and a channel in the upper half of its eight that is always the largest of its token: the sum of
    # a digit of the weight and the digit of 16 times the weight (up to 510) times 240 times 64 tokens, tile after tile.  444
    # ranges give as many digits.  The result is the row, half a step off at most.
    BH, T, D, chunk = 444, 100928, 32, 7232
    assert -(-(T // 64 * BH) // (296 * 8)) == 296 and -(-(T // 64 * BH) // (444 * 4)) == 395
    row = ((torch.arange(D) * 5 - 74) % D).float() / (D - 1)
    assert row.argmax().item() % 8 >= 4
    factor = torch.linspace(1.0, 2.0, BH + 1)[:BH]
    rows = (factor[:, None] * row[None]).half()
    cfg = qaq.make_config(1, BH, D, T, 1, 8, 1, 0.0)
    cache = qaq.Cache(cfg)
    thr = torch.tensor([-math.inf, math.inf] * 2).repeat(BH, 1).cuda().contiguous()
    K = torch.zeros((1, BH, chunk, D), dtype=torch.float16, device="cuda")
    V = rows.cuda().view(1, BH, 1, D).expand(1, BH, chunk, D).contiguous()
    bits = torch.full((BH, chunk), 8, dtype=torch.uint8, device="cuda")
    for t in range(0, T, chunk):
        n = min(chunk, T - t)
        qaq.qaq_quantize_append(cache, K[:, :, :n], V[:, :, :n], thr, bitsK=bits[:, :n].contiguous(), bitsV=bits[:, :n].contiguous())
    st = qaq.qaq_cache_stats(cache)
    assert st.device_status == 0 and st.tokens == T
    step = (rows.float().max(1).values - rows.float().min(1).values)[:, None] / 256
    for n_q in (1, 4):
        q = torch.zeros((BH, n_q, D), dtype=torch.float16, device="cuda")
        out = qaq.qaq_decode_attention_multi(cache, q, 1 / math.sqrt(D)).cpu()
        for j in range(n_q):
            off = ((out[:, j] - rows.float()).abs() / step).max().item()
            assert off <= 0.51, (n_q, j, off)


@pytest.mark.parametrize("tokens", [1, 100, 300])
def test_a_reset_cache_gives_the_bits_of_a_fresh_one(tokens):
    # the open tile of the second filling has places for tokens that the first one filled with values a thousand times larger
    wl = synth.scaled(synth.CONFIGS["C2"], heads=3, tokens=tokens, alpha=0.05)
    K, V, q, ring, nv = make_inputs(wl)
    pol = qaq.qaq_policy_from_hyper(*HYPER, 320)
    cfg, fresh, thr, out, scores, dev = gpu_pipeline(wl, K, V, q, ring, nv, pol, max_tokens=320)
    used = qaq.Cache(cfg)
    big = [torch.cat([x] * (320 // tokens + 1), dim=2)[:, :, :320].mul(1000).clamp(-60000, 60000).contiguous() for x in dev[:2]]
    wide = torch.full((wl.bh, 320), 8, dtype=torch.uint8, device="cuda")
    qaq.qaq_quantize_append(used, *big, qaq.qaq_outlier_thresholds(cfg, *big), bitsK=wide, bitsV=wide)
    used.reset()
    qaq.qaq_quantize_append(used, dev[0], dev[1], thr, policy=pol, ring=dev[3], nvalid=dev[4])
    row = torch.empty_like(scores)
    assert torch.equal(qaq.qaq_decode_attention(used, dev[2], 1 / math.sqrt(wl.head_dim), scores_out=row), out)
    assert torch.equal(row, scores)
    q4 = torch.stack([synth.make_query(wl, step=i).view(wl.bh, -1) for i in range(4)], dim=1).cuda().contiguous()
    a, b = (qaq.qaq_decode_attention_multi(c, q4, 1 / math.sqrt(wl.head_dim)) for c in (fresh, used))
    assert torch.equal(a, b)


@pytest.mark.parametrize("D", [32, 64, 128])
@pytest.mark.parametrize("beside", [2000.0, math.inf, math.nan])
def test_a_query_gives_what_it_gives_alone_whatever_is_beside_it(D, beside):
    wl = synth.scaled(synth.CONFIGS["C2"], heads=3, head_dim=D, tokens=700, alpha=0.05)
    K, V, q, ring, nv = make_inputs(wl)
    pol = qaq.qaq_policy_from_hyper(*HYPER, 700)
    cfg, cache, thr, out, scores, dev = gpu_pipeline(wl, K, V, q, ring, nv, pol)
    one = dev[2].view(wl.bh, D)
    for n_q in (2, 4, 8):
        qs = torch.stack([synth.make_query(wl, step=i).view(wl.bh, D) for i in range(n_q)], dim=1).cuda()
        qs[:, 1] = (qs[:, 1] * beside).half()
        qs[:, 0] = one
        got = qaq.qaq_decode_attention_multi(cache, qs.contiguous(), 1 / math.sqrt(D))[:, 0]
        # the same integer products, key corrections and weights; the accumulators are emptied at other tiles (11 of them), so
        # binary32 sums differ in their order
        assert (got - out).abs().max().item() <= 11 * 2.0 ** -22 * V.abs().max().item()


@pytest.mark.parametrize("n_q", [1, 2, 4])
def test_a_token_whose_logit_is_not_a_number_takes_no_part(n_q):
    # keys with infinities of both signs that are no outliers have no midpoint; the result is that of the other tokens
    D, BH, T = 64, 3, 210
    g = torch.Generator().manual_seed(1)
    K, V = (torch.randn((1, BH, T, D), generator=g).half() for _ in range(2))
    lost = torch.zeros(T, dtype=torch.bool)
    lost[[0, 7, 63, 64, 140, 141, 209]] = True
    K[:, :, lost, 5] = math.inf
    K[:, :, lost, 9] = -math.inf
    cfg = qaq.make_config(1, BH, D, T, 1, 8, 1, 0.0)
    thr = torch.tensor([-math.inf, math.inf] * 2).repeat(BH, 1).cuda().contiguous()
    q = torch.randn((BH, n_q, D), generator=g).half().cuda()
    outs = []
    for keep in (torch.ones(T, dtype=torch.bool), ~lost):
        cache, n = qaq.Cache(cfg), int(keep.sum())
        bits = torch.full((BH, n), 5, dtype=torch.uint8, device="cuda")
        qaq.qaq_quantize_append(cache, K[:, :, keep].cuda().contiguous(), V[:, :, keep].cuda().contiguous(), thr, bitsK=bits, bitsV=bits)
        outs.append(qaq.qaq_decode_attention_multi(cache, q, 1 / math.sqrt(D)))
    # the same tokens in other tiles: binary32 sums of 210 weights in another order, weights of 21 bits or more
    assert (outs[0] - outs[1]).abs().max().item() <= 210 * 2.0 ** -22 * V.abs().max().item()


@pytest.mark.parametrize("n_q", [3, 4, 5, 6, 7])
@pytest.mark.parametrize("D,alpha,scale", [(128, 0.1, 1.0), (128, 0.3, 1.0), (64, 0.5, 300.0)])
def test_several_queries_where_many_entries_are_outliers(n_q, D, alpha, scale):
    # two at a time or four, value outliers that are not staged (or too large for one word) in two words for two queries at once
    wl = synth.scaled(synth.CONFIGS["C2"], heads=3, head_dim=D, tokens=300, alpha=alpha)
    K, V, q, ring, nv = make_inputs(wl)
    K, V = (K * scale).half(), (V * scale).half()
    pol = qaq.qaq_policy_from_hyper(*HYPER, 300)
    bits = torch.full((wl.bh, 300), 8, dtype=torch.uint8)
    cfg, cache, thr, out, scores, dev = gpu_pipeline(wl, K, V, q, ring, nv, pol, bits=(bits, bits), max_outliers=300 * D)
    qs = torch.stack([synth.make_query(wl, step=i).view(wl.bh, D) for i in range(n_q)], dim=1).cuda() / scale
    got = qaq.qaq_decode_attention_multi(cache, qs.half().contiguous(), 1 / math.sqrt(D))
    for j in range(n_q):
        one = qaq.qaq_decode_attention(cache, qs[:, j].half().contiguous(), 1 / math.sqrt(D))
        # One word: units of 2^-24 of at most four times the largest term, D terms to a logit.  Two words: the same words for all
        # queries.  Beyond that binary32 sums of up to 128 terms in another order.
        terms = D * 2.0 ** -22 * (qs.abs().max() * K.abs().max()).item() / math.sqrt(D)
        assert (got[:, j] - one).abs().max().item() <= (2 * terms + 128 * 2.0 ** -23) * V.abs().max().item()


@pytest.mark.parametrize("heads,tokens,n_q", [(2, 100, 1), (3, 2100, 4), (14, 2100, 1), (14, 2100, 7), (200, 1000, 2)])
def test_an_infinite_logit_gives_zeros_however_the_sequence_is_split(heads, tokens, n_q):
    # one CTA, clusters, partials merged through memory: a key with an infinity that is no outlier has an infinite logit here
    D = 128
    g = torch.Generator().manual_seed(heads)
    K, V = (torch.randn((1, heads, tokens, D), generator=g).half() for _ in range(2))
    K[:, 0, tokens // 3, 5] = math.inf
    cfg = qaq.make_config(1, heads, D, tokens, 1, 8, 1, 0.0)
    thr = torch.tensor([-math.inf, math.inf] * 2).repeat(heads, 1).cuda().contiguous()
    cache = qaq.Cache(cfg)
    bits = torch.full((heads, tokens), 4, dtype=torch.uint8, device="cuda")
    qaq.qaq_quantize_append(cache, K.cuda(), V.cuda(), thr, bitsK=bits, bitsV=bits)
    out = qaq.qaq_decode_attention_multi(cache, torch.rand((heads, n_q, D), generator=g).half().cuda(), 1 / math.sqrt(D))
    assert (out[0] == 0).all() and torch.isfinite(out).all() and (out[1:] != 0).any(dim=2).all()


@pytest.mark.parametrize("D", [32, 64, 128])
@pytest.mark.parametrize("where", ["old", "new", "outlier", "none"])
def test_the_largest_value_of_a_tile_that_is_built_in_steps(D, where):
    # what decides between one and two words per outlier sum is kept with the tile: appended, lowered and raised, a tile gives what
    # the oracle gives for the final cache, wherever its values beyond 128 are (a token of the first append, of the second, an outlier only)
    wl = synth.scaled(synth.CONFIGS["C2"], heads=2, head_dim=D, tokens=150, alpha=0.05)
    K, V, q, ring, nv = make_inputs(wl)
    if where in ("old", "new"):
        t = 130 if where == "old" else 145
        K[:, :, t] *= 400; V[:, :, t] *= 400
    if where == "outlier":
        K[:, :, 133, 7] = 3000.0; V[:, :, 133, 9] = -3000.0
    cfg = qaq.make_config(wl.batch, wl.heads, D, 400, 2, 8, wl.window, wl.alpha)      # room for the tiles that grow again
    Kd, Vd, qd = K.cuda(), V.cuda(), q.cuda()
    thr = qaq.qaq_outlier_thresholds(cfg, Kd[:, :, :129], Vd[:, :, :129])
    cache = qaq.Cache(cfg)
    high = torch.full((wl.bh, 150), 6, dtype=torch.uint8, device="cuda")
    for a, b in ((0, 129), (129, 140), (140, 150)):
        bits = high[:, a:b].contiguous()
        qaq.qaq_quantize_append(cache, Kd[:, :, a:b], Vd[:, :, a:b], thr, bitsK=bits, bitsV=bits)
    low = torch.where(torch.arange(150, device="cuda") % 3 == 0, 3, 6).to(torch.uint8).repeat(wl.bh, 1).contiguous()
    qaq.qaq_requantize_down(cache, bitsK=low, bitsV=low)
    th = thr.cpu().numpy()
    u = lambda x: u16(x).reshape(wl.bh, 150, D)
    for bits in (low, high):
        if bits is high:
            qaq.qaq_requantize(cache, Kd, Vd, thr, bitsK=high, bitsV=high)
        out = qaq.qaq_decode_attention(cache, qd, 1 / math.sqrt(D)).cpu().numpy()
        assert qaq.qaq_cache_stats(cache).device_status == 0
        for bh in range(wl.bh):
            b = bits[bh].cpu().numpy()
            k = oracle.quantize(u(K)[bh], th[bh, 0], th[bh, 1], b)
            v = oracle.quantize(u(V)[bh], th[bh, 2], th[bh, 3], b)
            want, _ = oracle.decode(u16(q).reshape(wl.bh, D)[bh], k, v, 1 / math.sqrt(D))
            assert_attention_close(out[bh], want)
