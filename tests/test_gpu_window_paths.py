"""Score window after a prefill (Section 4.2): each way it is computed - few tiles (one CTA or a cluster per (b,h)), one pass of
resident CTAs, two passes over chunks - at the edges of tiles and of the sizes the ways divide at, against the oracle's causal
softmax rows.  Bound of a row: 1e-6 + 1e-2 of the entry, as everywhere for scores (the logits differ by binary32 sums of 128 products)."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2403_04643_b200 import qaq, synth

from gpu_helpers import make_inputs, u16

pytestmark = pytest.mark.gpu


def rows_match(K, Q, heads, which):
    B, H, T, D = K.shape
    n, scale = Q.shape[1], 1.0 / math.sqrt(D)
    cfg = qaq.make_config(B, heads, D, T, 2, 8, n, 0.01)
    ring, nvalid = qaq.qaq_prefill_window(cfg, Q.cuda(), K, scale)
    ring, nvalid = ring.view(B * H, n, T), nvalid.view(B * H, T)
    for bh in which:
        want, nv, _ = oracle.prefill_window(u16(Q[bh]), u16(K[bh // H, bh % H]), scale)
        got = ring[bh].cpu().numpy().astype(np.float64)
        assert np.array_equal(nvalid[bh].cpu().numpy(), nv)
        assert np.all(got[want == 0] == 0)
        assert np.all(np.abs(got - want) <= 1e-6 + 1e-2 * want), (bh, np.abs(got - want).max())
    return ring


def keys(B, H, T, D, token_major, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    K = torch.randn((B, T, H, D) if token_major else (B, H, T, D), generator=g, device="cuda").half()
    return K.transpose(1, 2) if token_major else K


@pytest.mark.parametrize("D", [32, 64, 128])
@pytest.mark.parametrize("heads,T,n", [
    (2, 1, 1), (2, 127, 16), (2, 129, 17), (3, 1024, 33),           # few tiles: clusters of one-tile CTAs
    (320, 128, 32), (110, 300, 5), (160, 385, 64), (320, 512, 17),  # a (b,h) to a CTA, in turn too
    (80, 512, 64), (32, 1025, 32), (24, 1793, 64), (12, 3969, 32),  # clusters of CTAs of two to four tiles, the last of them empty
    (40, 600, 16), (24, 1281, 5), (64, 1921, 1), (32, 4097, 16), (9, 8190, 16),      # up to 16 rows: two tiles to a group of warps
    (160, 640, 1), (300, 640, 33), (100, 1025, 64), (9, 2048, 16), (5, 4097, 32), (3, 8191, 64),   # one pass, clusters of several sizes
    (256, 2000, 64), (160, 1700, 32), (70, 8100, 64), (96, 5000, 16),                # one pass, several (b,h) per cluster
    (2, 8193, 64), (2, 16385, 32), (2, 33000, 16), (1, 9000, 5),    # two passes
    (24, 8193, 64), (20, 16400, 17),                                # two passes, several chunks of a CTA
    (96, 8193, 64),                                                 # two passes, chunks of more than four tiles
])
def test_window_rows_of_every_way(D, heads, T, n):
    K = keys(1, heads, T, D, token_major=heads % 2 == 1, seed=D + T)
    Q = torch.randn((heads, n, D), generator=torch.Generator().manual_seed(n)).half()
    ring = rows_match(K, Q, heads, {0, heads // 2, heads - 1})
    seen = min(n, T)                                                # queries that exist: their rows come first
    assert torch.allclose(ring[:, :seen].sum(2), torch.ones(heads, seen, device="cuda"), atol=1e-4) and (ring[:, seen:] == 0).all()


@pytest.mark.parametrize("T,n", [(700, 40), (4100, 32), (8200, 64)])
def test_a_reference_far_below_a_later_logit(T, n):
    # the logits of the first tiles are near zero, those of later tokens beyond 2^64 times their exponentials
    K = keys(2, 2, T, 64, token_major=False, seed=T) * 0.01
    K[:, :, T - T // 3:] *= 3000.0
    Q = torch.randn((4, n, 64), generator=torch.Generator().manual_seed(n)).half() * 4
    ring = rows_match(K, Q, 2, range(4))
    assert torch.allclose(ring.sum(2), torch.ones(4, n, device="cuda"), atol=1e-4)


@pytest.mark.parametrize("T", [100, 1500, 9000])
@pytest.mark.parametrize("n", [8, 40])
def test_heads_that_share_keys_and_keys_that_are_not_numbers(T, n):
    # one set of keys under several heads by a stride of zero; NaNs stay in their tokens and rows, the other tokens of the rows become 0,
    # whether one token is not a number or most of them, to the edge of a warp's 32
    K = keys(1, 1, T, 128, token_major=False, seed=T)
    Q = torch.randn((3, n, 128), generator=torch.Generator().manual_seed(1)).half()
    shared = rows_match(K.expand(1, 3, T, 128), Q, 3, range(3))
    assert shared.sum() > 0
    cfg = qaq.make_config(1, 3, 128, T, 2, 8, n, 0.01)
    for none in (slice(T // 2, T // 2 + 1), slice(0, T - n - 10), slice(0, (T - n - 1) // 32 * 32)):
        bad = K.clone()
        bad[0, 0, none, 5] = math.nan
        ring, _ = qaq.qaq_prefill_window(cfg, Q.cuda(), bad.expand(1, 3, T, 128), 1 / math.sqrt(128))
        ring = ring.view(3, n, T)
        assert torch.isnan(ring[:, :, none]).all()
        ring[:, :, none] = 0
        assert (ring == 0).all()


@pytest.mark.parametrize("D", [32, 64, 128])
@pytest.mark.parametrize("heads,T,n", [(2, 100, 5), (2, 700, 33), (300, 400, 16), (3, 1500, 16), (2, 3000, 32), (160, 1700, 32), (2, 4100, 64), (2, 9000, 64)])
def test_logits_of_minus_infinity(D, heads, T, n):
    # the first two thirds of the tokens have logits of -inf in every row, the others are far below zero: entries of 0, and rows that
    # are normalised over the rest (logits of about -1000, whose binary32 sums are off by 2^-24 of 8000 a few times: 1e-3 of an entry)
    K = keys(1, heads, T, D, token_major=False, seed=T)
    K[..., 0] = -1000.0
    K[:, :, :2 * T // 3, 0] = -math.inf
    Q = torch.randn((heads, n, D), generator=torch.Generator().manual_seed(n)).half()
    Q[..., 0] = math.sqrt(D)
    ring = rows_match(K, Q, heads, {0, heads - 1})
    assert torch.allclose(ring.sum(2), torch.ones(heads, n, device="cuda"), atol=1e-4)


LOST = torch.tensor([0x7F7E105E], dtype=torch.int32).view(torch.float32)      # QAQ_SCORE_LOST


@pytest.mark.parametrize("D", [32, 128])
@pytest.mark.parametrize("W", [5, 40])
@pytest.mark.parametrize("how", ["tiles", "open", "select", "lower", "raise"])
def test_a_lost_window_is_reported_by_the_calls_that_take_it(D, W, how):
    # what a window kernel whose wait ran out leaves in the rows of its tokens: their values take bits_max and the device status says so,
    # nothing else changes; a window without a number for another reason is not reported
    wl = synth.scaled(synth.CONFIGS["C2"], heads=2, head_dim=D, tokens=150, window=W)
    K, V, q, ring, nv = (t.cuda() for t in make_inputs(wl))
    nan, lost = ring.clone(), ring.clone()
    nan[..., 70:90] = math.nan
    lost[..., 70:90] = LOST.cuda()
    if how == "open":
        nan[..., 149] = math.nan
        lost[..., 149] = LOST.cuda()
    pol = qaq.qaq_policy_from_hyper(0.006, 0.03, 64.0, 150)
    cfg = qaq.make_config(wl.batch, wl.heads, D, 400, 2, 8, W, wl.alpha)
    thr = qaq.qaq_outlier_thresholds(cfg, K, V)

    def widths(r):
        if how == "select":
            return *qaq.qaq_select_bits(cfg, pol, K, V, r, nv, thr), None
        cache = qaq.Cache(cfg)
        if how == "open":
            for a, b in ((0, 149), (149, 150)):
                qaq.qaq_quantize_append(cache, K[:, :, a:b], V[:, :, a:b], thr, policy=pol, ring=r[..., a:b].contiguous(), nvalid=nv[..., a:b].contiguous())
        elif how == "tiles":
            qaq.qaq_quantize_append(cache, K, V, thr, policy=pol, ring=r, nvalid=nv)
        else:
            bits = torch.full((wl.bh, 150), 8 if how == "lower" else 1, dtype=torch.uint8, device="cuda")
            qaq.qaq_quantize_append(cache, K, V, thr, bitsK=bits, bitsV=bits)
            if how == "lower":
                qaq.qaq_requantize_down(cache, policy=pol, ring=r, nvalid=nv)
            else:
                qaq.qaq_requantize(cache, K, V, thr, policy=pol, ring=r, nvalid=nv)
        return *(qaq.qaq_cache_export(cache, x)["bits"] for x in (0, 1)), qaq.qaq_cache_stats(cache).device_status

    k0, v0, s0 = widths(nan)
    k1, v1, s1 = widths(lost)
    there = (lost < 2).all(dim=2).view(wl.bh, 150)
    assert torch.equal(k0, k1) and torch.equal(v0[there], v1[there])
    assert (v0[~there] == 2).all() and (v1[~there] == 8).all()
    assert how == "select" or (s0, s1) == (qaq.QAQ_OK, 4)


def laid_out(X, how):
    """The values of X [B,H,T,D] with other strides (elements; 16-byte aligned rows, as the calls ask for)."""
    B, H, T, D = X.shape
    big = {
        "padded rows": lambda: torch.empty((B, H, T, D + 8), dtype=X.dtype, device=X.device)[..., :D],
        "gap between heads": lambda: torch.empty((B, H, T * D + 24), dtype=X.dtype, device=X.device).as_strided((B, H, T, D), (H * (T * D + 24), T * D + 24, D, 1)),
        "slice": lambda: torch.empty((B, H, T + 40, D), dtype=X.dtype, device=X.device)[:, :, 7:7 + T],
        "some of many heads": lambda: torch.empty((B, T, H + 3, D), dtype=X.dtype, device=X.device)[:, :, 2:2 + H].transpose(1, 2),
        "batch inside": lambda: torch.empty((H, T, B, D), dtype=X.dtype, device=X.device).permute(2, 0, 1, 3),
    }[how]()
    big.copy_(X)
    return big


@pytest.mark.parametrize("D", [32, 64, 128])
@pytest.mark.parametrize("how", ["padded rows", "gap between heads", "slice", "some of many heads", "batch inside"])
@pytest.mark.parametrize("T,n", [(300, 9), (3000, 16), (4100, 64), (9000, 64)])
def test_keys_of_any_strides(D, how, T, n):
    # few tiles with one and with several tiles to a CTA, one pass, two passes: the copies of tiles take the caller's strides
    K = laid_out(keys(2, 2, T, D, token_major=False, seed=T), how)
    Q = torch.randn((4, n, D), generator=torch.Generator().manual_seed(n)).half()
    rows_match(K, Q, 2, range(4))
