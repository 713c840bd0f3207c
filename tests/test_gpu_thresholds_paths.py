"""Every path of qaq_outlier_thresholds (Section 4.2, "Outliers": order statistics at the alpha/2 tails) gives the exact
order statistic: inputs built so that the sample's bracket fails in each possible way."""
import numpy as np
import pytest
import torch

import oracle
from paper_2403_04643_b200 import qaq, synth

from gpu_helpers import u16

pytestmark = pytest.mark.gpu


def check(K, V, wl, alpha):
    cfg = qaq.make_config(wl.batch, wl.heads, wl.head_dim, K.shape[2], 2, 8, wl.window, alpha)
    thr = qaq.qaq_outlier_thresholds(cfg, K.cuda(), V.cuda()).cpu().numpy()
    Ku, Vu = u16(K).reshape(wl.bh, K.shape[2], wl.head_dim), u16(V).reshape(wl.bh, K.shape[2], wl.head_dim)
    for bh in range(wl.bh):
        want = np.array([*oracle.thresholds(Ku[bh], alpha), *oracle.thresholds(Vu[bh], alpha)], dtype=np.float32)
        assert np.array_equal(thr[bh], want), (bh, thr[bh], want)


def sampled_tokens(T):
    return [s * T // 64 for s in range(64)]      # the 64 tokens the bracket is taken from


def test_bracket_collapses_and_the_candidate_lists_overflow():
    # the sampled tokens are all zero: the bracket is [0, 0], every non-zero entry is a candidate, the lists overflow
    # and the problem is redone by the exact two-pass select over its data
    wl = synth.scaled(synth.CONFIGS["C2"], heads=3, tokens=4096)
    K, V = synth.make_kv(wl, 0)
    K[:, :, sampled_tokens(4096)] = 0
    V[:, :, sampled_tokens(4096)] = 0
    check(K, V, wl, wl.alpha)


def test_bracket_too_wide_to_hold_rank_k():
    # the sampled tokens are a hundred times larger than the rest: the bracket lies far outside the bulk and fewer
    # than k+1 entries fall beyond it
    wl = synth.scaled(synth.CONFIGS["C2"], heads=3, tokens=4096)
    K, V = synth.make_kv(wl, 0)
    K[:, :, sampled_tokens(4096)] *= 100
    V[:, :, sampled_tokens(4096)] *= 100
    check(K, V, wl, wl.alpha)


def test_more_candidates_than_the_select_kernel_keeps_on_chip():
    # alpha = 8 % of 4096 x 128 entries: about 40 thousand candidates per tail, above the 16384 keys held in shared
    # memory but inside the list: rank select over the list in global memory
    wl = synth.scaled(synth.CONFIGS["C2"], heads=2, tokens=4096)
    K, V = synth.make_kv(wl, 0)
    check(K, V, wl, 0.08)


def test_constant_tensor_and_single_distinct_tail_value():
    wl = synth.scaled(synth.CONFIGS["C2"], heads=2, tokens=1024)
    K, V = synth.make_kv(wl, 0)
    K[:] = 1.5                       # every entry equal: both thresholds are that value, no outliers
    V[:, :, :, ::2] = -2.0           # half of the entries tie at the lower tail
    check(K, V, wl, wl.alpha)


@pytest.mark.parametrize("alpha", [0.3, 0.5, 1.0])
def test_tails_so_heavy_that_most_entries_are_candidates(alpha):
    # a third of the entries (or more) beyond the bracket per tail: scan blocks of 64 tokens, whose lists hold them, and lists of
    # a problem that are longer than what the select keeps on chip (blocks that find more than they hold: the tests of tails
    # in one part of the sequence, and the collapsed bracket)
    wl = synth.scaled(synth.CONFIGS["C2"], heads=2, tokens=2048)
    K, V = synth.make_kv(wl, 0)
    check(K, V, wl, alpha)


@pytest.mark.parametrize("alpha", [0.01, 0.05])
@pytest.mark.parametrize("part,factor", [(4, 2.0), (4, 40.0), (16, 4.0), (64, 4.0)])
def test_tails_that_lie_in_one_part_of_the_sequence(alpha, part, factor):
    # the scan blocks of the first 1/part of the tokens find several times the candidates that their lists are laid out for:
    # what these do not hold goes to the problem's list
    wl = synth.scaled(synth.CONFIGS["C2"], heads=3, tokens=4096)
    K, V = synth.make_kv(wl, 0)
    K[:, :, :4096 // part] *= factor
    V[:, 1:, -4096 // part:] *= factor
    check(K, V, wl, alpha)


@pytest.mark.parametrize("D,T,alpha", [(128, 4096, 0.01), (64, 2049, 0.3), (32, 700, 1.0), (32, 2500, 1.0), (128, 4097, 0.2)])
def test_the_exact_select_over_the_data_passes_over_nans(D, T, alpha):
    # sampled tokens all zero: lists overflow (700 tokens of 32 channels: the kernel of short sequences, which samples nothing); NaNs of
    # both signs, infinities, a problem of NaNs alone in its unsampled tokens
    wl = synth.scaled(synth.CONFIGS["C2"], heads=3, head_dim=D, tokens=T)
    K, V = synth.make_kv(wl, 0)
    g = torch.Generator().manual_seed(D)
    for X in (K, V):
        m = torch.rand(X.shape, generator=g)
        X[m < 0.02] = float("nan"); X[(m > 0.02) & (m < 0.04)] = -float("nan")
        X[(m > 0.04) & (m < 0.041)] = float("inf"); X[(m > 0.041) & (m < 0.042)] = -float("inf")
    K[:, 2] = float("nan")
    K[:, :, sampled_tokens(T)] = 0
    V[:, :, sampled_tokens(T)] = 0
    check(K, V, wl, alpha)


@pytest.mark.parametrize("D,T,heads", [(32, 1, 3), (128, 33, 3), (128, 256, 3), (64, 512, 3), (128, 257, 3), (32, 2048, 3), (64, 1024, 3), (128, 513, 3),
                                       (32, 2049, 3), (64, 1025, 3), (32, 1024, 75), (32, 1025, 74), (32, 1025, 75), (128, 400, 75),
                                       (32, 2048, 8), (64, 768, 7), (64, 769, 7), (32, 1, 149), (128, 33, 149), (64, 64, 149), (32, 65, 149)])
@pytest.mark.parametrize("alpha", [0.0, 0.01, 0.3, 1.0])
def test_short_sequences(D, T, heads, alpha):
    # up to the keys that one CTA holds with 8 and with 16 pieces to a thread (these only up to 74 (b,h); up to 7 (b,h) 12 pieces), and one
    # token beyond; up to 64 tokens of more than 148 (b,h); ranks beyond the number of pieces (0.3, 1.0); NaNs of both signs, infinities, both zeros, a tail of ties
    wl = synth.scaled(synth.CONFIGS["C2"], heads=heads, head_dim=D, tokens=T)
    K, V = synth.make_kv(wl, 0)
    flat = V.view(-1)
    for i, x in enumerate((float("nan"), -float("nan"), float("inf"), -float("inf"), 0.0, -0.0)):
        flat[(i * 37 + 5) % D::D * 7] = x
    K[:, 0, :, D // 2:] = 3.0
    K[:, 1] = float("nan") if T < 40 else K[:, 1]
    check(K, V, wl, alpha)
