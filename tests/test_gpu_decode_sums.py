"""GPU checks of what the decode kernels sum in integers."""
import math

import pytest
import torch

from paper_2403_04643_b200 import qaq

pytestmark = pytest.mark.gpu


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
