"""GPU checks of the code pools at their ends: what follows a tile that found no room."""
import math

import pytest
import torch

from paper_2403_04643_b200 import qaq

pytestmark = pytest.mark.gpu


def _pool(D, tokens):
    """Bytes of a (b,h) pool: per tile 64 tokens at 8 bits, a header of 16 bytes and room for six tokens."""
    return (-(-tokens // 64) * (16 + 64 * D + 6 * D + 32) + 256 + 255) // 256 * 256


# head_dim 32, pools of 9472 bytes; a tile of keys takes 16 + 4 * (sum of its widths) bytes, so an open tile seldom ends on a
# multiple of 16.  Closed tiles that are raised move behind each other to the end of the pool:
#   open tile of 63 tokens (2028 bytes): tile 0 to 8 bits, the open tile behind it (7196 of 9472), tile 1 to 6 bits (8764): the
#       open tile finds no room behind it.  The token that would complete it is lost, a narrow tile still fits.
#   open tile of one token (44 bytes), which follows every move: 8588 of 9472 at the end.  63 tokens of 8 bits that would complete
#       it find no room, a narrow tile behind them does.
@pytest.mark.parametrize("first,open_bits,moves,head", [
    (63, [8] * 62 + [7], [(8, 2), (8, 6)], [8]),
    (1, [7], [(8, 2), (8, 8), (2, 8), (8, 8), (8, 2), (8, 4)], [8] * 63),
])
def test_tiles_behind_an_open_tile_that_found_no_room(first, open_bits, moves, head):
    D, BH, T0 = 32, 2, 128
    T1 = T0 + first
    T2 = T1 + len(head) + 64
    assert T2 == 256 and _pool(D, T2) == 9472
    g = torch.Generator().manual_seed(first)
    K, V = (torch.randn((1, BH, T2, D), generator=g).half().cuda() for _ in range(2))
    thr = torch.tensor([-2.5, 2.5] * 2).repeat(BH, 1).cuda().contiguous()
    cfg = qaq.make_config(1, BH, D, T2, 1, 8, 1, 0.05)
    tb = lambda b: torch.tensor(b, dtype=torch.uint8).repeat(BH, 1).cuda().contiguous()
    cache = qaq.Cache(cfg)
    qaq.qaq_quantize_append(cache, K[:, :, :T1], V[:, :, :T1], thr, bitsK=tb([2] * T0 + open_bits), bitsV=tb([2] * T0 + open_bits))
    for a, b in moves:
        bits = tb([a] * 64 + [b] * 64 + open_bits)
        qaq.qaq_requantize(cache, K, V, thr, bitsK=bits, bitsV=bits)
    new = tb(head + [1] * 64)
    qaq.qaq_quantize_append(cache, K[:, :, T1:], V[:, :, T1:], thr, bitsK=new, bitsV=new)
    out = qaq.qaq_decode_attention(cache, torch.zeros((BH, D), dtype=torch.float16, device="cuda"), 1 / math.sqrt(D))
    st = qaq.qaq_cache_stats(cache)
    assert st.device_status == 3 and st.tokens == T2 and torch.isfinite(out).all()
    a, b = moves[-1]
    want = [a] * 64 + [b] * 64 + open_bits + [0] * len(head) + [1] * 64
    whole = qaq.Cache(cfg)
    full = tb([max(w, 1) for w in want])
    qaq.qaq_quantize_append(whole, K, V, thr, bitsK=full, bitsV=full)
    for x in range(2):
        got, ref = qaq.qaq_cache_export(cache, x), qaq.qaq_cache_export(whole, x)
        assert got["bits"].tolist() == [want] * BH
        for bh in range(BH):
            for t in range(T2):
                if want[t]:
                    i, j, n = int(got["off"][bh, t]), int(ref["off"][bh, t]), D * want[t] // 8
                    assert torch.equal(got["codes"][bh, i:i + n], ref["codes"][bh, j:j + n]), (x, bh, t)


def test_pool_use_between_the_steps_of_a_stream():
    # asked for between two one-token appends it leaves the count and its arrival counter alone: every token is where it belongs
    D, BH, T0, n = 64, 5, 60, 9
    g = torch.Generator().manual_seed(4)
    K, V = (torch.randn((1, BH, T0 + n, D), generator=g).half().cuda() for _ in range(2))
    thr = torch.tensor([-2.5, 2.5] * 2).repeat(BH, 1).cuda().contiguous()
    cfg = qaq.make_config(1, BH, D, T0 + n, 1, 8, 1, 0.05)
    bits = torch.randint(1, 9, (BH, T0 + n), generator=g, dtype=torch.uint8).cuda()
    one, whole = qaq.Cache(cfg), qaq.Cache(cfg)
    qaq.qaq_quantize_append(whole, K, V, thr, bitsK=bits, bitsV=bits)
    first = bits[:, :T0].contiguous()
    qaq.qaq_quantize_append(one, K[:, :, :T0], V[:, :, :T0], thr, bitsK=first, bitsV=first)
    qaq.qaq_stream_begin(one)
    for t in range(T0, T0 + n):
        b = bits[:, t:t + 1].contiguous()
        qaq.qaq_stream_append(one, K[:, :, t:t + 1], V[:, :, t:t + 1], thr, bitK=b, bitV=b)
        use = qaq.qaq_cache_pool_use(one)
        assert 0 < use[0] <= use[2] and 0 < use[1] <= use[2]
    assert qaq.qaq_stream_end(one) == T0 + n
    for x in range(2):
        a, b = qaq.qaq_cache_export(one, x), qaq.qaq_cache_export(whole, x)
        assert all(torch.equal(a[k], b[k]) for k in ("bits", "off", "codes", "rowptr", "ch"))
