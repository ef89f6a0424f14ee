"""CTAs with one query tile against CTAs with two: the same arithmetic in the same order, so a head's
output does not depend on how many heads share the launch (which decides who gets a pair), bit for bit."""
import pytest
import torch

import paper_2609_15810_b200 as vc
from paper_2609_15810_b200.binding import Params, alloc_buffers

pytestmark = pytest.mark.gpu

FORMATS = {"fp8": (8, vc.VC_P_DEFAULT, 0), "int8qk": (8, vc.VC_P_DEFAULT, vc.VC_FLAG_INT8_QK),
           "nvfp4": (4, vc.VC_P_DEFAULT, 0), "hybrid": (4, vc.VC_P_EXPCAST_E4M3, 0)}


def _attn(q, k, v, grid, fmt, smooth):
    bits, pf, flags = FORMATS[fmt]
    flags |= vc.VC_FLAG_ALL if smooth else vc.VC_FLAG_ALL & ~vc.VC_FLAG_V_SMOOTH
    B, H, N, d = q.shape
    p = Params.make(B, H, N, d, grid, bits=bits, p_format=pf, flags=flags)
    quant, work = alloc_buffers(p)
    o = torch.empty_like(q)
    vc.vc_attn(p, q, k, v, None, o, quant, work)
    vc.vc_poll_status(work)
    return o


@pytest.mark.parametrize("smooth", [True, False])
@pytest.mark.parametrize("fmt", list(FORMATS))
@pytest.mark.parametrize("N,grid,d,H", [(300, (3, 10, 10), 128, 160),    # 3 tiles: every second pair is half empty
                                        (512, (2, 16, 16), 64, 84),      # 168 pairs: whole waves and 20 pairs behind
                                        (129, (1, 3, 43), 128, 75),      # 2 tiles, the last wave more than half full
                                        (1153, (1, 1, 1153), 64, 20)])   # 10 tiles: every buffer several times
def test_output_does_not_depend_on_the_split(N, grid, d, H, fmt, smooth):
    g = torch.Generator(device="cuda").manual_seed(N + H)
    q, k, v = [torch.randn(1, H, N, d, generator=g, device="cuda").bfloat16() for _ in range(3)]
    k += 2 * torch.randn(1, H, 1, d, generator=g, device="cuda").bfloat16()
    many = _attn(q, k, v, grid, fmt, smooth)
    for h in (0, H // 2, H - 2, H - 1):
        alone = _attn(*[t[:, h:h + 1].contiguous() for t in (q, k, v)], grid, fmt, smooth)
        assert torch.equal(many[:, h:h + 1], alone), h


@pytest.mark.parametrize("fmt", list(FORMATS))
@pytest.mark.parametrize("N,grid,d,H", [(4096, (4, 32, 32), 64, 32), (4096, (4, 32, 32), 128, 32), (2048, (2, 32, 32), 64, 8)])
def test_calls_without_value_smoothing_are_repeatable(N, grid, d, H, fmt):
    """Without block means the correction warps skip their waits for products; the output must still wait for the last.
    (A repeated call cannot show an order that is only likely: tests/test_handoff_order.py goes through all of them.)"""
    g = torch.Generator(device="cuda").manual_seed(N + d)
    q, k, v = [torch.randn(1, H, N, d, generator=g, device="cuda").bfloat16() for _ in range(3)]
    first = _attn(q, k, v, grid, fmt, False)
    for _ in range(5):
        assert torch.equal(_attn(q, k, v, grid, fmt, False), first)


@pytest.mark.parametrize("moving", [0, 3])
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("fmt", list(FORMATS))
def test_one_warp_rescales_at_every_key_tile_and_the_others_never(fmt, d, moving):
    """Scores that grow by about a factor of two per key tile for the 32 rows of one warp and fall for the rows of
    the others: without block means the others hand over at once while that warp still rescales.  One head alone
    (one query tile per CTA) against 37 copies of it (296 pairs of tiles: whole waves on 148 SMs), bit for bit.
    (No order of events can be forced here; tests/test_handoff_order.py goes through all of them.)"""
    nb = 16
    N, copies = 128 * nb, 37
    bits, pf, extra = FORMATS[fmt]
    g = torch.Generator(device="cuda").manual_seed(d + moving)
    q, k, v = [torch.randn(1, 1, N, d, generator=g, device="cuda") for _ in range(3)]
    rows = torch.arange(N, device="cuda")
    sign = torch.where((rows // 32) % 4 == moving, 1.0, -1.0)
    q, k = 0.05 * q, 0.05 * k
    q[..., 0] += 4.0 * sign
    k[..., 0] += (rows // 128 + 1) * (0.6931 * d ** 0.5 / 4.0)       # log2 of exp(q k / sqrt(d)) moves by one per tile
    q, k, v = [t.bfloat16() for t in (q, k, v)]

    def attn(heads):
        p = Params.make(1, heads, N, d, (1, 1, N), bits=bits, p_format=pf, flags=extra)
        quant, work = alloc_buffers(p)
        o = torch.empty(1, heads, N, d, dtype=torch.bfloat16, device="cuda")
        vc.vc_attn(p, *[t.expand(1, heads, N, d).contiguous() for t in (q, k, v)], None, o, quant, work)
        vc.vc_poll_status(work)
        return o

    pairs = attn(copies)
    assert torch.equal(pairs, pairs[:, :1].expand_as(pairs))
    for _ in range(10):
        assert torch.equal(attn(1), pairs[:, :1])
    ref = torch.softmax((q.double() @ k.double().transpose(-1, -2)) / d ** 0.5, dim=-1) @ v.double()
    assert torch.nn.functional.cosine_similarity(pairs[0, 0].double().flatten(), ref.flatten(), dim=0) > (0.999 if bits == 8 else 0.98)
