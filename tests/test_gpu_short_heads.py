"""vc_attn on short heads: one preprocessing launch whose clusters hold a head's blocks in shared memory, one block a CTA, up to
eight.  The bundle is the one vc_prep writes with its launch per phase, byte for byte, and the output is the one vc_attn_fwd makes of it."""
import pytest
import torch

import paper_2609_15810_b200 as vc
from paper_2609_15810_b200.binding import Params, alloc_buffers

pytestmark = pytest.mark.gpu

ALL = vc.VC_FLAG_ALL
FORMATS = [(8, vc.VC_P_DEFAULT, ALL), (8, vc.VC_P_DEFAULT, ALL | vc.VC_FLAG_INT8_QK), (4, vc.VC_P_DEFAULT, ALL), (4, vc.VC_P_EXPCAST_E4M3, ALL),
           (8, vc.VC_P_DEFAULT, ALL & ~vc.VC_FLAG_K_SMOOTH), (8, vc.VC_P_DEFAULT, ALL & ~vc.VC_FLAG_V_SMOOTH),
           (4, vc.VC_P_DEFAULT, ALL & ~vc.VC_FLAG_K_SMOOTH), (4, vc.VC_P_EXPCAST_E4M3, ALL & ~vc.VC_FLAG_V_SMOOTH)]


def _inputs(H, grid, d, perm, token_major, B=1):
    N = grid[0] * grid[1] * grid[2]
    g = torch.Generator(device="cuda").manual_seed(N + d + H)
    q, k, v = [torch.randn(B, N, H, d, generator=g, device="cuda", dtype=torch.bfloat16).transpose(1, 2) for _ in range(3)]
    k += 2 * torch.randn(1, H, 1, d, generator=g, device="cuda", dtype=torch.bfloat16)
    if not token_major:
        q, k, v = [t.contiguous() for t in (q, k, v)]
    return q, k, v, torch.argsort(torch.rand(B, H, N, generator=g, device="cuda"), dim=-1).int() if perm else None


def _params(q, grid, bits, p_format, flags, **kw):
    B, H, N, d = q.shape
    return Params.make(B, H, N, d, grid, bits=bits, p_format=p_format, flags=flags, stride_b=q.stride(0), stride_h=q.stride(1), stride_n=q.stride(2), **kw)


def _same_bundle_and_output(q, k, v, perm, p, short):
    """vc_attn against vc_prep and vc_attn_fwd; `short`: whether vc_attn takes its two launches."""
    got, want = [], []
    for out, alone in ((got, False), (want, True)):
        quant, work = alloc_buffers(p)
        quant.zero_()
        work.fill_(0xff)
        o = torch.empty(q.shape, dtype=torch.bfloat16, device="cuda")
        n0 = vc.vc_launch_count()
        if alone:
            vc.vc_prep(p, q, k, v, perm, quant, work)
            vc.vc_attn_fwd(p, quant, o, work)
        else:
            vc.vc_attn(p, q, k, v, perm, o, quant, work)
        assert (vc.vc_launch_count() - n0 == 2) == (short and not alone)
        vc.vc_poll_status(work)
        out += [quant, o]
        if p.bits == 8:
            out += [t.clone() for t in vc.vc_prep_stats_view(p, quant, work)]
    for a, b in zip(got, want):
        assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))


# one block up to eight, ragged and whole; one token
@pytest.mark.parametrize("grid", [(1, 1, 1), (2, 10, 10), (2, 8, 8), (3, 7, 17), (4, 8, 16), (4, 12, 12), (3, 16, 15), (5, 7, 23), (4, 16, 16)])
@pytest.mark.parametrize("bits,p_format,flags", FORMATS)
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("perm,token_major", [(True, False), (False, True)])
def test_same_bundle_and_output(grid, bits, p_format, flags, d, perm, token_major):
    q, k, v, pm = _inputs(3, grid, d, perm, token_major, B=2)
    _same_bundle_and_output(q, k, v, pm, _params(q, grid, bits, p_format, flags), True)


# rows wider than the head, heads and batches with gaps between them, other frequencies and another scale
@pytest.mark.parametrize("bits", [8, 4])
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("order", ["bhn", "bnh", "hbn"])
def test_other_strides_and_frequencies(bits, d, order):
    grid, sizes = (3, 7, 17), {"b": 2, "h": 3, "n": 357 + 5}
    g = torch.Generator(device="cuda").manual_seed(d)
    views = []
    for _ in range(3):
        full = torch.randn(*[sizes[c] for c in order], d + 24, generator=g, device="cuda", dtype=torch.bfloat16)
        views.append(full.permute(*[order.index(c) for c in "bhn"], 3)[:, :, :357, :d])
    perm = torch.argsort(torch.rand(2, 3, 357, generator=g, device="cuda"), dim=-1).int()
    p = _params(views[0], grid, bits, vc.VC_P_DEFAULT, ALL, rope_theta=500.0, softmax_scale=0.07)
    _same_bundle_and_output(*views, perm, p, True)


# RoPE tables of 1390 to 1408 entries, the largest that leave two CTAs on an SM (d128: 44 / 42 / 42 channels, d64: 24 / 20 / 20), and of
# 1409 and 1412, which take the launch per phase; a head of nine blocks, which takes it too
@pytest.mark.parametrize("d,grid,short", [(128, (1, 2, 64), True), (128, (2, 2, 62), True), (128, (2, 8, 56), True), (64, (4, 1, 135), True),
                                          (64, (1, 3, 136), True), (128, (2, 3, 62), False), (64, (1, 1, 139), False), (128, (5, 11, 19), False)])
@pytest.mark.parametrize("bits", [8, 4])
def test_largest_tables(d, grid, short, bits):
    q, k, v, pm = _inputs(6, grid, d, True, False)
    _same_bundle_and_output(q, k, v, pm, _params(q, grid, bits, vc.VC_P_DEFAULT, ALL), short)


# the most heads that take the one launch (8 bits: every CTA resident at once, two an SM; 4 bits: a second wave of clusters), and one more
@pytest.mark.parametrize("bits,waves", [(8, 1), (4, 2)])
@pytest.mark.parametrize("grid", [(4, 16, 16), (4, 12, 12), (2, 10, 10)])
@pytest.mark.parametrize("d", [64, 128])
def test_most_heads(bits, waves, grid, d):
    nb = (grid[0] * grid[1] * grid[2] + 127) // 128
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    most = 2 * waves * sms // (3 * nb)
    for H, short in ((most, True), (most + 1, False)):
        q, k, v, pm = _inputs(H, grid, d, True, False)
        _same_bundle_and_output(q, k, v, pm, _params(q, grid, bits, vc.VC_P_DEFAULT, ALL), short)


@pytest.mark.parametrize("bits", [8, 4])
def test_captured_and_on_two_streams(bits):
    """A captured call reads its inputs when it is replayed; calls on two streams, each with its own buffers, do not meet."""
    grid = (3, 16, 15)
    calls = []
    for H in (4, 5):
        q, k, v, pm = _inputs(H, grid, 128, True, False)
        p = _params(q, grid, bits, vc.VC_P_DEFAULT, ALL)
        calls.append((p, q, k, v, pm, torch.empty_like(q), *alloc_buffers(p)))
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    want = []
    for c in calls:
        vc.vc_attn(*c)
        want.append(c[5].clone())
    torch.cuda.synchronize()
    for c in calls:
        c[5].zero_()
    torch.cuda.synchronize()
    for _ in range(20):
        for c, s in zip(calls, streams):
            with torch.cuda.stream(s):
                vc.vc_attn(*c)
    torch.cuda.synchronize()
    for c, w in zip(calls, want):
        assert torch.equal(c[5], w)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=streams[0]):
        vc.vc_attn(*calls[0])
        vc.vc_attn(*calls[0])
    calls[0][1].copy_(calls[0][1].flip(2).contiguous())      # other queries than at capture
    calls[0][5].zero_()
    graph.replay()
    torch.cuda.synchronize()
    got = calls[0][5].clone()
    vc.vc_attn(*calls[0])
    vc.vc_poll_status(calls[0][7])
    assert torch.equal(got, calls[0][5]) and not torch.equal(got, want[0])


def test_one_launch_instead_of_four():
    p = Params.make(1, 2, 1024, 128, (4, 16, 16))
    q, k, v = [torch.randn(1, 2, 1024, 128, device="cuda", dtype=torch.bfloat16) for _ in range(3)]
    quant, work = alloc_buffers(p)
    n0 = vc.vc_launch_count()
    vc.vc_attn(p, q, k, v, None, torch.empty_like(q), quant, work)
    n1 = vc.vc_launch_count()
    vc.vc_prep(p, q, k, v, None, quant, work)
    torch.cuda.synchronize()
    assert n1 - n0 == 2 and vc.vc_launch_count() - n1 == 4
