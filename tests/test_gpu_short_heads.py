"""vc_attn on short heads: one preprocessing launch whose clusters hold a head's blocks in shared memory.  The bundle is
the one vc_prep writes with its launch per phase, byte for byte, and the output is the one vc_attn_fwd makes of it."""
import pytest
import torch

import paper_2609_15810_b200 as vc
from paper_2609_15810_b200.binding import Params, alloc_buffers

pytestmark = pytest.mark.gpu

ALL = vc.VC_FLAG_ALL
FORMATS = [(8, vc.VC_P_DEFAULT, ALL), (8, vc.VC_P_DEFAULT, ALL | vc.VC_FLAG_INT8_QK), (4, vc.VC_P_DEFAULT, ALL), (4, vc.VC_P_EXPCAST_E4M3, ALL),
           (8, vc.VC_P_DEFAULT, ALL & ~vc.VC_FLAG_K_SMOOTH), (8, vc.VC_P_DEFAULT, ALL & ~vc.VC_FLAG_V_SMOOTH),
           (4, vc.VC_P_DEFAULT, ALL & ~vc.VC_FLAG_K_SMOOTH), (4, vc.VC_P_EXPCAST_E4M3, ALL & ~vc.VC_FLAG_V_SMOOTH)]


# one block up to sixteen, ragged and whole; clusters of one, two, four and eight, one and two blocks a CTA, and a CTA
# whose second block is missing; one token; tables just within and just beyond the limit; a head too many blocks long
@pytest.mark.parametrize("grid", [(1, 1, 1), (2, 10, 10), (2, 8, 8), (3, 7, 17), (4, 8, 16), (5, 7, 23), (4, 16, 16), (3, 19, 18), (5, 17, 23),
                                  (8, 16, 16), (2, 3, 62), (2, 2, 64), (4, 16, 33)])
@pytest.mark.parametrize("bits,p_format,flags", FORMATS)
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("perm_kind,token_major", [("random", False), (None, True)])
def test_same_bundle_and_output(grid, bits, p_format, flags, d, perm_kind, token_major):
    B, H, N = 2, 3, grid[0] * grid[1] * grid[2]
    g = torch.Generator(device="cuda").manual_seed(N + d)
    q, k, v = [torch.randn(B, N, H, d, generator=g, device="cuda", dtype=torch.bfloat16).transpose(1, 2) for _ in range(3)]
    k += 2 * torch.randn(1, H, 1, d, generator=g, device="cuda", dtype=torch.bfloat16)
    if not token_major:
        q, k, v = [t.contiguous() for t in (q, k, v)]
    perm = torch.argsort(torch.rand(B, H, N, generator=g, device="cuda"), dim=-1).int() if perm_kind else None
    p = Params.make(B, H, N, d, grid, bits=bits, p_format=p_format, flags=flags, stride_b=v.stride(0), stride_h=v.stride(1), stride_n=v.stride(2))
    got, want = [], []
    for out, alone in ((got, False), (want, True)):
        quant, work = alloc_buffers(p)
        quant.zero_()
        work.fill_(0xff)
        o = torch.empty(B, H, N, d, dtype=torch.bfloat16, device="cuda")
        if alone:
            vc.vc_prep(p, q, k, v, perm, quant, work)
            vc.vc_attn_fwd(p, quant, o, work)
        else:
            vc.vc_attn(p, q, k, v, perm, o, quant, work)
        vc.vc_poll_status(work)
        out += [quant, o]
        if bits == 8:
            out += [t.clone() for t in vc.vc_prep_stats_view(p, quant, work)]
    for a, b in zip(got, want):
        assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))


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
