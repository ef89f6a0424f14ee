"""Preprocessing launches whose CTAs take every pass in turn against launches whose CTAs belong to one pass:
the bundle of a call whose heads go through in groups of three does not differ in one byte."""
import pytest
import torch

import paper_2609_15810_b200 as vc
from paper_2609_15810_b200.binding import Params, alloc_buffers

pytestmark = pytest.mark.gpu

N, GRID = 333, (3, 3, 37)             # three blocks, the last one ragged
TUNED, OTHER = 80, 16                 # items per CTA behind which the CTAs take turns


def _bundle(p, q, k, v, perm, stats=None):
    quant, work = alloc_buffers(p)
    quant.zero_()
    if stats is None:
        vc.vc_prep(p, q, k, v, perm, quant, work)
    else:
        vc.vc_prep_with_stats(p, q, k, v, perm, *stats, quant, work)
    vc.vc_poll_status(work)
    return quant, work


@pytest.mark.parametrize("more", [0, 1, 5])          # heads beyond the last call with shares
@pytest.mark.parametrize("bits,p_format,flags,limit,passes", [
    (8, vc.VC_P_DEFAULT, vc.VC_FLAG_ALL, TUNED, 3),
    (8, vc.VC_P_DEFAULT, vc.VC_FLAG_ALL | vc.VC_FLAG_INT8_QK, TUNED, 2),
    (8, vc.VC_P_DEFAULT, vc.VC_FLAG_ALL & ~vc.VC_FLAG_ROPE, TUNED, 3),
    (8, vc.VC_P_DEFAULT, vc.VC_FLAG_ALL & ~vc.VC_FLAG_K_SMOOTH, OTHER, 2),
    (4, vc.VC_P_DEFAULT, vc.VC_FLAG_ALL, OTHER, 3),
    (4, vc.VC_P_EXPCAST_E4M3, vc.VC_FLAG_ALL, OTHER, 2)])
@pytest.mark.parametrize("d", [64, 128])
def test_bundle_does_not_depend_on_who_takes_the_items(d, bits, p_format, flags, limit, passes, more):
    if d == 64:
        limit = OTHER
    ctas = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    H = limit * ctas // (3 * passes) + more
    g = torch.Generator(device="cuda").manual_seed(H)
    q, k, v = [torch.randn(1, H, N, d, generator=g, device="cuda", dtype=torch.bfloat16) for _ in range(3)]
    k += 2 * torch.randn(1, H, 1, d, generator=g, device="cuda", dtype=torch.bfloat16)
    perm = torch.argsort(torch.rand(1, H, N, generator=g, device="cuda"), dim=-1).int()
    make = lambda **kw: Params.make(1, H, N, d, GRID, bits=bits, p_format=p_format, flags=flags, **kw)
    whole, work = _bundle(make(), q, k, v, perm)
    assert torch.equal(whole, _bundle(make(heads_per_pass=3), q, k, v, perm)[0])
    if bits == 8 and not more:
        stats = [t.clone() for t in vc.vc_prep_stats_view(make(), whole, work)]
        assert torch.equal(whole, _bundle(make(), q, k, v, perm, stats)[0])
