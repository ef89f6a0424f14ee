"""Preprocessing launches whose CTAs take every pass in turn against launches whose CTAs belong to one pass:
the bundle of a call whose heads go through in groups of three does not differ in one byte."""
import pytest
import torch

import paper_2609_15810_b200 as vc
from paper_2609_15810_b200.binding import Params, alloc_buffers, section

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


@pytest.mark.parametrize("d,grid,H", [(128, (3, 37, 125), 3),       # a table of 3468 entries: just too long for two CTAs of the row pass on an SM
                                      (128, (3, 36, 125), 3),       # 3447: two fit
                                      (128, (2, 110, 170), 3),      # 5924: one of the column sums as well
                                      (64, (1, 300, 600), 1)])      # 9012: d64, one
@pytest.mark.parametrize("bits,p_format,flags", [(8, vc.VC_P_DEFAULT, vc.VC_FLAG_ALL), (8, vc.VC_P_DEFAULT, vc.VC_FLAG_ALL | vc.VC_FLAG_INT8_QK),
                                                 (4, vc.VC_P_DEFAULT, vc.VC_FLAG_ALL), (4, vc.VC_P_EXPCAST_E4M3, vc.VC_FLAG_ALL)])
def test_wide_grids(d, grid, H, bits, p_format, flags):
    """Around the table sizes where the passes over rows leave the shared launches: the bundle does not differ from
    one whose heads go through one by one, nor with the statistics supplied; the mean of K against doubles."""
    n = grid[0] * grid[1] * grid[2]
    g = torch.Generator(device="cuda").manual_seed(n)
    q, k, v = [torch.randn(1, H, n, d, generator=g, device="cuda", dtype=torch.bfloat16) for _ in range(3)]
    perm = torch.argsort(torch.rand(1, H, n, generator=g, device="cuda"), dim=-1).int()
    make = lambda **kw: Params.make(1, H, n, d, grid, bits=bits, p_format=p_format, flags=flags, **kw)
    whole, work = _bundle(make(), q, k, v, perm)
    assert torch.equal(whole, _bundle(make(heads_per_pass=1), q, k, v, perm)[0])
    side = 2 * (d // 6)
    dims, t = (d - 2 * side, side, side), torch.arange(n, device="cuda")
    pos = (t // (grid[1] * grid[2]), (t // grid[2]) % grid[1], t % grid[2])
    phi = torch.cat([pos[a].double()[:, None] * 10000.0 ** (-torch.arange(0, dims[a], 2, device="cuda").double() / dims[a]) for a in range(3)], dim=1)
    x, cos, sin = k[0, H - 1].double(), phi.cos(), phi.sin()
    mean = torch.stack([(x[:, 0::2] * cos - x[:, 1::2] * sin).mean(0), (x[:, 0::2] * sin + x[:, 1::2] * cos).mean(0)], dim=1).flatten()
    got = section(vc.vc_quant_view(make(), whole), "k_mean", whole, torch.float32).view(H, d)[H - 1].double()
    # 2 * 128 products per block and channel added in fp32: at most 256 roundings of 2^-24 of the sum of magnitudes
    bound = 256 * 2.0 ** -24 * (x[:, 0::2].abs() + x[:, 1::2].abs()).mean(0).repeat_interleave(2)
    assert bool(((got - mean).abs() <= bound).all())
    if bits == 8:
        stats = [s.clone() for s in vc.vc_prep_stats_view(make(), whole, work)]
        assert torch.equal(whole, _bundle(make(), q, k, v, perm, stats)[0])
