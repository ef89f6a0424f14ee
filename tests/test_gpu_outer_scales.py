"""The NVFP4 outer scales: K's formed by the items of the codes' pass up to 16 items per CTA, by a launch in front of it
beyond; Q's by the items where their launch does not go in turns, by the finalization beyond.  A head's codes and scales are
the same bytes in every form, and the same as in a call of its own."""
import pytest
import torch

import paper_2609_15810_b200 as vc
from paper_2609_15810_b200 import binding
from paper_2609_15810_b200.binding import Params, alloc_buffers

pytestmark = pytest.mark.gpu

ALL = vc.VC_FLAG_ALL
SECTIONS = ["q_codes", "k_codes", "v_codes", "q_micro", "k_micro", "v_micro", "q_scale", "k_scale", "v_means", "k_mean"]


def _prep(q, k, v, grid, p_format, flags, heads_per_pass=0):
    B, H, N, d = q.shape
    p = Params.make(B, H, N, d, grid, bits=4, p_format=p_format, flags=flags, heads_per_pass=heads_per_pass)
    quant, work = alloc_buffers(p)
    quant.zero_()
    n0 = vc.vc_launch_count()
    vc.vc_prep(p, q, k, v, None, quant, work)
    launches = vc.vc_launch_count() - n0
    vc.vc_poll_status(work)
    view = vc.vc_quant_view(p, quant)
    return {n: binding.section(view, n, quant).view(H, -1) for n in SECTIONS}, launches


# the packed row transform and the general one (no RoPE)
@pytest.mark.parametrize("flags", [ALL, ALL & ~vc.VC_FLAG_ROPE])
@pytest.mark.parametrize("p_format", [vc.VC_P_DEFAULT, vc.VC_P_EXPCAST_E4M3])
@pytest.mark.parametrize("d", [64, 128])
def test_both_forms_give_the_same_bundle(d, p_format, flags):
    grid, nb = (2, 10, 51), 8                                # 1020 tokens: the last block is ragged
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    most = 16 * 2 * sms // nb                                # heads of the largest call whose items form the scale
    g = torch.Generator(device="cuda").manual_seed(d)
    q, k, v = [torch.randn(1, most + 1, 1020, d, generator=g, device="cuda", dtype=torch.bfloat16) for _ in range(3)]
    q[:, 1], k[:, 2] = 0, 0                                  # scales of one
    k *= torch.linspace(0.1, 10.0, most + 1, device="cuda")[:, None, None]
    by_items, n_items = _prep(q[:, :most].contiguous(), k[:, :most].contiguous(), v[:, :most].contiguous(), grid, p_format, flags)
    by_launch, n_launch = _prep(q, k, v, grid, p_format, flags)
    assert (n_items, n_launch) == (5, 6)
    for n in SECTIONS:
        assert torch.equal(by_launch[n][:most], by_items[n]), n
    for group in (most // 2, most // 2 + 1):                 # the most heads whose Q items form the scale, and one more
        groups, _ = _prep(q, k, v, grid, p_format, flags, heads_per_pass=group)
        for n in SECTIONS:
            assert torch.equal(by_launch[n], groups[n]), (n, group)
    for h in (0, 1, 2, most):
        alone, _ = _prep(*[t[:, h:h + 1].contiguous() for t in (q, k, v)], grid, p_format, flags)
        for n in SECTIONS:
            assert torch.equal(by_launch[n][h:h + 1], alone[n]), (n, h)
