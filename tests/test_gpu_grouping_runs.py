"""Runs of chunks in the grouping kernel: a CTA crosses from head to head and through chunks of one to
eight tiles.  A head's labels, centroids and permutation do not depend on the heads around it, bit for
bit, and the permutation is the stable sort of the labels."""
import pytest
import torch

import paper_2609_15810_b200 as vc
from paper_2609_15810_b200.binding import Params

pytestmark = pytest.mark.gpu


def _group(v, k, iters):
    B, H, N, d = v.shape
    p = Params.make(B, H, N, d, (1, 1, N))
    work = torch.empty(vc.vc_group_workspace_bytes(p), dtype=torch.uint8, device="cuda")
    c = torch.empty(B, H, k, d, device="cuda")
    perm = torch.empty(B, H, N, dtype=torch.int32, device="cuda")
    vc.vc_group(p, v, k, iters, False, c, perm, work)
    vc.vc_poll_status(work)
    at = vc.VC_GROUP_LABELS_OFFSET
    return work[at:at + 4 * B * H * N].view(torch.int32).view(B, H, N).clone(), c, perm


@pytest.mark.parametrize("H,N,d,k", [(200, 129, 128, 64),     # chunks of two tiles, a head each
                                     (300, 64, 64, 7),        # chunks of one tile: three or two heads per CTA
                                     (80, 1025, 128, 64),     # a full chunk and one of a single token
                                     (40, 4999, 64, 33),      # runs that start and end inside a head
                                     (5, 3000, 128, 1)])
def test_heads_of_a_run_do_not_touch_one_another(H, N, d, k):
    g = torch.Generator(device="cuda").manual_seed(H + N)
    v = torch.randn(1, H, N, d, generator=g, device="cuda").bfloat16()
    labels, c, perm = _group(v, k, 3)
    assert torch.equal(perm.long(), torch.argsort(labels, dim=-1, stable=True))
    for h in (0, 1, H // 2, H - 1):
        l1, c1, p1 = _group(v[:, h:h + 1].contiguous(), k, 3)
        assert torch.equal(labels[:, h:h + 1], l1) and torch.equal(c[:, h:h + 1], c1) and torch.equal(perm[:, h:h + 1], p1), h
