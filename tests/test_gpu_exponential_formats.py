"""Probabilities by exponential and cast (VC_P_EXP_E4M3 on E4M3 and INT8 scores, VC_P_EXP_MIX_E4M3): their code stores and
score buffers are their own.  Outputs against the oracle, and their time against the ExpCast kernel's on the same GPU."""
import pytest
import torch

import paper_2609_15810_b200 as vc
import vc_inputs
from paper_2609_15810_b200.binding import Params, alloc_buffers
from oracle import attention as OA

import helpers as Hh

pytestmark = pytest.mark.gpu

FORMATS = {"exp": (vc.VC_P_EXP_E4M3, 0), "exp_int8": (vc.VC_P_EXP_E4M3, vc.VC_FLAG_INT8_QK), "mix": (vc.VC_P_EXP_MIX_E4M3, 0)}


# one key tile and a key, five whole ones, ten of which the last is ragged: every buffer once, and several times
@pytest.mark.parametrize("grid", [(1, 3, 43), (5, 8, 16), (1, 1, 1153)])
@pytest.mark.parametrize("fmt", list(FORMATS))
@pytest.mark.parametrize("d", [64, 128])
def test_outputs_match_the_oracle(grid, fmt, d):
    p_format, extra = FORMATS[fmt]
    H, N = 2, grid[0] * grid[1] * grid[2]
    q, k, v = [t.cuda() for t in vc_inputs.make_qkv(vc_inputs.Workload("t", 1, H, N, d, grid, (8,), 77, "gauss"))]
    p = Params.make(1, H, N, d, grid, p_format=p_format, flags=vc.VC_FLAG_ALL | extra)
    quant, work = alloc_buffers(p)
    o = torch.empty(1, H, N, d, dtype=torch.bfloat16, device="cuda")
    vc.vc_attn(p, q, k, v, None, o, quant, work)
    vc.vc_poll_status(work)
    for h in range(H):
        bundle, cfg = Hh.oracle_prep(p, q, k, v, None, 0, h)
        ref = OA.emulate_head(bundle, cfg, p_format=OA.P_EXP_E4M3)
        Hh.check_output(o[0, h].float().cpu().numpy(), ref, float(v[0, h].float().abs().max()))


# Codes that left eight columns at a time, from two score buffers at d = 64, made these 1.84 and 1.42 times as long as ExpCast;
# they are 1.61 and 1.30 times as long.  (Both sides in turn, the best of ten.)
@pytest.mark.parametrize("d,most", [(64, 1.72), (128, 1.36)])
def test_time_beside_expcast(d, most):
    grid, H = (16, 32, 32), 16
    N = 16384
    q, k, v = [torch.randn(1, H, N, d, device="cuda", dtype=torch.bfloat16) for _ in range(3)]
    o, calls = torch.empty_like(q), []
    for p_format in (vc.VC_P_EXPCAST_E4M3, vc.VC_P_EXP_E4M3):
        p = Params.make(1, H, N, d, grid, p_format=p_format)
        quant, work = alloc_buffers(p)
        vc.vc_prep(p, q, k, v, None, quant, work)
        calls.append((p, quant, work))
    best = [float("inf"), float("inf")]
    for _ in range(12):
        for i, (p, quant, work) in enumerate(calls):
            start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            vc.vc_attn_fwd(p, quant, o, work)
            start.record()
            vc.vc_attn_fwd(p, quant, o, work)
            end.record()
            torch.cuda.synchronize()
            best[i] = min(best[i], start.elapsed_time(end))
    assert best[1] < most * best[0], best
