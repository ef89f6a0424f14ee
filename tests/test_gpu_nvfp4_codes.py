"""NVFP4 probabilities as the softmax stage of the 4-bit attention kernel forms them, taken out of it through the library's
test hook: E4M3 factors of the 16-key groups and E2M1 codes, those of the polynomial groups and those of the exponential,
against the format in 64 bits.

A code may differ only where the exact value lies on one of the format's rounding thresholds to within the FP32 arithmetic.
In the log2 domain that is x = s cs + (c - m - log2 f): the sum in brackets and the fused multiply-add are rounded once each
(2^-24 of their sizes), c, cs and m are FP32 numbers, the table of logarithms, ex2.approx and the polynomial are within 2^-21
together.  So: 2^-23 (|s cs| + |m| + 32) + 2^-21."""
import numpy as np
import pytest
import torch

import paper_2609_15810_b200 as vc
import vc_inputs
from paper_2609_15810_b200.binding import Params, alloc_buffers
from oracle import attention as OA
from oracle import codecs as OC

import helpers as Hh

pytestmark = pytest.mark.gpu

TOP = np.log2(2688.0)
E2M1_EDGES = np.log2([0.25, 0.75, 1.25, 1.75, 2.5, 3.5, 5.0])


def _rows(rows, cs, seed):
    rng = np.random.default_rng(seed)
    m = rng.uniform(-8.0, 24.0, rows).astype(np.float32)
    drop = np.where(rng.random((rows, 128)) < 0.5, rng.exponential(3.0, (rows, 128)), rng.uniform(0.0, 30.0, (rows, 128)))
    drop += np.repeat(rng.choice([0.0, 0.0, 6.0, 18.0], (rows, 8)), 16, axis=1)        # groups with small factors, and with none
    drop += rng.choice([0.0, 0.0, 5.0], rows)[:, None]                                 # rows below a maximum of an earlier tile
    s = ((m[:, None].astype(np.float64) - drop) / float(np.float32(cs))).astype(np.float32)
    s = np.round(s * 4.0) / np.float32(4.0)
    top = (m / np.float32(cs)).astype(np.float32)
    s = np.minimum(s, np.nextafter(top, np.float32(-np.inf))[:, None]).astype(np.float32)
    s[0::7, 0] = np.nextafter(top, np.float32(-np.inf))[0::7]                           # the maximum itself
    s[1::7, 100:] = -np.inf                                                             # padded keys: parts of a group, whole groups
    s[2::7, 3] = -1.0e30
    return s, m


@pytest.mark.parametrize("polynomial", [True, False])
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("cs", [3.1e-5, 0.37, 1.0 / 128.0, 7.7e-4])
def test_codes_and_factors(d, cs, polynomial):
    rows = 4100                                              # (more than a block, a ragged last one)
    s, m = _rows(rows, cs, d)
    codes, factors = [t.cpu().numpy() for t in vc.vc_test_nvfp4_codes(torch.from_numpy(s).cuda(), torch.from_numpy(m).cuda(), d, cs, polynomial)]
    codes = np.stack([codes & 15, codes >> 4], axis=2).reshape(rows, 8, 16)
    with np.errstate(divide="ignore", invalid="ignore", over="ignore"):
        z = (s.astype(np.float64) * float(np.float32(cs))).reshape(rows, 8, 16)
        eps = 2.0 ** -23 * (np.abs(z) + np.abs(m.astype(np.float64))[:, None, None] + 32.0) + 2.0 ** -21
        eps = np.where(np.isfinite(eps), eps, 0.0)
        x = z - m.astype(np.float64)[:, None, None] + TOP
        # factors: the code between the codes of both ends of the error interval
        top = x.max(axis=2)
        err = np.take_along_axis(eps, x.argmax(axis=2)[:, :, None], axis=2)[:, :, 0]
        lo, hi = [OC.e4m3_encode((2.0 ** (top + side * (err + 2.0 ** -23)) / 6.0).astype(np.float64)) for side in (-1, 1)]
        assert np.all((lo <= factors) & (factors <= hi))
        assert np.mean(lo == hi) > 0.99
        # codes under the factors as they are
        f = OC.e4m3_decode(factors)[:, :, None]
        w = np.where(f > 0, x - np.log2(np.where(f > 0, f, 1.0)), -np.inf)
    want = np.searchsorted(E2M1_EDGES, w, side="right")
    clear = np.abs(w[..., None] - E2M1_EDGES).min(axis=-1) > eps
    clear |= ~np.isfinite(w)
    for g in range(8):
        assert np.array_equal(codes[:, g][clear[:, g]], want[:, g][clear[:, g]]), (g, np.mean(codes[:, g] != want[:, g]))
        assert np.abs(codes[:, g].astype(int) - want[:, g]).max() <= 1
        assert set(np.unique(codes[:, g])) == set(range(8))
    assert clear.mean() > 0.99
    assert (factors == 0).any() and not codes[factors == 0].any() and not codes.reshape(rows, 128)[~np.isfinite(s)].any()


def test_hook_rejects_bad_arguments():
    s, m = torch.zeros(4, 128, device="cuda"), torch.zeros(4, device="cuda")
    for d, cs in ((96, 1.0), (64, 0.0)):
        with pytest.raises(vc.VcError):
            vc.vc_test_nvfp4_codes(s, m, d, cs)
    assert vc.vc_test_nvfp4_codes(s[:0], m[:0], 64, 1.0)[0].numel() == 0


# five key tiles (no polynomial) and six (the sixth with one key)
@pytest.mark.parametrize("grid", [(4, 10, 16), (1, 1, 641)])
@pytest.mark.parametrize("v_smooth", [True, False])
@pytest.mark.parametrize("d", [64, 128])
def test_outputs_on_both_sides_of_the_line(grid, v_smooth, d):
    H, N = 2, grid[0] * grid[1] * grid[2]
    q, k, v = [t.cuda() for t in vc_inputs.make_qkv(vc_inputs.Workload("t", 1, H, N, d, grid, (8,), 91, "gauss"))]
    p = Params.make(1, H, N, d, grid, bits=4, flags=vc.VC_FLAG_ALL if v_smooth else vc.VC_FLAG_ALL & ~vc.VC_FLAG_V_SMOOTH)
    quant, work = alloc_buffers(p)
    o = torch.empty(1, H, N, d, dtype=torch.bfloat16, device="cuda")
    vc.vc_attn(p, q, k, v, None, o, quant, work)
    vc.vc_poll_status(work)
    for h in range(H):
        bundle, cfg = Hh.oracle_prep(p, q, k, v, None, 0, h)
        Hh.check_output(o[0, h].float().cpu().numpy(), OA.emulate_head(bundle, cfg), float(v[0, h].float().abs().max()))
