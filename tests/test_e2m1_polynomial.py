"""The polynomial that stands in for the exponential in front of an E2M1 conversion (vc_nvfp4_codes.cuh): evaluated in FP32
as the kernel does, it gives the code of 2^(x - 2) everywhere but within a rounding error of a threshold."""
import os
import re

import numpy as np
import pytest

SOURCE = os.path.join(os.path.dirname(__file__), "..", "paper_2609_15810_b200", "csrc", "vc_nvfp4_codes.cuh")
THRESHOLDS = np.array([0.25, 0.75, 1.25, 1.75, 2.5, 3.5, 5.0])


def _coefficients():
    text = open(SOURCE).read()
    body = re.search(r"e2m1_poly2.*?c\[8\] = \{(.*?)\};", text, re.S).group(1)
    return [np.float32(c.strip().rstrip("f")) for c in body.split(",")]


def _poly(x):
    c = _coefficients()
    r = np.full_like(x, c[7])
    for k in range(6, -1, -1):                       # (a product of two FP32 numbers is exact in FP64: one rounding)
        r = (r.astype(np.float64) * x + np.float64(c[k])).astype(np.float32)
    return r


def _code(v):
    return np.searchsorted(THRESHOLDS, v.astype(np.float64), side="right")


@pytest.mark.parametrize("lo,hi", [(-300.0, 0.0), (0.0, 5.2)])
def test_codes_are_those_of_the_exponential(lo, hi):
    x = np.linspace(lo, hi, 400001).astype(np.float32)
    edges = np.log2(THRESHOLDS) + 2.0
    # an FP32 sum of the value's size has an error of a few 2^-24 of it; the slope there is at least 0.2 of the value
    clear = np.abs(x[:, None].astype(np.float64) - edges).min(axis=1) > 1e-6
    assert np.array_equal(_code(_poly(x))[clear], _code(2.0 ** (x.astype(np.float64) - 2.0))[clear])


def test_thresholds_and_minus_infinity():
    edges = np.log2(THRESHOLDS) + 2.0
    below, above = (edges - 5e-7 - 2e-7 * edges).astype(np.float32), (edges + 5e-7 + 2e-7 * edges).astype(np.float32)
    assert np.array_equal(_code(_poly(below)), np.arange(7)) and np.array_equal(_code(_poly(above)), np.arange(1, 8))
    assert _poly(np.array([-np.inf], dtype=np.float32))[0] == -np.inf
