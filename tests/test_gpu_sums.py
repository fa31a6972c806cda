"""FP64 mass of hlb_reduce against a correctly rounded sum of the same state.

A block sums four sites a thread over 256 threads: sizes around one warp, one
block (1,024 sites) and several.  FP32 and 16-bit values are summed as hi + lo
pairs of FP32: every addition's rounding error goes to lo, whose own rounding
is 2^-24 of at most 19 x 2^-24 of the site's absolute sum, so 2^-43 of the
absolute sum of the state bounds it; the FP64 additions above it are fewer
than 64 in a chain, 2^-53 of the absolute sum each, and mass = n + sum rounds
once more.  A site whose sum leaves the FP32 range is summed in FP64.
"""
import math

import numpy as np
import pytest

from paper_2202_11770_gb300 import geometry as geo

pytestmark = pytest.mark.gpu
hemegb = pytest.importorskip("paper_2202_11770_gb300.hemegb")


def _closed(n):
    xyz = np.zeros((n, 3), np.int32)
    xyz[:, 0] = 2 * np.arange(n)
    return geo.from_arrays(xyz, np.full((18, n), -1, np.int32))


@pytest.mark.parametrize("prec", ["fp32", "bf16", "fp16", "fp64"])
@pytest.mark.parametrize("n", [1, 33, 255, 1023, 1024, 1025, 5000])
def test_mass_equals_the_exact_sum(n, prec):
    h = np.random.default_rng(n).normal(0.0, 0.01, (19, n)) * 10.0 ** np.random.default_rng(n + 1).uniform(-6, 0, (19, n))
    if prec == "bf16":
        raw = (h.astype(np.float32).view(np.uint32) >> 16).astype(np.uint16)
        val = hemegb.bf16_to_float(raw).astype(np.float64)
    else:
        raw = h.astype({"fp32": np.float32, "fp16": np.float16, "fp64": np.float64}[prec])
        val = raw.astype(np.float64)
    s = hemegb.Solver(_closed(n), tau=0.8, precision=prec)
    s.set_state(raw, 0)
    want, scale = math.fsum(val.ravel()), float(np.abs(val).sum())
    assert abs((s.reduce()[0] - n) - want) <= (2.0 ** -43 + 64 * 2.0 ** -53) * scale + 2.0 ** -52 * n


def test_site_sum_beyond_the_fp32_range():
    n = 300
    h = np.zeros((19, n), np.float32)
    h[3, 7] = h[5, 7] = 3.0e38                 # their sum is not an FP32 number
    h[4, 290] = h[8, 290] = -3.0e38
    h[1, 100] = 0.25
    s = hemegb.Solver(_closed(n), tau=0.8, precision="fp32")
    s.set_state(h, 0)
    assert abs(s.reduce()[0]) <= 1e25          # FP64: the four large values cancel to its rounding
