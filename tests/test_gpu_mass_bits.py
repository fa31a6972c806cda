"""The FP64 mass sums keep the bits of an FP64 sum, whatever the storage.

Every site holds the same populations, chosen so that the rounding of a sum in
fewer bits adds up instead of averaging out: one large value and eighteen near
1, whose sum as an FP32 pair is off by some 2^-43 of the absolute sum.  Bound:
fewer than 64 FP64 additions in a chain (19 populations, 4 sites, a block of
256, the blocks, the site count), 2^-53 of the absolute sum each.
"""
import ctypes as C
import math

import numpy as np
import pytest

from paper_2202_11770_gb300 import geometry as geo

pytestmark = pytest.mark.gpu
hemegb = pytest.importorskip("paper_2202_11770_gb300.hemegb")
torch = pytest.importorskip("torch")

SITES = {"1.3": [2.0 ** 24] + [1.3] * 18, "1 + 3 ulp": [2.0 ** 24] + [1.0 + 3 * 2.0 ** -23] * 18,
         "cancelling": [2.0 ** 24] + [0.7] * 17 + [-(2.0 ** 24)]}


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("site", list(SITES))
@pytest.mark.parametrize("n", [1, 300, 5000, 1_100_000])
def test_equal_sites(n, site, prec):
    dtype = {"fp32": np.float32, "fp64": np.float64}[prec]
    h = np.repeat(np.array(SITES[site], dtype)[:, None], n, axis=1)
    xyz = np.zeros((n, 3), np.int32)
    xyz[:, 0] = 2 * np.arange(n)
    s = hemegb.Solver(geo.from_arrays(xyz, np.full((18, n), -1, np.int32)), tau=0.8, precision=prec)
    s.set_state(h, 0)
    one = math.fsum(float(v) for v in h[:, 0])
    bound = 64 * 2.0 ** -53 * n * (1.0 + float(np.abs(h[:, 0].astype(np.float64)).sum()))
    assert abs(s.reduce()[0] - n * (1.0 + one)) <= bound
    f = torch.from_numpy(h).cuda()
    out = torch.empty(1, dtype=torch.float64, device="cuda")
    assert hemegb.library().hlb_mass_static(C.c_void_p(f.data_ptr()), s.precision, n, C.c_void_p(out.data_ptr()),
                                            C.c_void_p(torch.cuda.current_stream().cuda_stream)) == hemegb.HLB_OK
    assert abs(float(out.item()) - n * (1.0 + one)) <= bound
