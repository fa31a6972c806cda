"""hlb_iolet_monitor without `flux` reads the iolet sites alone.

The same values as with `flux`, and a call that does not pass over the whole
lattice: on 3.8M FP64 sites (570 MB of populations, 70 us at 8 TB/s) it must be
at least half of that faster than the call that also sums the mass.  A run that
has blown up is reported to the caller of `flux` only, as ever.
"""
import time

import numpy as np
import pytest

from paper_2202_11770_gb300 import geometry as geo

pytestmark = pytest.mark.gpu
hemegb = pytest.importorskip("paper_2202_11770_gb300.hemegb")


def _solver(lat, prec, scheme):
    s = hemegb.Solver(lat, tau=0.8, precision=prec, scheme=scheme)
    for k, io in enumerate(lat.iolets):
        if io.kind == geo.VELOCITY:
            s.set_velocity(k, np.ones(io.n_groups), {"kind": "cosine", "mean": 0.01, "rel": 0.5, "period": 40.0})
        else:
            s.set_pressure(k, 1.0)
    s.init_equilibrium()
    s.step(3)
    return s


def _monitor(s, flux):
    k = len(s.iolets)
    f, u, r = np.full(k, -1.0), np.full(k, -1.0), np.full(k, -1.0)
    rc = hemegb.library().hlb_iolet_monitor(s.handle, f.ctypes.data if flux else None, u.ctypes.data, r.ctypes.data)
    return rc, f, u, r


@pytest.mark.parametrize("scheme", ["ab", "aa"])
@pytest.mark.parametrize("prec", ["fp32", "bf16", "fp64"])
def test_values_without_flux(prec, scheme):
    s = _solver(geo.pipe(6.0, 21), prec, scheme)
    (rc0, _, u0, r0), (rc1, _, u1, r1) = _monitor(s, False), _monitor(s, True)
    assert rc0 == rc1 == hemegb.HLB_OK and np.array_equal(u0, u1) and np.array_equal(r0, r1) and u0[0] > 0
    h = s.state()[0]
    h.view({2: np.uint16, 4: np.uint32, 8: np.uint64}[h.itemsize])[3, h.shape[1] // 2] = {
        "fp32": 0x7fc00000, "bf16": 0x7fc0, "fp64": 0x7ff8000000000000}[prec]
    s.set_state(h, 5)
    assert _monitor(s, False)[0] == hemegb.HLB_OK and _monitor(s, True)[0] == hemegb.HLB_ERR_DIVERGED


def test_no_pass_over_the_lattice():
    s = _solver(geo.pipe(100.0, 120), "fp64", "aa")
    assert s.n > 3_700_000
    best = {}
    for flux in (False, True) * 15:
        t0 = time.perf_counter()
        _monitor(s, flux)
        best[flux] = min(best.get(flux, 1.0), time.perf_counter() - t0)
    assert best[True] - best[False] >= 0.5 * s.n * 19 * 8 / 8e12
