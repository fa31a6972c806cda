"""Many pull steps in one launch against the same steps launched one by one.

The launch passes populations between sites as they are produced; the
arithmetic is the step kernels', so the states must be equal bit for bit.
Sizes around a block (64 sites) and a lane group of the iolet blocks (8 sites a
block); more steps than one launch takes (2,048 boundary values); Windkessel
outlets, whose model runs inside the launch; a lattice with a one-sided link,
which is stepped one by one.
"""
import numpy as np
import pytest

from helpers import hand_lattice
from paper_2202_11770_gb300 import geometry as geo

pytestmark = pytest.mark.gpu
hemegb = pytest.importorskip("paper_2202_11770_gb300.hemegb")


def _pair(lat, prec, steps, setup, state=None):
    out = []
    for chunks in ([steps], [1] * steps):
        s = hemegb.Solver(lat, tau=0.7, precision=prec, scheme="ab")
        setup(s)
        if state is None:
            s.init_equilibrium()
        else:
            s.set_state(state.copy(), 0)
        for c in chunks:
            s.step(c)
        out.append((s.state(), s.reduce(), s))
    (fa, ta), (ma, qa), a = out[0]
    (fb, tb), (mb, qb), b = out[1]
    assert ta == tb == steps
    assert fa.tobytes() == fb.tobytes()
    assert ma == mb and np.array_equal(qa, qb)
    assert np.isfinite(ma)
    return a, b


def _waves(lat):
    def setup(s):
        for k, io in enumerate(lat.iolets):
            if io.kind == geo.VELOCITY:
                s.set_velocity(k, np.ones(io.n_groups), {"kind": "cosine", "mean": 0.02, "rel": 0.5, "period": 40.0})
            else:
                s.set_pressure(k, {"kind": "cosine", "mean": 1.0, "rel": 0.001, "period": 30.0})
    return setup


@pytest.mark.parametrize("prec", ["fp32", "bf16", "fp16", "fp64"])
@pytest.mark.parametrize("radius,length,inlet,outlet", [(1.2, 3, 0, 1), (1.2, 13, 0, 1), (2.9, 5, 1, 1), (4.0, 31, 0, 2),
                                                       (6.5, 40, 2, 2), (8.0, 64, 0, 1), (10.0, 70, 0, 1)])
def test_pipes(radius, length, inlet, outlet, prec):
    lat = geo.pipe(radius, length, inlet, outlet)
    _pair(lat, prec, 37, _waves(lat))


@pytest.mark.parametrize("n", [1, 2, 63, 64, 65, 129])
def test_closed_boxes(n):
    x = np.arange(300)
    lat = hand_lattice(np.stack([x % 7, x // 7 % 5, x // 35], 1)[:n], geo.CI)
    h0 = np.random.default_rng(n).uniform(-0.01, 0.01, (19, n)).astype(np.float32)
    _pair(lat, "fp32", 12, lambda s: None, h0)


def test_more_steps_than_a_launch_takes():
    lat = geo.pipe(5.0, 20)
    _pair(lat, "fp32", 1030, _waves(lat))          # two iolets: 1,024 steps a launch


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_windkessel_outlets(prec):
    lat = geo.tree(2, 2202, target_sites=30_000, length_ratio=5.0)

    def setup(s):
        _waves(lat)(s)
        s.set_windkessel(1, 2e-4, 2e4, 3e-4, 1.0)
        s.set_windkessel(3, 1e-4, 0.0, 2e-4, 1.0)
        s.set_windkessel(4, 0.0, 5e3, 4e-4, 1.0, 1.001)
    a, b = _pair(lat, prec, 23, setup)
    for k in (1, 3, 4):
        # q is an FP64 sum over the outlet's links in another order
        assert np.allclose(a.windkessel_state(k), b.windkessel_state(k), rtol=1e-12, atol=1e-15)


def test_one_sided_link_is_stepped_one_by_one():
    n = 100
    xyz = np.zeros((n, 3), np.int32)
    xyz[:, 0] = 3 * np.arange(n)
    src = np.full((18, n), -1, np.int32)
    src[0, 5] = 9                                  # site 5 pulls from 9, nothing pulls from 5
    lat = geo.from_arrays(xyz, src)
    h0 = np.random.default_rng(3).uniform(-0.01, 0.01, (19, n)).astype(np.float32)
    _pair(lat, "fp32", 9, lambda s: None, h0)
