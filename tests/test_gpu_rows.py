"""Row form of the compact index table and the two-site step kernels.

A tile of 256 sites has the row form when every source of its sites lies where
its lattice row says and the rows' shifts span at most 8 bits; any other tile
keeps 16-bit offsets.  Both forms name the same sources as the int32 table, so
every run must equal the int32-table run bit for bit.  Sizes: around one warp
(32), one pair of warps' sites (64), one tile (256) and two tiles, and a single
site; boxes without holes (row form) and with holes (offset form).
"""
import numpy as np
import pytest

from helpers import hand_lattice
from paper_2202_11770_gb300 import geometry as geo

pytestmark = pytest.mark.gpu
hemegb = pytest.importorskip("paper_2202_11770_gb300.hemegb")


def _box(n, holes):
    """The first n sites in (z, y, x) order of a 13 x 7 x .. box, every seventh one missing with `holes`."""
    x = np.arange(13 * 7 * 60)
    pts = np.stack([x % 13, x // 13 % 7, x // 91], axis=1)
    if holes:
        pts = pts[x % 7 != 3]
    return hand_lattice(pts[:n], geo.CI)


def _raw(a, prec):
    if prec == "bf16":
        return (np.ascontiguousarray(a, np.float32).view(np.uint32) >> 16).astype(np.uint16)
    return a.astype({"fp32": np.float32, "fp16": np.float16, "fp64": np.float64}[prec])


def _same_bits(lat, prec, scheme, seed, wide=False):
    h0 = _raw(np.random.default_rng(seed).uniform(-0.01, 0.01, (19, lat.n)), prec)
    out = []
    for full in (False, True):
        s = hemegb.Solver(lat, tau=0.7, precision=prec, scheme=scheme, full_index=full, wide_offsets=wide)
        s.set_state(h0.copy(), 0)
        s.step(5)
        out.append((s.state()[0], s.reduce()[0], s.macros()))
    (fa, ma, qa), (fb, mb, qb) = out
    assert fa.tobytes() == fb.tobytes() and ma == mb
    assert all(np.array_equal(a, b, equal_nan=True) for a, b in zip(qa, qb))


@pytest.mark.parametrize("scheme", ["ab", "aa"])
@pytest.mark.parametrize("holes", [False, True], ids=["rows", "holes"])
@pytest.mark.parametrize("n", [1, 2, 31, 33, 63, 65, 255, 256, 257, 289, 511, 1000])
def test_ragged_sizes_equal_the_int32_table(n, holes, scheme):
    lat = _box(n, holes)
    for prec in ("fp32", "bf16"):
        _same_bits(lat, prec, scheme, n)
    _same_bits(lat, "fp16", scheme, n, wide=True)
    _same_bits(lat, "fp64", scheme, n)


@pytest.mark.parametrize("scheme", ["ab", "aa"])
@pytest.mark.parametrize("span", [255, 256, 300])
@pytest.mark.parametrize("bent", [0, 1])
def test_widest_row_shift(span, bent, scheme):
    """Sites 0 and 1 pull direction 3 (0, 1, 0) with row shifts that differ by
    exactly `span`; site 0 also pulls direction 7 (1, 1, 0) of the same row,
    from the neighbour that the row form expects or (bent) the one beside it."""
    n = 1000
    xyz = np.zeros((n, 3), np.int32)
    xyz[:, 0] = np.arange(n)
    src = np.full((18, n), -1, np.int32)

    def link(i, x, s):          # x pulls direction i from s, and s the opposite one from x
        src[i - 1, x] = s
        src[i if i % 2 else i - 2, s] = x

    link(3, 0, 310)
    link(3, 1, 311 + span)
    link(7, 0, 309 - bent)
    lat = geo.from_arrays(xyz, src)
    for prec in ("fp32", "bf16", "fp64"):
        _same_bits(lat, prec, scheme, span)


@pytest.mark.parametrize("prec", ["fp32", "bf16", "fp16"])
@pytest.mark.parametrize("radius,length,inlet,outlet", [(1.2, 3, 0, 1), (1.2, 12, 1, 0), (2.9, 5, 1, 1), (4.0, 7, 0, 1),
                                                       (4.0, 8, 0, 2), (8.0, 64, 0, 1)])
def test_aa_iolet_sites_in_the_grid_equal_the_pass(radius, length, inlet, outlet, prec):
    """Iolet sites stepped inside the AA step's grid (compact table) against the
    pass after it (int32 table): states, fluxes and mass bit for bit, after an
    even and an odd number of steps; 5 to 197 iolet sites an end, odd and even
    site counts (the 16-bit even step pairs neighbours when it is even)."""
    lat = geo.pipe(radius, length, inlet, outlet)
    runs = []
    for full in (False, True):
        s = hemegb.Solver(lat, tau=0.7, precision=prec, scheme="aa", full_index=full)
        for k, io in enumerate(lat.iolets):
            if io.kind == geo.VELOCITY:
                s.set_velocity(k, np.ones(io.n_groups), {"kind": "cosine", "mean": 0.02, "rel": 0.5, "period": 40.0})
            else:
                s.set_pressure(k, {"kind": "cosine", "mean": 1.0, "rel": 0.001, "period": 30.0})
        s.init_equilibrium()
        got = []
        for steps in (8, 3):
            s.step(steps)
            got.append((s.state()[0].tobytes(), s.reduce()))
        runs.append(got)
    for (fa, (ma, qa)), (fb, (mb, qb)) in zip(*runs):
        assert fa == fb and ma == mb and np.array_equal(qa, qb)
