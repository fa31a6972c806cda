"""The two-site step kernels, launched step by step, against the int32 table.

Both forms of the compact index table name the sources that the int32 table
names, and the two-site kernels keep the operations of the one-site ones, so
every state must equal the int32-table run's bit for bit.  Pull steps are taken
one a call (several in one call of a small lattice run in one launch).  Sizes:
ragged ones around a warp, a pair of warps' sites, a tile and two; and around
the sizes from which tiles with holes take two sites at once (FP32 175,000,
16 bits 225,000), 16-bit AA odd steps two sites a thread (450,000), and FP32 AA
steps their iolet sites in a pass (4,000,000).
"""
import functools

import numpy as np
import pytest

from paper_2202_11770_gb300 import geometry as geo

pytestmark = pytest.mark.gpu
hemegb = pytest.importorskip("paper_2202_11770_gb300.hemegb")


@functools.lru_cache(maxsize=2)
def _box(n, holes, width=61, height=43):
    """The first n sites in (z, y, x) order of a width x height x .. box, every eleventh row's every
    seventh site missing with `holes` (some tiles keep the row form)."""
    depth = 2 + n // (width * height * 9 // 10)
    z, y, x = np.meshgrid(np.arange(depth), np.arange(height), np.arange(width), indexing="ij")
    keep = ~((x % 7 == 3) & ((y + z) % 11 == 5)) if holes else np.ones_like(x, bool)
    flat = np.nonzero(keep.ravel())[0][:n]
    index = np.full((depth + 2, height + 2, width + 2), -1, np.int32)   # a rim of solid sites
    z, y, x = flat // (width * height), flat // width % height, flat % width
    index[z + 1, y + 1, x + 1] = np.arange(n)
    c = geo.CI
    src = np.stack([index[z + 1 - c[i][2], y + 1 - c[i][1], x + 1 - c[i][0]] for i in range(1, 19)])
    return geo.from_arrays(np.stack([x, y, z], 1).astype(np.int32), src)


def _raw(a, prec):
    if prec == "bf16":
        return (np.ascontiguousarray(a, np.float32).view(np.uint32) >> 16).astype(np.uint16)
    return a.astype({"fp32": np.float32, "fp16": np.float16, "fp64": np.float64}[prec])


def _same(lat, prec, scheme, seed, wide=False, steps=4):
    h0 = _raw(np.random.default_rng(seed).uniform(-0.01, 0.01, (19, lat.n)), prec)
    out = []
    for full in (False, True):
        s = hemegb.Solver(lat, tau=0.7, precision=prec, scheme=scheme, full_index=full, wide_offsets=wide)
        assert s.compact_index == (not full)
        for k, io in enumerate(lat.iolets):
            if io.kind == geo.VELOCITY:
                s.set_velocity(k, np.ones(io.n_groups), {"kind": "cosine", "mean": 0.02, "rel": 0.5, "period": 40.0})
            else:
                s.set_pressure(k, 1.001)
        s.set_state(h0.copy(), 0)
        for _ in range(steps):
            s.step(1)
        out.append((s.state()[0].tobytes(), s.reduce()))
    (fa, (ma, qa)), (fb, (mb, qb)) = out
    assert fa == fb and ma == mb and np.array_equal(qa, qb)


@pytest.mark.parametrize("scheme", ["ab", "aa"])
@pytest.mark.parametrize("holes", [False, True], ids=["rows", "holes"])
@pytest.mark.parametrize("n", [1, 2, 31, 33, 63, 65, 255, 256, 257, 289, 511, 1000, 5003])
def test_small_lattices(n, holes, scheme):
    lat = _box(n, holes, 13, 7)
    for prec in ("fp32", "bf16", "fp16", "fp64"):
        for wide in (False, True):
            _same(lat, prec, scheme, n, wide, 5)


@pytest.mark.parametrize("prec,n", [("fp32", 174_999), ("fp32", 175_000), ("fp32", 175_105), ("fp32", 200_001),
                                    ("bf16", 224_999), ("bf16", 225_025), ("fp16", 225_033), ("fp16", 240_127)])
def test_pull_steps_of_tiles_with_holes(prec, n):
    for wide in (False, True):
        _same(_box(n, True), prec, "ab", n, wide)


@pytest.mark.parametrize("prec,n", [("fp32", 175_105), ("bf16", 449_999), ("bf16", 450_001), ("bf16", 450_432),
                                    ("fp16", 450_033), ("fp16", 460_126)])
def test_aa_steps_of_tiles_with_holes(prec, n):
    for wide in (False, True):
        _same(_box(n, True), prec, "aa", n, wide)


@pytest.mark.parametrize("prec,scheme,sites", [("fp32", "ab", 190_000), ("bf16", "ab", 240_000), ("fp16", "ab", 240_000),
                                               ("fp32", "aa", 190_000), ("bf16", "aa", 470_000), ("fp16", "aa", 470_000),
                                               ("fp32", "aa", 4_100_000)])
def test_trees(prec, scheme, sites):
    """Vessel trees: iolet sites in tiles of both forms, walls, ragged ends."""
    lat = geo.tree(2, 2202, target_sites=sites, length_ratio=5.0)
    assert lat.n % 256
    for wide in (False, True) if sites < 1_000_000 else (False,):
        _same(lat, prec, scheme, sites, wide)


@pytest.mark.parametrize("order", ["x, y, z", "backwards"])
@pytest.mark.parametrize("sites", [3_000, 49_000, 470_000])
def test_sites_in_another_order(sites, order):
    """Lattices whose tiles have the offset form throughout: their own kernels'
    choice and prefetch, in both schemes and every storage."""
    base = geo.tree(2, 2202, target_sites=sites, length_ratio=5.0)
    x, y, z = base.xyz.T
    perm = np.lexsort((z, y, x)) if order == "x, y, z" else np.arange(base.n)[::-1]
    inv = np.empty(base.n, np.int64)
    inv[perm] = np.arange(base.n)
    src = base.src[:, perm]
    lat = geo.from_arrays(base.xyz[perm], np.where(src >= 0, inv[np.maximum(src, 0)], src), iolets=base.iolets,
                          wall_normal=base.wall_normal[:, perm], amp_group=base.amp_group[perm])
    for prec in ("fp32", "bf16", "fp16", "fp64"):
        for scheme in ("ab", "aa"):
            for wide in (False, True):
                _same(lat, prec, scheme, sites, wide)
