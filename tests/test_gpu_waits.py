"""Multi-step launches whose waits run out, do not fit, are captured or overlap.

The blocks of such a launch wait for one another, each wait bounded by a number
of polls.  A wait that runs out must reach the caller as HLB_ERR_WAIT from
every call that synchronises, until the state is set anew; here the limit of
one kind of wait is zero polls, so that whatever is not there at the first look
has run out, and the kernel returns.  A launch that does not fit on the device,
or whose stream is being captured, is taken step by step, and solvers on
several streams do not disturb one another: the same bits each time.
"""
import ctypes as C

import numpy as np
import pytest

from paper_2202_11770_gb300 import geometry as geo

pytestmark = pytest.mark.gpu
hemegb = pytest.importorskip("paper_2202_11770_gb300.hemegb")
torch = pytest.importorskip("torch")

KINDS = ["bulk", "iolet", "flux"]
POLLS = 1 << 22


def _tune(s, limits=(POLLS,) * len(KINDS), next_step=0, blocks=0):
    """hlb_multi_test: poll limits by kind, number of the next step, blocks taken to fit."""
    fn = hemegb.library().hlb_multi_test
    fn.argtypes = [C.c_void_p, C.POINTER(C.c_uint32), C.c_uint32, C.c_int]
    assert fn(s.handle, (C.c_uint32 * len(KINDS))(*limits), next_step, blocks) == hemegb.HLB_OK


def _start(lat, prec="fp32", windkessel=True):
    s = hemegb.Solver(lat, tau=0.7, precision=prec, scheme="ab")
    return _set(s, windkessel)


def _set(s, windkessel=True, model=(0.02, 50.0, 0.05)):
    for k, io in enumerate(s.iolets):
        if io.kind == geo.VELOCITY:
            s.set_velocity(k, np.ones(io.n_groups), {"kind": "cosine", "mean": 0.02, "rel": 0.5, "period": 40.0})
        elif windkessel:
            s.set_windkessel(k, *model, 1.0)
        else:
            s.set_pressure(k, 1.0)
    s.init_equilibrium()
    return s


def _code(call):
    with pytest.raises(hemegb.HlbError) as err:
        call()
    return err.value.code


@pytest.mark.parametrize("steps", [5, 30])
@pytest.mark.parametrize("kind", KINDS)
def test_a_wait_that_runs_out_is_reported(kind, steps):
    lat = geo.pipe(8.0, 64)
    s = _start(lat)
    s.step(9)
    s.reduce()                                   # a sound launch reports nothing
    # without its link masses an outlet's block gives up, and its links' wait for the ghost density
    # runs out by itself before the others do
    _tune(s, [0 if k == kind else POLLS if kind == "flux" else 1 << 14 for k in KINDS])
    s.step(steps)
    for call in (s.reduce, s.state, s.macros, s.iolet_monitor, lambda: s.windkessel_state(1), s.reduce):
        assert _code(call) == hemegb.HLB_ERR_WAIT
    rho, u, _ = s.macros_device()
    assert not bool(torch.isfinite(rho).all())
    _tune(s)
    a, b = _set(s), _start(lat)                  # set anew: as good as a new solver
    for x in (a, b):
        x.step(steps)
    assert a.state()[0].tobytes() == b.state()[0].tobytes()
    assert a.reduce()[0] == b.reduce()[0] and a.windkessel_state(1) == b.windkessel_state(1)


def test_a_launch_that_does_not_fit_is_taken_step_by_step():
    lat = geo.tree(2, 2202, target_sites=60_000, length_ratio=5.0)
    a, b = _start(lat, "fp64", windkessel=False), _start(lat, "fp64", windkessel=False)
    _tune(a, blocks=1 << 20)                     # 940 blocks, of which the device holds some 600
    a.step(9)
    for _ in range(9):
        b.step(1)
    assert a.state()[0].tobytes() == b.state()[0].tobytes() and a.t == b.t == 9


def test_captured_steps():
    lat = geo.pipe(4.0, 31)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        a, b = _start(lat, windkessel=False), _start(lat, windkessel=False)
        for x in (a, b):
            x.step(7)
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=stream):
            a.step(8)
        graph.replay()
        b.step(8)
        assert a.t == b.t == 15
        assert a.state()[0].tobytes() == b.state()[0].tobytes()


def test_solvers_on_two_streams():
    lats = [geo.pipe(8.0, 64), geo.pipe(10.0, 70)]
    want = []
    for lat in lats:
        s = _start(lat, windkessel=False)
        s.step(1200)
        want.append(s.state()[0].tobytes())
    runs = []
    for lat in lats:
        with torch.cuda.stream(torch.cuda.Stream()):
            runs.append(_start(lat, windkessel=False))
    for _ in range(6):
        for s in runs:
            s.step(200)
    assert [s.state()[0].tobytes() for s in runs] == want


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("before", [1, 2, 37, 38])
def test_step_numbers_that_start_again(before, prec):
    """The 32-bit step numbers run out `before` steps into a run of 37 with
    outlet models: the numbers after that must not match the words that hold
    no number yet (0)."""
    lat = geo.pipe(8.0, 64)
    a, b = _start(lat, prec), _start(lat, prec)
    _tune(a, next_step=2 ** 32 - before)
    for s in (a, b):
        s.step(1)
        s.step(37)
        s.step(20)
    assert a.state()[0].tobytes() == b.state()[0].tobytes()
    assert a.windkessel_state(1) == b.windkessel_state(1)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("sites", [0, 30_000])
def test_windkessel_runs_do_not_depend_on_the_cut(sites, prec):
    """The outlet models of a multi-step launch and of single steps sum the link
    masses in one order: states and models equal bit for bit, at resistances
    that carry the last bits of an outflow into the ghost density, and outlets
    of fewer and more links than the 512 that a block takes at once.  400 steps:
    the inlet's flow has come to the outlets."""
    lat = geo.tree(2, 2202, target_sites=sites, length_ratio=5.0) if sites else geo.pipe(8.0, 64)
    a, b = (_set(_start(lat, prec), model=(0.01, 200.0, 0.03)) for _ in range(2))
    a.step(400)
    for _ in range(400):
        b.step(1)
    assert a.state()[0].tobytes() == b.state()[0].tobytes()
    assert np.isfinite(a.reduce()[0])
    for k in range(1, len(lat.iolets)):
        assert a.windkessel_state(k) == b.windkessel_state(k)
