"""Device allocations that fail behind a batch (lbm_test_fail_device_alloc
makes the n-th one report out-of-memory; nothing faults): what a batch can do
without is not needed for it to work.  Fields are held against the FP64
oracle at 1e-12 of each field's largest value, as in the parity tests."""
import numpy as np
import pytest

import oracle
from oracle import thermo
from paper_1611_00907_gb300 import Batch, LbmError, Simulation, _lib, inputs

pytestmark = pytest.mark.gpu

SIZES = [(70, 21, False), (64, 48, True), (96, 64, False)]


@pytest.fixture(autouse=True)
def disarm():
    yield
    _lib.load().lbm_test_fail_device_alloc(-1)


def _lattices():
    e = thermo.make_eos("cs", 1.0, 4.0, 1.0, 0.85)
    rv, rl, mc, _ = thermo.maxwell(e)
    specs, rhos, refs = [], [], []
    for nx, ny, walls in SIZES:
        r = min(nx, ny) / 4
        rho = (inputs.wall_drop if walls else inputs.drop)(nx, ny, r, rl, rv)
        ref = oracle.Lattice(nx, ny, e, 1.1, 0.5, walls=walls, mu_bottom=mc + 0.01)
        specs.append(dict(nx=nx, ny=ny, eos="cs", a=1.0, b=4.0, Tr=0.85, tau=1.1, kappa=0.5,
                          walls=walls, mu_bottom=mc + 0.01))
        rhos.append(rho)
        refs.append(ref.init_equilibrium(rho))
    return specs, rhos, refs


def _batch(specs, rhos):
    b = Batch(specs, precision="f64")
    for k, rho in enumerate(rhos):
        b.init(k, rho)
    return b


def _compare(b, refs):
    for k, ref in enumerate(refs):
        got, want = b.moments(k), ref.moments()
        for key in ("rho", "mu", "vx", "vy"):
            assert np.abs(got[key] - want[key]).max() < 1e-12 * np.abs(want[key]).max(), (k, key)


def _held_by_lattices(specs):
    lib = _lib.load()
    base, n = lib.lbm_test_device_allocs(), 0
    for s in specs:
        with Simulation(precision="f64", **s):
            n += lib.lbm_test_device_allocs() - base
    return n


@pytest.mark.parametrize("failing", [0, 1])
def test_steps_without_the_on_chip_steps_memory(failing, oracle_threads):
    """A batch small enough for the on-chip steps holds nothing for them until
    it makes one, and steps on the tile kernels when it cannot have it."""
    lib = _lib.load()
    specs, rhos, refs = _lattices()
    own = _held_by_lattices(specs)
    base = lib.lbm_test_device_allocs()
    with Batch(specs, precision="f64") as b:
        # the lattices' own, descriptors and work list
        assert lib.lbm_test_device_allocs() - base == own + 2
    with _batch(specs, rhos) as b:
        held = lib.lbm_test_device_allocs()
        lib.lbm_test_fail_device_alloc(failing)
        b.step(8)
        lib.lbm_test_fail_device_alloc(-1)
        assert lib.lbm_test_device_allocs() == held
        b.step(8)
        for ref in refs:
            ref.step(16)
        _compare(b, refs)
    with _batch(specs, rhos) as b:             # and with it
        held = lib.lbm_test_device_allocs()
        b.step(16)
        assert lib.lbm_test_device_allocs() == held + 2
        _compare(b, refs)


def _fails(n, call):
    lib = _lib.load()
    lib.lbm_test_fail_device_alloc(n)
    with pytest.raises(LbmError) as ei:
        call()
    lib.lbm_test_fail_device_alloc(-1)
    assert ei.value.status == _lib.LBM_ERR_OOM


@pytest.mark.parametrize("tile", [None, (32, 32)])
@pytest.mark.parametrize("failing", [0, 1])
def test_a_failed_change_leaves_the_batch_as_it_was(failing, tile, oracle_threads):
    """A change of the active lattices or of the tile shape that runs out of
    memory changes nothing: the batch goes on with the lattices, shape and work
    list it had."""
    specs, rhos, refs = _lattices()
    with _batch(specs, rhos) as b:
        if tile:
            b.set_tile(*tile)
        was = b.info()["tile"]
        b.step(4)
        _fails(failing, lambda: b.set_active(0, False))
        b.step(18)                              # every lattice still moves
        _fails(failing, lambda: b.set_tile(64, 16))
        assert b.info()["tile"] == was
        b.step(18)
        for ref in refs:
            ref.step(40)
        _compare(b, refs)
        b.set_active(1, False).step(18)
        _fails(failing, lambda: b.set_active(1, True))
        b.step(18)                              # the middle one still rests
        for k in (0, 2):
            refs[k].step(36)
        _compare(b, refs)
        b.set_active(1, True).step(18)
        for ref in refs:
            ref.step(18)
        _compare(b, refs)


@pytest.mark.parametrize("failing", range(9))
def test_a_failed_autotune_leaves_the_batch_as_it_was(failing, oracle_threads):
    """Its state copies (three lattices) or a candidate's work list cannot be
    had: state, step counts and tile shape are those before the call."""
    specs, rhos, refs = _lattices()
    with _batch(specs, rhos) as b:
        was = b.info()["tile"]
        b.step(6)
        _fails(failing, lambda: b.autotune(4))
        assert b.info()["tile"] == was and b.info()["steps"] == 6
        b.step(19)
        for ref in refs:
            ref.step(25)
        _compare(b, refs)
