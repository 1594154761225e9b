"""Device allocations that fail behind a batch (lbm_test_fail_device_alloc
makes the n-th one report out-of-memory; nothing faults): what a batch can do
without is not needed for it to work.  Fields are held against the FP64
oracle at 1e-12 of each field's largest value, as in the parity tests."""
import numpy as np
import pytest

import oracle
from oracle import thermo
from paper_1611_00907_gb300 import Batch, Simulation, _lib, inputs

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
