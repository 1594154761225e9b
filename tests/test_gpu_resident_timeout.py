"""A wait of the on-chip steps that runs out (a limit of zero cycles, set from
the host): it is reported, and the lattice, initialised or loaded again,
follows the oracle.  An odd number of steps too, where the step count that the
host keeps has the other in-place order than the untouched state.

That a CTA stores nothing before its last exchange has succeeded cannot be
brought about from outside (a limit of zero cycles stops every CTA at the
first step): test_resident_source.py."""
import numpy as np
import pytest

import oracle
from oracle import thermo
from paper_1611_00907_gb300 import LbmError, Simulation, _lib, inputs

pytestmark = pytest.mark.gpu


def _setup(walls):
    e = thermo.make_eos("cs", 1.0, 4.0, 1.0, 0.85)
    rv, rl, mc, _ = thermo.maxwell(e)
    rho = (inputs.wall_drop if walls else inputs.drop)(96, 64, 16, rl, rv)
    sim = Simulation(96, 64, "cs", 1.0, 4.0, 1.0, 0.85, tau=1.0, kappa=0.5, walls=walls,
                     precision="f64", mu_bottom=mc + 0.01)
    ref = oracle.Lattice(96, 64, e, 1.0, 0.5, walls=walls, mu_bottom=mc + 0.01)
    return sim, ref.init_equilibrium(rho), rho


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("steps", [5, 8])
@pytest.mark.parametrize("again", ["init", "set_state"])
def test_a_reported_timeout_and_what_follows(again, steps, walls):
    lib = _lib.load()
    sim, ref, rho = _setup(walls)
    with sim:
        saved = sim.init(rho).step(7).get_state()     # odd: the other order
        assert lib.lbm_test_set_wait_cycles(sim._ctx, 0) == _lib.LBM_OK
        sim.step(steps)
        with pytest.raises(LbmError) as ei:
            sim.moments()
        assert ei.value.status == _lib.LBM_ERR_CUDA and "timed out" in str(ei.value)
        assert lib.lbm_test_set_wait_cycles(sim._ctx, -1) == _lib.LBM_OK
        if again == "init":
            sim.init(rho).step(steps)
            ref.step(steps)
        else:
            sim.set_state(saved).step(steps)
            ref.step(7 + steps)
        got, want = sim.moments(), ref.moments()
        for key in ("rho", "mu", "vx", "vy"):
            assert np.abs(got[key] - want[key]).max() < 1e-12 * np.abs(want[key]).max(), key
