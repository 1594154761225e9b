"""Blocks of 16 tile-kernel steps from a captured CUDA graph on a lattice small
enough for the on-chip steps, which a chosen tile shape turns off: a change of
tile shape, wall chemical potential or wait limit between calls reaches the
replayed steps, on the legacy stream and on one of the caller's."""
import numpy as np
import pytest

import oracle
from oracle import thermo
from paper_1611_00907_gb300 import Simulation, _lib, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("own_stream", [False, True])
def test_a_change_recaptures_the_graph(own_stream, oracle_threads):
    import torch
    nx, ny = 192, 66
    e = thermo.make_eos("cs", 1.0, 4.0, 1.0, 0.85)
    rv, rl, mc, _ = thermo.maxwell(e)
    rho = inputs.wall_drop(nx, ny, 24, rl, rv, 4.0)
    stream = torch.cuda.Stream() if own_stream else None
    sim = Simulation(nx, ny, "cs", 1.0, 4.0, 1.0, 0.85, tau=1.0, kappa=0.5, walls=True,
                     precision="f64", mu_bottom=mc + 0.01,
                     stream=stream.cuda_stream if stream else None)
    ref = oracle.Lattice(nx, ny, e, 1.0, 0.5, walls=True, mu_bottom=mc + 0.01)
    ref.init_equilibrium(rho)
    lib = _lib.load()

    def both(n):
        sim.step(n)
        ref.step(n)
        got, want = sim.moments(), ref.moments()
        for key in ("rho", "mu", "vx", "vy"):
            assert np.abs(got[key] - want[key]).max() < 1e-11 * np.abs(want[key]).max(), key

    with sim:
        sim.set_tile(32, 32)
        sim.init(rho)
        both(37)                          # two graphs, then single launches
        for tile in ((64, 32), (32, 16)):
            sim.set_tile(*tile)
            both(33)                      # one single launch, then graphs
        sim.set_wall_mu(mc - 0.02)
        ref.mu_bottom = mc - 0.02
        both(32)
        assert lib.lbm_test_set_wait_cycles(sim._ctx, 1 << 40) == _lib.LBM_OK
        both(16)
