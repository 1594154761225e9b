"""Ragged last tiles on the two-nodes-per-lane path (64-wide shapes) against
the general tile path (tensor maps switched off) of the same lattice:
remainders of 4, odd and even widths, a remainder of one pair less than a
tile, both directions, and with walls.

Tolerances: both paths round the same FP32 update in different order.  Over n
steps the density differs by at most n 2 2^-24 of its largest value (each
step rounds a population by at most 2^-24 of itself on either side), mu, a
difference of terms of size 2 a rho with |psi''| + kappa 20/3 < 6, by six
times that, the velocity, which follows tau grad(mu), by twelve times."""
import numpy as np
import pytest

from paper_1611_00907_gb300 import Simulation, eos_coexistence, inputs

pytestmark = pytest.mark.gpu

SIZES = [(196, 96), (197, 53), (199, 100), (233, 52), (254, 63), (255, 85), (256, 56), (319, 101)]
STEPS = 7


def _rho(nx, ny, walls):
    rv, rl, mc = eos_coexistence("cs", 1.0, 4.0, 1.0, 0.85)
    r = min(nx, ny) / 4
    return (inputs.wall_drop(nx, ny, r, rl, rv) if walls
            else inputs.drop(nx, ny, r, rl, rv)), rl, mc


def _check(got, want, rl):
    drho = STEPS * 2 * 2.0 ** -24 * rl
    for key, tol in (("rho", drho), ("mu", 6 * drho), ("vx", 12 * drho), ("vy", 12 * drho)):
        assert np.abs(got[key] - want[key]).max() < tol, key


def _run(nx, ny, walls, tile, precision):
    rho, rl, mc = _rho(nx, ny, walls)
    ux = 0.02 * np.cos(2 * np.pi * np.arange(nx) / nx)[None, :] * np.ones((ny, 1))
    with Simulation(nx, ny, "cs", 1.0, 4.0, 1.0, 0.85, tau=1.0, kappa=0.5, walls=walls,
                    precision=precision, rho_ref=0.15, mu_bottom=mc + 0.01) as sim:
        sim.set_tile(*tile)
        sim.init(rho, ux, 0.5 * ux).step(STEPS)
        return sim.moments(), rl


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("precision", ["f32", "f32_offset"])
@pytest.mark.parametrize("tile", [(64, 16), (64, 32)])
def test_ragged_pair_tiles_match_the_general_path(tile, precision, walls, monkeypatch):
    for nx, ny in SIZES:
        got, rl = _run(nx, ny, walls, tile, precision)
        with monkeypatch.context() as m:
            m.setenv("CPLBM_NO_TMA", "1")
            want, _ = _run(nx, ny, walls, tile, precision)
        _check(got, want, rl)
