"""What autotuning leaves a small lattice or batch with.  On the sizes here the
on-chip steps are faster than every tile shape by a factor of about 1.5 or
more (FP64 64 x 64: eight), so autotuning has to end on them, whatever number
of steps it is asked to time.  Which steps run shows in the results: each kind
is deterministic, and the two round sums in different order, so equal bits
after a run mean the same kind."""
import numpy as np
import pytest

from paper_1611_00907_gb300 import Batch, Simulation, eos_coexistence, inputs

pytestmark = pytest.mark.gpu
STEPS = 48


def _field(nx, ny, walls):
    rv, rl, mc = eos_coexistence("cs", 1.0, 4.0, 1.0, 0.85)
    r = min(nx, ny) / 4
    return (inputs.wall_drop if walls else inputs.drop)(nx, ny, r, rl, rv), mc


def _sim(nx, ny, walls, precision):
    rho, mc = _field(nx, ny, walls)
    sim = Simulation(nx, ny, "cs", 1.0, 4.0, 1.0, 0.85, tau=1.0, kappa=0.5, walls=walls,
                     precision=precision, rho_ref=0.15, mu_bottom=mc + 0.01)
    return sim, rho


def _bits(m):
    return np.concatenate([m[k].ravel() for k in ("rho", "vx", "vy", "mu")])


def _run(nx, ny, walls, precision, how):
    sim, rho = _sim(nx, ny, walls, precision)
    with sim:
        sim.init(rho, np.full_like(rho, 0.01))
        how(sim)
        return _bits(sim.step(STEPS).moments()), sim.tile


# asked for more steps, for the default (20: fewer than the 24 from which
# FP32 lattices of this size take the on-chip steps), and for too few
@pytest.mark.parametrize("args", [(64,), (), (2,)])
@pytest.mark.parametrize("nx,ny,walls,precision", [(64, 64, False, "f64"), (64, 64, True, "f64"),
                                                   (512, 256, True, "f32"),
                                                   (512, 256, True, "f32_offset"),
                                                   (256, 128, True, "f32")])
def test_a_small_lattice_keeps_its_on_chip_steps(nx, ny, walls, precision, args):
    want, tile = _run(nx, ny, walls, precision, lambda s: None)
    tiles, _ = _run(nx, ny, walls, precision, lambda s: s.set_tile(*tile))
    assert not np.array_equal(want, tiles)
    got, kept = _run(nx, ny, walls, precision, lambda s: s.autotune(*args))
    assert kept == tile and np.array_equal(got, want)


@pytest.mark.parametrize("precision", ["f32", "f32_offset"])
def test_a_periodic_fp32_lattice_gets_them_by_autotuning(precision):
    tiles, tile = _run(256, 256, False, precision, lambda s: None)
    same, _ = _run(256, 256, False, precision, lambda s: s.set_tile(*tile))
    assert np.array_equal(tiles, same)          # the tile kernels by default
    got, kept = _run(256, 256, False, precision, lambda s: s.autotune())
    assert kept == tile and not np.array_equal(got, tiles)


@pytest.mark.parametrize("args", [(64,), (), (2,)])
@pytest.mark.parametrize("precision,walls", [("f32", True), ("f32", False), ("f64", True)])
def test_a_small_batch_keeps_its_on_chip_steps(precision, walls, args):
    nx, ny, count = (256, 128, 4) if precision == "f32" else (64, 48, 4)
    rho, mc = _field(nx, ny, walls)
    specs = [dict(nx=nx, ny=ny, walls=walls, mu_bottom=mc + 0.002 * k, tau=1.0 + 0.1 * k)
             for k in range(count)]

    def run(how):
        with Batch(specs, precision=precision) as b:
            for k in range(count):
                b.init(k, rho)
            tile = b.info()["tile"]
            how(b, tile)
            b.step(STEPS)
            return np.concatenate([_bits(b.moments(k)) for k in range(count)])

    want = run(lambda b, tile: None)
    assert not np.array_equal(want, run(lambda b, tile: b.set_tile(*tile)))
    assert np.array_equal(want, run(lambda b, tile: b.autotune(*args)))


def test_autotuning_the_pressure_tensor_leaves_the_other_force_alone():
    def back(tune):
        def how(sim):
            rho, _ = _field(64, 64, False)
            sim.set_force_model("pressure_tensor")
            if tune:
                sim.autotune(4)
                sim.set_force_model("chemical_potential")
                sim.set_force_model("pressure_tensor")   # back on its default shape
            sim.set_force_model("chemical_potential")
            sim.init(rho, np.full_like(rho, 0.01))
        return how

    want, _ = _run(64, 64, False, "f64", back(False))
    got, _ = _run(64, 64, False, "f64", back(True))
    assert np.array_equal(got, want)
