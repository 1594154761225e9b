"""On-chip steps (csrc/resident.cu) of lattices whose tiles hold more than 256
nodes, which run other kernels than the small ones: FP64 with 384 threads, FP32
with 512 and two nodes, one above the other, per thread.  Sides odd and ragged,
so that tiles of odd height have a second node beyond them, and lattices up to
the largest that fit.  Tolerances as in test_gpu_resident.py, whose derivation
for 30 steps holds for any size."""
import numpy as np
import pytest

from paper_1611_00907_gb300 import Batch
from test_gpu_resident import _rel, _sim, _state

pytestmark = pytest.mark.gpu

SIZES = [(331, 173), (500, 201), (519, 509)]


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("size", SIZES)
@pytest.mark.parametrize("blocks", [(4,), (1, 5, 7)])
def test_large_tiles_fp64(size, walls, blocks, oracle_threads):
    nx, ny = size
    eos = ("cs", "rks", "pr", "vdw")[(nx + ny + walls) % 4]
    sim, ref = _sim(eos, nx, ny, walls, "f64", 1.1, top_mode=nx % 2)
    with sim:
        for n in blocks:
            sim.step(n)
            ref.step(n)
        got, want = sim.moments(), ref.moments()
        for key in ("rho", "mu", "vx", "vy"):
            assert _rel(got[key], want[key]) < 1e-12, key
        f = sim.populations()
        for i in range(9):
            assert _rel(f[i], ref.f[i]) < 1e-12, i


def test_large_tiles_fp64_in_a_batch(oracle_threads):
    shapes = [("cs", 211, 131, False), ("pr", 173, 97, True), ("vdw", 260, 95, False)]
    made = [_sim(eos, nx, ny, walls, "f64", 1.1) for eos, nx, ny, walls in shapes]
    specs = []
    for (sim, _), (eos, nx, ny, walls) in zip(made, shapes):
        sim.close()
        _, par, rho, ux, uy, mc = _state(eos, nx, ny, walls)
        specs.append((dict(nx=nx, ny=ny, eos=eos, a=par[0], b=par[1], Tr=0.85, tau=1.1,
                           kappa=par[2], walls=walls, mu_bottom=mc + 0.01), rho, ux, uy))
    with Batch([s[0] for s in specs], precision="f64") as b:
        for k, s in enumerate(specs):
            b.init(k, *s[1:])
        b.step(4).step(7)
        for k, (_, ref) in enumerate(made):
            ref.step(11)
            got, want = b.moments(k), ref.moments()
            for key in ("rho", "mu", "vx", "vy"):
                assert _rel(got[key], want[key]) < 1e-12, (k, key)


def _close_fp32(a, b):
    drho = 3.6e-6 * b["rho"].max()
    for key, tol in (("rho", drho), ("mu", 6 * drho), ("vx", 12 * drho), ("vy", 12 * drho)):
        assert np.abs(a[key] - b[key]).max() < tol, key


@pytest.mark.parametrize("precision", ["f32", "f32_offset"])
@pytest.mark.parametrize("size", SIZES + [(64, 48), (697, 601)])
def test_a_walled_fp32_lattice_by_itself(size, precision):
    chip, _ = _sim("cs", *size, True, precision, 1.0)
    tiles, _ = _sim("cs", *size, True, precision, 1.0)
    with chip, tiles:
        tiles.set_tile(64, 16)
        a, b = chip.step(30).moments(), tiles.step(30).moments()
        assert not np.array_equal(a["rho"], b["rho"])   # two kinds of step
        _close_fp32(a, b)


@pytest.mark.parametrize("precision", ["f32", "f32_offset"])
@pytest.mark.parametrize("walls", [False, True])
def test_fp32_lattices_in_a_batch(walls, precision):
    for size in SIZES:
        tiles, _ = _sim("cs", *size, walls, precision, 1.0)
        _, par, rho, ux, uy, mc = _state("cs", *size, walls)
        spec = dict(nx=size[0], ny=size[1], eos="cs", a=par[0], b=par[1], Tr=0.85, omega=0.344,
                    tau=1.0, kappa=par[2], walls=walls, mu_bottom=mc + 0.01, mu_top=mc - 0.01)
        with Batch([spec], precision=precision) as many, tiles:
            many.init(0, rho, ux, uy)
            tiles.set_tile(64, 16)
            _close_fp32(many.step(30).moments(0), tiles.step(30).moments())
