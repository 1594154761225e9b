"""Blocks of steps with the lattice in shared memory (csrc/resident.cu), the
path of small lattices and batches when no tile shape has been chosen:
against the FP64 oracle, at sizes where its cut into tiles has edges (one
tile, tiles of a few nodes, ragged last tiles, tiles on one or both walls),
from both in-place parities, and against the tile kernels in FP32.

Tolerances.  FP64: 1e-12 of each field's largest value over a few tens of
steps, as the tile kernels' parity tests.  FP32, two paths that round the
same update in different order for 30 steps: each step rounds a population
by at most 2^-24 of itself and the two may differ by twice that, so the
density differs by at most 30 * 2 * 2^-24 = 3.6e-6 of rho_l.  mu is the
difference of terms of the size of 2 a rho: it moves by |psi''| + kappa 20/3
< 6 times the density's difference.  The velocity follows tau grad(mu) over
the steps the momentum remembers (tau of them): below twice that per unit
length."""
import numpy as np
import pytest

import oracle
from oracle import thermo
from paper_1611_00907_gb300 import Batch, LbmError, Simulation, _lib, inputs

pytestmark = pytest.mark.gpu

SIZES = [(5, 5), (7, 9), (17, 13), (64, 64), (65, 33), (131, 70), (200, 9), (250, 120)]


def _state(eos, nx, ny, walls, Tr=0.85):
    par = dict(cs=(1.0, 4.0, 0.5, 4.0), rks=(2 / 49, 2 / 21, 0.01, 2.0),
               pr=(2 / 49, 2 / 21, 0.01, 2.0), vdw=(9 / 49, 2 / 21, 0.01, 2.0))[eos]
    e = thermo.make_eos(eos, par[0], par[1], 1.0, Tr, 0.344)
    rv, rl, mc, _ = thermo.maxwell(e)
    r = max(2.0, min(nx, ny) / 4)
    rho = (inputs.wall_drop(nx, ny, r, rl, rv, par[3]) if walls
           else inputs.drop(nx, ny, r, rl, rv, par[3]))
    ux = 0.02 * np.cos(2 * np.pi * np.arange(ny) / ny)[:, None] * np.ones((1, nx))
    return e, par, rho, ux, np.full_like(ux, 0.01), mc


def _rel(got, want):
    return np.abs(got - want).max() / np.abs(want).max()


def _sim(eos, nx, ny, walls, precision, tau, top_mode=0):
    e, par, rho, ux, uy, mc = _state(eos, nx, ny, walls)
    sim = Simulation(nx, ny, eos, par[0], par[1], 1.0, 0.85, 0.344, tau=tau, kappa=par[2],
                     walls=walls, precision=precision, mu_bottom=mc + 0.01, top_mode=top_mode,
                     mu_top=mc - 0.01)
    sim.init(rho, ux, uy)
    ref = oracle.Lattice(nx, ny, e, tau, par[2], walls=walls, mu_bottom=mc + 0.01,
                         top_mode=top_mode, mu_top=mc - 0.01)
    ref.init_equilibrium(rho, ux, uy)
    return sim, ref


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("size", SIZES)
@pytest.mark.parametrize("blocks", [(4,), (1, 5, 7), (37,)])
def test_blocks_of_steps_fp64(size, walls, blocks, oracle_threads):
    nx, ny = size
    if walls and ny < 7:
        pytest.skip("walls need seven rows")
    eos = ("cs", "rks", "pr", "vdw")[(nx + ny) % 4]
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


@pytest.mark.parametrize("precision", ["f32", "f32_offset"])
@pytest.mark.parametrize("walls", [False, True])
def test_blocks_of_steps_fp32_match_the_tile_kernels(precision, walls):
    for size in SIZES[3:]:
        tiles, _ = _sim("cs", *size, walls, precision, 1.0)
        _, par, rho, ux, uy, mc = _state("cs", *size, walls)
        spec = dict(nx=size[0], ny=size[1], eos="cs", a=par[0], b=par[1], Tr=0.85, omega=0.344,
                    tau=1.0, kappa=par[2], walls=walls, mu_bottom=mc + 0.01, mu_top=mc - 0.01)
        # (a batch: a periodic FP32 lattice by itself stays on the tile kernels)
        with Batch([spec], precision=precision) as many, tiles:
            many.init(0, rho, ux, uy)
            tiles.set_tile(64, 16)
            a, b = many.step(30).moments(0), tiles.step(30).moments()
            drho = 3.6e-6 * b["rho"].max()
            for key, tol in (("rho", drho), ("mu", 6 * drho), ("vx", 12 * drho),
                             ("vy", 12 * drho)):
                assert np.abs(a[key] - b[key]).max() < tol, (size, key)


def test_batch_of_small_lattices_fp64(oracle_threads):
    made = [_sim(eos, nx, ny, walls, "f64", 1.1) for eos, nx, ny, walls in
            (("cs", 70, 21, False), ("pr", 33, 40, True), ("vdw", 64, 64, False))]
    specs = []
    for (sim, ref), (eos, nx, ny, walls) in zip(made, (("cs", 70, 21, False),
                                                       ("pr", 33, 40, True),
                                                       ("vdw", 64, 64, False))):
        _, par, rho, ux, uy, mc = _state(eos, nx, ny, walls)
        specs.append((dict(nx=nx, ny=ny, eos=eos, a=par[0], b=par[1], Tr=0.85, tau=1.1,
                           kappa=par[2], walls=walls, mu_bottom=mc + 0.01), rho, ux, uy))
        sim.close()
    with Batch([s[0] for s in specs], precision="f64") as b:
        for k, s in enumerate(specs):
            b.init(k, *s[1:])
        b.step(6)
        b.set_active(1, False)         # the cut follows the active lattices
        b.step(8)
        b.set_active(1, True)
        b.step(5)
        for k, (_, ref) in enumerate(made):
            ref.step(11 if k == 1 else 19)
            got, want = b.moments(k), ref.moments()
            for key in ("rho", "mu", "vx", "vy"):
                assert _rel(got[key], want[key]) < 1e-12, (k, key)


def test_batch_steps_inside_a_callers_graph_capture(oracle_threads):
    """A block of batch steps that the caller captures into its own CUDA graph
    is launched on the tile kernels and may be replayed: a resident launch
    could not, the tags of its exchange words are those of one run."""
    import torch
    sim, ref = _sim("cs", 70, 21, False, "f64", 1.1)
    sim.close()
    _, par, rho, ux, uy, mc = _state("cs", 70, 21, False)
    stream = torch.cuda.Stream()
    with Batch([dict(nx=70, ny=21, eos="cs", a=par[0], b=par[1], Tr=0.85, tau=1.1, kappa=par[2],
                     mu_bottom=mc + 0.01)], precision="f64", stream=stream.cuda_stream) as b:
        b.init(0, rho, ux, uy)
        b.step(2)                         # kernel attributes set outside the capture
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            b.step(8)
        for _ in range(3):
            g.replay()
        torch.cuda.synchronize()
        b.step(4)                         # resident, from where the replays ended
        ref.step(2 + 3 * 8 + 4)
        got, want = b.moments(0), ref.moments()
        for key in ("rho", "mu", "vx", "vy"):
            assert _rel(got[key], want[key]) < 1e-12, key


def test_wait_limit_leaves_the_state_and_is_reported():
    # a limit of zero cycles: every tile gives up at its first exchange
    lib = _lib.load()
    sim, ref = _sim("cs", 96, 64, False, "f64", 1.0)
    with sim:
        f0 = sim.populations()
        assert lib.lbm_test_set_wait_cycles(sim._ctx, 0) == _lib.LBM_OK
        sim.step(8)
        with pytest.raises(LbmError) as ei:
            sim.moments()
        assert "timed out" in str(ei.value)
        assert np.array_equal(sim.populations(), f0)
        assert lib.lbm_test_set_wait_cycles(sim._ctx, -1) == _lib.LBM_OK
        _, _, rho, ux, uy, _ = _state("cs", 96, 64, False)
        sim.init(rho, ux, uy).step(8)
        ref.step(8)
        assert _rel(sim.moments()["rho"], ref.moments()["rho"]) < 1e-12
