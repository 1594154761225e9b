"""Densities below the normal numbers of FP32: what is read back, the density,
the sums and mu, is what the lattice holds.

Tolerances.  The density is exact.  The sums add at most 1470 FP64 values, each
addition rounding by 2^-53.  mu of a uniform near-vacuum is R T (ln rho + a few)
in FP32: four times 2^-24 of the approximate logarithm (its documented bound)
and six roundings of constants, products and sums: 10 x 2^-24, of which twice
is allowed."""
import numpy as np
import pytest

from paper_1611_00907_gb300 import Simulation

pytestmark = pytest.mark.gpu


def _sim(precision):
    return Simulation(70, 21, "cs", 1.0, 4.0, 1.0, 0.85, precision=precision)


@pytest.mark.parametrize("precision", ["f32", "f32_offset", "f16_offset"])
@pytest.mark.parametrize("value", [1e-40, 2e-45, 1.1754943e-38, 1.2e-38, 1e-30])
def test_densities_are_read_back(precision, value):
    rho = np.full((21, 70), value)
    rho[3, 5] = 0.25
    want = rho.astype(np.float32).astype(np.float64)
    with _sim(precision) as sim:
        sim.init(rho)
        assert np.array_equal(sim.moments(fields=("rho",))["rho"], want)
        assert abs(sim.reduce()[0] - want.sum()) <= 1470 * 2.0 ** -53 * want.sum()
    uniform = np.full((21, 70), float(np.float32(value)))
    with _sim(precision) as sim, _sim("f64") as ref:
        mass = sim.init(uniform).reduce()[0]
        assert abs(mass - uniform.sum()) <= 1470 * 2.0 ** -53 * mass
        mu = ref.init(uniform).moments(fields=("mu",))["mu"]
        assert (np.abs(sim.moments(fields=("mu",))["mu"] - mu) <= 20 * 2.0 ** -24 *
                np.abs(mu)).all()
