"""FP64 arithmetic outside the range of the kernels' own reciprocal, quotient and square
root: subnormal arguments and results, a vanishing denominator, infinities.  There the values
are those of IEEE division and square root."""
import numpy as np
import pytest

import oracle
from tests import pairs

pytestmark = pytest.mark.gpu


def ieee_psi(rho, c):
    """Eq. 24 with Eq. 30 in numpy's FP64, factored as the kernels evaluate it."""
    with np.errstate(all="ignore"):
        x = pairs.B / 4.0 * rho
        omx = 1.0 - x
        z = (1.0 + x * (1.0 + x * omx)) / (omx * omx * omx)
        arg = 2.0 / c["G"] * rho * (c["T"] * z - c["a"] * rho - 1.0 / 3.0)
        return np.where(arg > 0.0, np.sqrt(arg), 0.0)


def test_psi_of_subnormal_arguments():
    """2 / G rho (..) is subnormal: a rounding there is up to 5e-324 / arg relative, half of
    it in psi."""
    c = pairs.case(8, 8, tr=0.7)
    rho = np.geomspace(1e-312, 3e-308, 200)
    ref = ieee_psi(rho, c)
    with pairs.gpu_lattice(c, "fp64") as L:
        got = L.eval_psi(rho)
    assert np.all(ref > 0) and np.all(np.isfinite(got))
    assert np.all(np.abs(got - ref) <= ref * (4e-15 + 4 * 5e-324 / ref / ref))


@pytest.mark.parametrize("G", [-1.0, 1.0])
def test_psi_where_the_division_has_no_finite_result(G):
    c = pairs.case(8, 8, tr=0.7, G=G)
    rho = np.array([0.0, 4.0 / pairs.B, np.inf, -np.inf, np.nan])
    with pairs.gpu_lattice(c, "fp64") as L:
        assert np.array_equal(L.eval_psi(rho), ieee_psi(rho, c))


@pytest.mark.parametrize("nx,rows", [(40, 1), (40, 4), (200, 1), (200, 4)])
def test_step_of_a_subnormal_density(nx, rows):
    """A resting density below the smallest normal number is positive: the step keeps it, to
    a few of its last places."""
    c = pairs.case(nx, 12, tr=0.7, sigma=0.114)
    rho = np.full((12, nx), 1.5e-308)
    f = oracle.equilibrium(rho, np.zeros_like(rho), np.zeros_like(rho))
    with pairs.gpu_lattice(c, "fp64", tile_rows=rows) as L:
        L.set_populations(f)
        L.step(2)
        got = L.get_populations()
    ref = oracle.run(pairs.oracle_params(c), f, 2)
    assert np.max(np.abs(got - ref)) <= 100 * 5e-324
