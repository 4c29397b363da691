"""The FP64 kernel at the widths where its sweep changes: full-width strips (nx at most the
CTA's threads, the periodic neighbours read across the row) up to and beyond the CTA width,
odd widths, single columns and rows, chunks that end with one row, periodic and walled.
Against the oracle to 1e-12 (its stated bound per step, kept over 12 steps with room: the
rounding of an update is about 1e-16)."""
import numpy as np
import pytest

import oracle
from tests import pairs

pytestmark = pytest.mark.gpu

SIZES = [(1, 5), (2, 3), (3, 1), (31, 9), (63, 7), (64, 7), (65, 7), (127, 6), (128, 6), (129, 6),
         (252, 5), (253, 5)]


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("nt,rows", [(64, 1), (64, 4), (128, 1), (128, 3), (0, 0)])
def test_fp64_widths_match_the_oracle(nt, rows, walls):
    rng = np.random.default_rng(7)
    for nx, ny in SIZES:
        c = pairs.case(nx, ny, tr=0.7, sigma=0.114, walls=walls, visc="linear", nu_l=0.05,
                       nu_v=0.3)
        rho = 0.1 + 0.05 * rng.random((ny, nx))
        f = oracle.equilibrium(rho, 0.02 * rng.standard_normal((ny, nx)),
                               0.02 * rng.standard_normal((ny, nx)))
        with pairs.gpu_lattice(c, "fp64", tile_threads=nt, tile_rows=rows) as L:
            L.set_populations(f)
            start = L.get_populations()
            L.step(12)
            got = L.get_populations()
        ref = oracle.run(pairs.oracle_params(c), start, 12)
        assert np.max(np.abs(got - ref)) <= 1e-12 * np.max(np.abs(ref)), (nx, ny)
