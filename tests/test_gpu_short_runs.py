"""Runs of any length give the same bits however they are queued: call by call, as launches
(also as programmatic dependents), and as replays of the graphs that runs of 2, 4, .. 64 steps
get when they come back; from either slab, after a change of tiling, and for batches of one and
of two launch groups."""
import numpy as np
import pytest

from tests import pairs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,nx,ny", [("fp32", 64, 64), ("fp32", 193, 61), ("fp32", 600, 40),
                                             ("fp32", 512, 300), ("fp64", 60, 31)])
def test_run_lengths_give_the_same_bits(precision, nx, ny):
    c = pairs.case(nx, ny, tr=0.75, sigma=0.114, visc="linear", nu_l=0.05, nu_v=0.3)
    f = pairs.droplet_state(c, vel=0.02)
    with pairs.gpu_lattice(c, precision) as L:
        L.set_populations(f)
        for _ in range(311):
            L.step(1)
        ref = L.get_populations()
    with pairs.gpu_lattice(c, precision) as L:
        for tiling in ((0, 0, 0), (64, 0, 5)):
            L.set_tiling(*tiling)
            for lengths in ([36, 36, 36, 3, 100, 100], [63, 63, 63, 63, 59], [7] * 44 + [3],
                            [311], [1, 62, 62, 62, 62, 62]):
                assert sum(lengths) == 311
                L.set_populations(f)
                for n in lengths:
                    L.step(n)
                assert np.array_equal(L.get_populations(), ref), (tiling, lengths)


def test_run_lengths_of_a_batch():
    from paper_1211_6932_gb300 import Batch
    from tests.test_gpu_batch import CASES, instance, start_fields
    out = []
    for lengths in ([1] * 75, [36, 36, 3], [7] * 10 + [5]):
        b = Batch([instance(c) for c in CASES], precision="fp32", tile_threads=64)
        for i, c in enumerate(CASES):
            b.init_fields(i, *start_fields(c, 20 + i))
        for n in lengths:
            b.step(n)
        out.append([b.get_populations(i) for i in range(len(CASES))])
        b.close()
    for o in out[1:]:
        for x, y in zip(o, out[0]):
            assert np.array_equal(x, y)
