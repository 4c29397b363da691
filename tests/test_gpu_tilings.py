"""Every tiling of the pair kernel gives the same bits (the arithmetic of a node does not
depend on the CTA that computes it), so the default tiling of small and ragged lattices,
with chunks down to one row (one and two rows have a kernel of their own), is compared with chunks of eight rows of 128-thread CTAs: full
width and strips, even and odd widths (ghost columns written as pairs and one by one), a last
strip of one column or of two, walls."""
import numpy as np
import pytest

from tests import pairs

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (2, 5), (7, 3), (64, 64), (65, 40), (66, 9), (125, 33), (126, 20), (193, 147),
         (253, 21), (257, 30), (300, 17), (601, 47)]


@pytest.mark.parametrize("walls", [False, True])
def test_default_tiling_equals_eight_row_chunks(walls):
    for k, (nx, ny) in enumerate(SIZES):
        c = pairs.case(nx, ny, tr=0.75, sigma=0.114, walls=walls, visc="step", nu_l=0.05,
                       nu_v=0.3)
        f = pairs.droplet_state(c, vel=0.02, seed=k)
        got = []
        for kw in ({}, {"tile_threads": 128, "tile_rows": 8}, {"tile_threads": 32, "tile_rows": 1},
                   {"tile_threads": 96, "tile_rows": 2}, {"tile_threads": 64, "tile_rows": 3}):
            with pairs.gpu_lattice(c, "fp32", **kw) as L:
                L.set_populations(f)
                L.step(70)
                got.append(L.get_populations())
        for g in got[1:]:
            assert np.array_equal(got[0], g), (nx, ny)


@pytest.mark.parametrize("wide,narrow,branches", [(12, 40, True), (14, 4, False), (2, 110, False)])
def test_batches_of_both_kinds_of_strips_choose_their_stepping(monkeypatch, wide, narrow, branches):
    """At the default tiling a batch with three tenths of its nodes or more in either kind steps
    with a launch per step and kind, others as one persistent launch: same bits as with
    LBM_PERSISTENT=1, which always takes the one launch, over runs with and without a graph."""
    from paper_1211_6932_gb300 import Batch
    from tests.test_gpu_batch import instance, start_fields
    cs = [pairs.case(500, 420 + i % 3, tr=0.75, sigma=0.114) for i in range(wide)]
    cs += [pairs.case(250 - i % 2, 250, tr=0.8, sigma=0.11) for i in range(narrow)]
    fields = [start_fields(c, 60 + i) for i, c in enumerate(cs)]
    got = []
    for env in (None, "1"):
        monkeypatch.delenv("LBM_PERSISTENT", raising=False)
        if env:
            monkeypatch.setenv("LBM_PERSISTENT", env)
        b = Batch([instance(c) for c in cs], precision="fp32")
        try:
            for i, fl in enumerate(fields):
                b.init_fields(i, *fl)
            if env:
                assert b.persistent and b.launches_per_step == 1
            else:
                assert b.persistent == (not branches)
                assert b.launches_per_step == (2 if branches else 1)
            b.step(70)
            b.step(6)
            got.append([b.get_populations(i) for i in range(0, len(cs), 7)])
        finally:
            b.close()
    for x, y in zip(*got):
        assert np.array_equal(x, y)
