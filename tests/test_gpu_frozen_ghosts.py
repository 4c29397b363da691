"""A frozen instance of a batch keeps its fields whatever the others do: full-width strips leave
its periodic ghost columns stale, and a tiling chosen later may sweep it in strips, which read
them, from either slab."""
import numpy as np
import pytest

from tests import pairs
from tests.test_gpu_batch import instance, start_fields

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,widths,tile,tol", [
    ("fp64", (100, 300), "64,1,8", 1e-13), ("fp32", (200, 300), "32,2,8", 1e-6),
    ("fp32", (200, 300), "64,1,8", 1e-6)])
def test_frozen_instance_after_a_change_of_tiling(monkeypatch, precision, widths, tile, tol):
    """The fields at the freeze, read back after each step under the new tiling: the same state
    in another order of summation, so equal to a few roundings of the storage type."""
    from paper_1211_6932_gb300 import Batch
    cs = [pairs.case(nx, 40, tr=0.75, sigma=0.114) for nx in widths]
    monkeypatch.delenv("LBM_TILE", raising=False)
    b = Batch([instance(c, layout="rows") for c in cs], precision=precision)
    try:
        for i, c in enumerate(cs):
            rho, ux, uy = start_fields(c, 30 + i)
            shift = c["nx"] // 2  # the droplet across the periodic edge
            b.init_fields(i, np.roll(rho, shift, 1), ux, uy)
        b.step(33)
        b.retire(0)
        ref = b.moments(0)
        monkeypatch.setenv("LBM_TILE", tile)
        assert b.autotune(steps=2)[:3] == tuple(int(v) for v in tile.split(","))
        for _ in range(4):
            got = b.moments(0)
            for k in ("rho", "ux", "uy"):
                assert np.max(np.abs(got[k] - ref[k])) <= tol, k
            b.step(1)
    finally:
        b.close()
