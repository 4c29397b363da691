"""Steps inside a caller's own stream capture, where runs of fewer than 64 steps are queued launch
by launch: replaying the caller's graph gives the bits of stepping without it."""
import numpy as np
import pytest

from tests import pairs

pytestmark = pytest.mark.gpu

REPLAYS = 3


def captured(stream, step):
    """The caller's graph of step()."""
    import torch
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream, capture_error_mode="thread_local"):
        step()
    return g


@pytest.mark.parametrize("steps", [2, 36, 62])
@pytest.mark.parametrize("precision,nx,ny,persistent", [
    ("fp32", 64, 48, 0), ("fp32", 600, 40, 0), ("fp64", 60, 31, 0), ("fp64", 200, 31, 0),
    ("fp32", 300, 200, 2)])
def test_captured_steps_of_a_lattice(monkeypatch, precision, nx, ny, persistent, steps):
    import torch
    monkeypatch.setenv("LBM_PERSISTENT", str(persistent))
    c = pairs.case(nx, ny, tr=0.75, sigma=0.114, visc="linear", nu_l=0.05, nu_v=0.3)
    f = pairs.droplet_state(c, vel=0.02)
    with pairs.gpu_lattice(c, precision) as L:
        assert L.persistent == (persistent == 2)
        L.set_populations(f)
        for _ in range(REPLAYS):
            L.step(steps)
        ref = L.get_populations()
    s = torch.cuda.Stream()
    with pairs.gpu_lattice(c, precision, stream=s) as L:
        for _ in range(2):  # outside a capture the handle would replay its own graphs by now
            L.step(steps)
        L.set_populations(f)
        g = captured(s, lambda: L.step(steps))
        with torch.cuda.stream(s):
            for _ in range(REPLAYS):
                g.replay()
        s.synchronize()
        assert np.array_equal(L.get_populations(), ref)


@pytest.mark.parametrize("steps", [6, 62])
def test_captured_steps_of_a_batch_of_two_groups(steps):
    import torch
    from paper_1211_6932_gb300 import Batch
    from tests.test_gpu_batch import CASES, instance, start_fields
    out = []
    for capture in (False, True):
        s = torch.cuda.Stream()
        b = Batch([instance(c) for c in CASES], precision="fp32", tile_threads=64, stream=s)
        assert b.launches_per_step == 2
        for _ in range(2 if capture else 0):
            b.step(steps)
        for i, c in enumerate(CASES):
            b.init_fields(i, *start_fields(c, 20 + i))
        if capture:
            g = captured(s, lambda: b.step(steps))
            with torch.cuda.stream(s):
                for _ in range(REPLAYS):
                    g.replay()
            s.synchronize()
        else:
            for _ in range(REPLAYS):
                b.step(steps)
        out.append([b.get_populations(i) for i in range(len(CASES))])
        b.close()
    for x, y in zip(*out):
        assert np.array_equal(x, y)
