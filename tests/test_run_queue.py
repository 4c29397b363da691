"""How the steps of a call are queued, from the source that the library compiles (no GPU):
launches the first time, a capture when a run of that length comes back, replays from then on,
and an autotuner that times nothing but replays and persistent launches."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def queue(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("runs") / "runs")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I",
                    os.path.join(ROOT, "paper_1211_6932_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "c", "runs.cpp"), "-o", exe], check=True)

    def run(persist, capturing, steps, calls):
        out = subprocess.run([exe] + [str(int(v)) for v in (persist, capturing, steps, calls)],
                             capture_output=True, text=True, check=True).stdout
        return [line.split() for line in out.splitlines()]
    return run


def test_launches_then_captures_then_replays(queue):
    assert queue(False, False, 100, 3) == [["L64", "L32", "L4"],
                                           ["C6", "R6", "C5", "R5", "C2", "R2"],
                                           ["R6", "R5", "R2"]]
    # from either slab: an odd run leaves the state in the other one
    assert queue(False, False, 3, 5) == [["L2", "L1"], ["L2", "L1"], ["C1", "R1", "L1"],
                                         ["C1", "R1", "L1"], ["R1", "L1"]]
    assert queue(False, False, 128, 2) == [["L64", "C6", "R6"], ["R6", "R6"]]


def test_persistent_runs_and_a_callers_capture(queue):
    assert queue(True, False, 100, 2) == [["C6", "R6", "L36"], ["R6", "L36"]]
    assert queue(False, True, 100, 2) == [["C6", "R6", "L32", "L4"], ["R6", "L32", "L4"]]
    assert queue(False, True, 36, 2) == [["L32", "L4"]] * 2


@pytest.mark.parametrize("persist", [False, True])
@pytest.mark.parametrize("steps", [2, 6, 20, 36, 62, 64, 66, 100, 126, 128, 130, 200, 1000])
def test_the_autotuner_times_what_later_runs_do(queue, persist, steps):
    first, second = queue(persist, False, steps, 0)
    assert first == second and first
    for run in first:
        assert run[0] == "R" or (persist and run[0] == "L"), first
