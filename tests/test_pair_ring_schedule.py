"""Host replica of the FP32 pair kernel's row ring (no GPU): four slots of nine planes, row j
in slot j mod 4 on row barrier j mod 4; rows 0..3 issued before the loop, row s + 3 after the
row barrier of step s; step s waits for row s + 1 and pulls the planes ahead from row s + 1,
the centre planes from row s, the planes behind from row s - 1, and at a wall row its own
planes ahead and behind.  The planes that no step reads are not copied.  Checked for every
chunk length the kernel can meet, with and without walls."""
import pytest

NS, LEAD = 4, 3


def planes_of(j, nload, walls):
    edge = 1 if walls else 2
    return {"A": j >= edge, "C": 1 <= j < nload - 1, "B": j < nload - edge}


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("nload", list(range(5, 80)) + [203, 204])
def test_four_slot_ring_schedule(nload, walls):
    slot = [{} for _ in range(NS)]   # group -> row whose planes it holds
    phase = [-1] * NS                # the row whose copies a barrier counts
    waited = -1

    def issue(j):
        assert phase[j % NS] <= waited, "barrier reused before its row was waited for"
        phase[j % NS] = j
        have = planes_of(j, nload, walls)
        assert any(have.values())
        for g, on in have.items():
            if on:
                slot[j % NS][g] = j

    def read(g, j):
        assert j <= waited and slot[j % NS].get(g) == j, (g, j)

    last = nload - 2
    for j in range(min(nload, LEAD + 1)):
        issue(j)
    for j in (0, 1):
        assert phase[j % NS] == j
        waited = j
    phase_bit, o_lo = 0, 0  # the kernel's parity bookkeeping, two steps a round
    for s in range(1, last + 1):
        k = (s - 1) % 2
        j = s + 1
        assert phase[j % NS] == j
        assert (phase_bit ^ (1 if o_lo else 0)) == (j // NS) & 1
        waited = j
        behind = [o_lo, o_lo + 1][k]
        centre = [o_lo + 1, 2 - o_lo][k]
        ahead = [2 - o_lo, 3 - o_lo][k]
        assert (behind, centre, ahead) == ((s - 1) % NS, s % NS, (s + 1) % NS)
        read("B", s - 1)
        read("C", s)
        read("A", s + 1)
        if walls:
            read("A", s)
            read("B", s)
        if s + LEAD < nload:  # after the row barrier of step s
            issue(s + LEAD)
        if k == 1:
            phase_bit ^= 1 if o_lo else 0
            o_lo = 2 - o_lo


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_state_file_keeps_the_planes_in_velocity_order(tmp_path, precision):
    """A state file holds plane q of the D2Q9 order as its q-th plane, whatever order the
    planes have in device memory: uniform populations, a different value for each q."""
    import numpy as np
    from tests import pairs
    c = pairs.case(21, 13, tr=0.7, sigma=0.114)
    tw = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)
    f = np.empty((9, 13, 21))
    for q in range(9):
        f[q] = tw[q] * (0.2 + 0.01 * q)
    path = tmp_path / "state"
    with pairs.gpu_lattice(c, precision) as L:
        L.set_populations(f)
        L.save(str(path))
        L.load(str(path))
        assert np.allclose(L.get_populations(), f, rtol=0, atol=1e-7)
    dt = np.float64 if precision == "fp64" else np.float32
    pitch = (21 + 16 + 7) // 8 * 8
    n = 9 * 13 * pitch
    raw = path.read_bytes()
    planes = np.frombuffer(raw[-4 - n * dt().nbytes:-4], dtype=dt).reshape(9, 13, pitch)
    inner = planes[:, :, 8:8 + 21].astype(np.float64)
    shift = (inner - f) / tw[:, None, None]  # -rho_ref (0 in FP64), the same for every plane
    assert np.ptp(shift) < 1e-5
