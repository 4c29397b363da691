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
