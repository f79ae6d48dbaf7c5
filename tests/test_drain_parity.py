"""The producers' drain: stages and parities rebuilt from the ring position are
those of the last planes issued, whatever their number and the ring's depth."""
import pytest


@pytest.mark.parametrize("S", [3, 4, 6, 8])
def test_ring_position_gives_the_last_planes(S):
    ps, pph, wrapped = 0, 0, False
    for issued in range(4 * S + 2):
        want = {q % S: q // S & 1 for q in range(max(0, issued - S), issued)}
        seq = (0 if not wrapped else 1 if pph else 2) * S + ps
        assert {q % S: q // S & 1 for q in range(max(0, seq - S), seq)} == want
        assert {s: pph if s < ps else pph ^ 1 for s in range(S) if wrapped or s < ps} == want
        ps += 1
        if ps == S:
            ps, pph, wrapped = 0, pph ^ 1, True
