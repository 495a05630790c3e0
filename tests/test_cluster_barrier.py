"""The barrier of the panel kernel's cluster form, restated on the CPU: every CTA has a counter of
anonymous arrivals per mbarrier, each CTA arrives at every CTA, and arrivals land in any order
that the dependencies allow.  No CTA may pass a phase before every arrival for it has landed."""
import random

import pytest


def sound(ctas, phases, nbar, rng):
    count, done = ([[0] * nbar for _ in range(ctas)] for _ in range(2))
    landed = [[0] * phases for _ in range(ctas)]
    phase = [0] * ctas
    flight = [(d, 0) for _ in range(ctas) for d in range(ctas)]
    while flight:
        d, p = flight.pop(rng.randrange(len(flight)))
        b = p % nbar
        landed[d][p] += 1
        count[d][b] += 1
        if count[d][b] == ctas:
            count[d][b] = 0
            done[d][b] += 1
        for c in range(ctas):
            while phase[c] < phases and done[c][phase[c] % nbar] > phase[c] // nbar:
                if landed[c][phase[c]] < ctas:
                    return False
                phase[c] += 1
                if phase[c] < phases:
                    flight += [(e, phase[c]) for e in range(ctas)]
    return all(p == phases for p in phase)


@pytest.mark.parametrize("ctas", [2, 3, 4, 8, 16])
def test_two_alternating_mbarriers(ctas):
    rng = random.Random(ctas)
    assert all(sound(ctas, 12, 2, rng) for _ in range(3200 // ctas ** 2))


def test_one_mbarrier_is_not_enough():
    rng = random.Random(1)
    assert not all(sound(3, 12, 1, rng) for _ in range(50))
