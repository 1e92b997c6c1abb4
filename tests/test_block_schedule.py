"""The block schedule of a clustered slice SVT (fill_schedule of slice_svt.cu, restated): the
pairs of a round are those of the circle method, each on one CTA, and from one round to the next
every CTA keeps exactly one of its two blocks -- so that the other is all it has to trade."""
import pytest


def circle_pair(r, slot, nb):
    if slot == 0:
        return nb - 1, r
    return (r + slot) % (nb - 1), (r - slot + nb - 1) % (nb - 1)


def schedule(C):
    nb, at, rounds = 2 * C, {}, []
    for r in range(nb - 1):
        pairs = [circle_pair(r, s, nb) for s in range(C)]
        cta = [s if r == 0 else -1 for s in range(C)]
        for c in range(C if r else 0):
            cur, done = c, c in cta
            while not done:
                s = next(i for i in range(C) if cta[i] < 0 and cur in (at[pairs[i][0]], at[pairs[i][1]]))
                cta[s] = cur
                cur = at[pairs[s][1]] if at[pairs[s][0]] == cur else at[pairs[s][0]]
                done = cur == c
        rounds.append({cta[s]: pairs[s] for s in range(C)})
        at = {b: cta[s] for s in range(C) for b in pairs[s]}
    return rounds


@pytest.mark.parametrize("C", [1, 2, 4, 8])
def test_one_block_stays(C):
    rounds = schedule(C)
    met = [frozenset(p) for held in rounds for p in held.values()]
    assert len(met) == len(set(met)) == C * (2 * C - 1)       # every pair of blocks, once
    assert rounds[0] == {c: circle_pair(0, c, 2 * C) for c in range(C)}
    for old, new in zip(rounds, rounds[1:]):
        assert sorted(new) == list(range(C))
        assert all(len(set(old[c]) & set(new[c])) == 1 for c in range(C))
