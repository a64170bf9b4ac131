"""Model of the pivot kernel's inner ordering for every pivot order k (csrc/pivot.cu, phase 3),
restated from the kernel's slot arithmetic: every pair of columns meets exactly once in a sweep of
p + ceil(p/2) + ... + 1 steps, p = ceil(k/2); no slot is sent two columns in a step; the
block-oriented steps pair every column of one block with every column of the other once."""
import itertools

import pytest


def sweep(k, cross=None):
    p = (k + 1) // 2
    p2 = 1
    while p2 < p:
        p2 *= 2

    def order(i, w):
        return i if p == p2 else int(format(i, "0%db" % (w.bit_length() - 1))[::-1], 2) if w > 1 else 0

    res, trav = [None] * p2, [None] * p2
    first, second = cross if cross else (list(range(min(p, k))), list(range(p, k)))
    for i, c in enumerate(first):
        res[order(i, p2)] = c
    for i, c in enumerate(second):
        trav[order(i, p2)] = c
    met, steps, w, g = [], 0, p2, p
    while w >= (p2 if cross else 1):
        for st in range(g):
            steps += 1
            met += [tuple(sorted((a, b))) for a, b in zip(res, trav) if a is not None and b is not None]
            if st < g - 1:
                out = [None] * p2
                taken = set()
                for q in range(p2):
                    i = order(q & (w - 1), w)
                    d = (q & ~(w - 1)) + order((i + 1) % g, w) if i < g else q
                    assert d not in taken
                    taken.add(d)
                    assert i < g or trav[q] is None
                    out[d] = trav[q]
                trav = out
            elif w > 1 and not cross:
                give = [res[q] if q & (w >> 1) else trav[q] for q in range(p2)]
                for q in range(p2):
                    if q & (w >> 1):
                        res[q] = give[q ^ (w >> 1)]
                    else:
                        trav[q] = give[q ^ (w >> 1)]
        w >>= 1
        g = (g + 1) // 2
    left = sorted(c for c in res + trav if c is not None)
    assert left == sorted(first + second)
    return met, steps


@pytest.mark.parametrize("k", range(2, 65))
def test_every_pair_meets_once(k):
    met, steps = sweep(k)
    assert sorted(met) == list(itertools.combinations(range(k), 2))
    want, p = 0, (k + 1) // 2
    while True:
        want += p
        if p == 1:
            break
        p = (p + 1) // 2
    assert steps == want


@pytest.mark.parametrize("k", range(2, 65))
def test_cross_steps_pair_the_blocks_once(k):
    first, second = list(range((k + 1) // 2)), list(range((k + 1) // 2, k))
    met, steps = sweep(k, (first, second))
    assert sorted(met) == sorted(itertools.product(first, second)) and steps == (k + 1) // 2
