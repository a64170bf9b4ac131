"""The pair cache as the step kernels keep it (csrc/pair_cache.cuh), restated on the CPU.

The Gram kernel and the pivot look a pair up (pair_known); whoever decides it records it in the same
step (pair_record): the pivot when nothing rotates or it forms V_P itself, the kernel of phase 4 when
the phases run apart, the FP64 pivot for a block handed over.  A failed block and a hand-over that no
FP64 pivot takes (FP32 sweeps of the mixed mode) are not recorded and are looked at again.  With the
outcome of a pair a pure function of its two blocks, the cached run takes the same decisions.
"""
import itertools

import pytest

from test_pair_cache_model import h, schedule


def outcome(cp, cq, tol):
    x = h(cp, cq) % 1000
    return "none" if x >= tol else ("rotate", "rotate", "handover", "fail")[h(cq, cp) % 4]


def run(nb, ordering, tols, cached, fallback, fail):
    steps = [[(int(p), int(q)) for p, q in s] for s in schedule(nb, ordering)]
    content, bver = [h(nb, b) for b in range(nb)], [0] * nb
    pver = [[(-1, -1, -1, -1)] * (nb // 2) for _ in steps]
    decisions, evaluated = [], 0

    def known(s, i):
        p, q, vp, vq = pver[s][i]
        return (p, q) == steps[s][i] and p >= 0 and vp == bver[p] and vq == bver[q]

    def record(s, i, rotated):
        p, q = steps[s][i]
        if rotated:
            bver[p] += 1
            bver[q] += 1
        pver[s][i] = (p, q, -1 if rotated else bver[p], bver[q])

    for sw, tol in enumerate(tols):
        for s, pairs in enumerate(steps):
            skip = {}
            for i, (p, q) in enumerate(pairs):  # the pairs of a step are disjoint: any order
                if cached and known(s, i):
                    skip[i] = 1
                    decisions.append((sw, s, i, 1))
                    continue
                evaluated += 1
                o = outcome(content[p], content[q], tol)
                if o == "none":
                    skip[i] = 1
                    record(s, i, False)
                elif o == "rotate":
                    skip[i] = 0
                    record(s, i, True)
                else:
                    skip[i] = 2  # handed over; the FP64 pivot rotates it or finds it singular
                    if fallback:
                        if o == "handover" or not fail:
                            skip[i] = 0
                            record(s, i, True)
                        else:
                            skip[i] = 1
                decisions.append((sw, s, i, skip[i]))
            for i, (p, q) in enumerate(pairs):
                if skip[i] == 0:
                    content[p], content[q] = h(content[p], content[q], 1), h(content[p], content[q], 2)
    return decisions, evaluated


@pytest.mark.parametrize("ordering", ["round_robin", "modulus", "modulus_mod"])
@pytest.mark.parametrize("nb", [2, 4, 8, 16, 30])
def test_recorded_pairs_take_the_same_decisions(nb, ordering):
    tols = [900, 600, 300, 100, 30, 10, 0, 0]
    for fallback, fail in itertools.product((False, True), repeat=2):
        ref, n_ref = run(nb, ordering, tols, False, fallback, fail)
        got, n_got = run(nb, ordering, tols, True, fallback, fail)
        assert got == ref
        assert n_got <= n_ref - sum(len(s) for s in schedule(nb, ordering))  # the last sweep is all known
