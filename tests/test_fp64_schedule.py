"""The FP64 stage kernel's diagonal schedule (PairSched in esdg_kernels.cuh and
the host's pair_operator_t), replayed on the CPU for every rule it takes (up to
32 volume points): every non-zero pair of Q_skew is evaluated once, by the lane
of its volume row, and reaches its other row once, from the lane whose row that
row's receiver reads; likewise for the nodes of the DG-SBP rules (SbpSched, no
separate face rows).
"""

import pytest

POINTS = {"symmetric": {1: 3, 2: 6, 3: 12, 4: 16, 5: 25}, "collapsed": {N: (N + 1) ** 2 for N in range(1, 6)},
          "sbp": {1: 6, 2: 10, 3: 18, 4: 22, 5: 34}}


@pytest.mark.parametrize("rule", ["collapsed", "symmetric", "sbp"])
@pytest.mark.parametrize("N", [1, 2, 3, 4, 5])
def test_diagonal_schedule_covers_each_pair_once(N, rule):
    V, F = POINTS[rule][N], 0 if rule == "sbp" else 3 * (N + 1)
    L = max(V, F)
    if L > 32:
        pytest.skip("row-major pieces instead of diagonals")
    halves = 2 if L <= 16 else 1
    lanes = 32 // halves
    SVV = V // 2
    SVV0, SVF0 = -(-SVV // halves), -(-L // halves) if F else 0
    evaluated, received = {}, {}

    def stored(j, m):
        evaluated[(j, m)] = evaluated.get((j, m), 0) + 1

    for hf in range(halves):
        for k in range(SVV0):
            d = 1 + k + SVV0 * hf
            sent = {}
            for j in range(lanes):  # the host's entries: zero where there is no pair
                if j < V and d <= SVV and not (2 * d == V and j >= V // 2):
                    stored(j, (j + d) % V)
                    sent[j] = (j + d) % V
                m = j + d - (V if j + d >= V else 0)  # the kernel's partner record
                assert (m if j < V else 0) < V + F
            for j in range(V):  # lanes past V receive into sums that are not used
                src = j - d + (V if j < d else 0)
                assert 0 <= src < V
                if src in sent:
                    assert sent[src] == j
                    received[(src, j)] = received.get((src, j), 0) + 1
        for k in range(SVF0):
            t = k + SVF0 * hf
            sent = {}
            for j in range(lanes):
                if j < V and t < L and (j + t) % L < F:
                    stored(j, V + (j + t) % L)
                    sent[j] = (j + t) % L
                f = j + t - (L if j + t >= L else 0)
                assert j >= L or 0 <= f < L
            for j in range(F):
                src = j - t + (L if j < t else 0)
                assert 0 <= src < lanes
                if src in sent:
                    assert sent[src] == j
                    received[(src, V + j)] = received.get((src, V + j), 0) + 1
    want = {frozenset((l, m)) for l in range(V) for m in range(V + F) if m != l}
    assert {frozenset(p) for p in evaluated} == want and len(evaluated) == len(want)
    assert all(n == 1 for n in evaluated.values())
    assert received == {p: 1 for p in evaluated}
