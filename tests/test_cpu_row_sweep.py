"""CPU replica of the row sweep's index arithmetic (csrc/hm_row.cuh, tables of csrc/basis.cu): every
exchange target of every state of small sectors against brute-force numbering, and every table and
slot access inside its array."""
import itertools

import numpy as np
import pytest


def states_in_order(N, S2, A):
    """Digit tuples (a_0..a_{N-1}) of the sector, position N-1 most significant."""
    return sorted((a for a in itertools.product(range(S2 + 1), repeat=N) if sum(a) == A), key=lambda a: a[::-1])


def tables(N, S2, A):
    D = np.zeros((N + 1, S2 * N + 1), dtype=object)
    D[0, 0] = 1
    for k in range(1, N + 1):
        for a in range(S2 * k + 1):
            D[k, a] = sum(D[k - 1, a - n] for n in range(S2 + 1) if 0 <= a - n <= S2 * (k - 1))
    d = lambda k, a: D[k, a] if 0 <= a <= S2 * k else 0
    W = S2 + 2
    cd = np.zeros((N, A + 1, W), dtype=object)
    for p in range(N):
        for S in range(A + 1):
            if S <= S2 * (p + 1) and A - S <= S2 * (N - 1 - p):
                c = 0
                for a in range(S2 + 2):
                    cd[p, S, a] = c
                    if a <= S2:
                        c += d(p, S - a)
    ef = np.zeros((N, A + 1, W, 4), dtype=object)
    g = np.zeros((N, A + 1, W, 2), dtype=object)
    for p in range(1, N):
        for S in range(A + 1):
            for a in range(min(S, S2) + 1):
                c = cd[p, S, a]
                if S < A:
                    if a < S2:
                        ef[p, S, a, 0] = cd[p, S + 1, a + 1] - c
                    g[p, S, a, 0] = cd[p, S + 1, a] - c
                if a >= 1:
                    ef[p, S, a, 1] = cd[p, S, a - 1] - c
                if S >= 1:
                    if a >= 1:
                        ef[p, S, a, 2] = cd[p, S - 1, a - 1] - c
                    g[p, S, a, 1] = cd[p, S - 1, a] - c
                if a < S2:
                    ef[p, S, a, 3] = cd[p, S, a + 1] - c
    return cd, ef, g


def slots_of(N, bonds):
    last = [min([p for p, q in bonds if q == s], default=N) for s in range(N)]
    free, slot, n = [], [None] * N, 0
    for r in range(N - 1, -1, -1):
        if last[r] < r:
            if not free:
                free.append(n)
                n += 1
            slot[r] = free.pop()
        free += [slot[q] for q in range(r + 1, N) if last[q] == r]
    return slot, n


@pytest.mark.parametrize("N,S2,A", [(6, 1, 3), (7, 1, 2), (9, 1, 4), (5, 2, 5), (6, 2, 3), (5, 3, 7), (6, 3, 9), (4, 4, 8),
                                    (4, 5, 9), (4, 6, 11), (3, 7, 10), (5, 3, 0), (5, 3, 15), (2, 7, 7)])
def test_sweep_targets(N, S2, A):
    states = states_in_order(N, S2, A)
    index = {a: i for i, a in enumerate(states)}
    cd, ef, g = tables(N, S2, A)
    bonds = sorted(itertools.combinations(range(N), 2)) + [(0, N - 1)]       # all pairs, one of them twice
    slot, nslots = slots_of(N, bonds)
    assert nslots <= N
    for i, a in enumerate(states):
        S, res, qp, qm = A, i, 0, 0
        held = [None] * nslots
        digits = [None] * N
        for r in range(N - 1, -1, -1):
            assert 0 <= S <= A
            if r > 0:
                d = sum(cd[r, S, k] <= res for k in range(1, S2 + 1))
                res -= cd[r, S, d]
            else:
                d = S
            digits[r] = d
            assert d <= S2
            e, gg = ef[r, S, d], g[r, S, d]
            lp, lm = i + e[0] + qp, i + e[2] + qm
            qp += gg[0]
            qm += gg[1]
            if slot[r] is not None:
                held[slot[r]] = (r, e[1] - qp, e[3] - qm)
            for p, q in bonds:
                if p != r:
                    continue
                owner, rp, rm = held[slot[q]]
                assert owner == q                                            # not yet overwritten
                for dp, target in ((1, lp + rp), (-1, lm + rm)):
                    b = list(a)
                    b[p] += dp
                    b[q] -= dp
                    if 0 <= b[p] <= S2 and 0 <= b[q] <= S2:
                        assert target == index[tuple(b)]
            S -= d
        assert tuple(digits) == a
