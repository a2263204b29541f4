"""How the sparse solver's end-of-phase rounds decide feasibility, on the CPU.

The zero-cost phase starts with bids alone, where a price drop beyond 4n + 4
proves that no perfect matching exists. Once few rows are free, rounds of an
exact price update and of short bidding chains end the phase: every column is
lifted by min(D, K), D its distance to a free column in the residual graph and
K the largest distance of a free row. Columns that reach no free column rise
by K in every round, which the path argument behind 2n - 1 says nothing about,
so no price threshold may decide there. What decides is reachability itself: a
free row that reaches no free column has no augmenting path, so no perfect
matching exists; as long as every free row reaches one, the rounds go on.

Restated here in plain Python with the free rows' order and the hand-off drawn
at random. Nothing touches a GPU or shares code with the CUDA path."""

import random

from test_feasibility_bound import _feasible, _random_graph

FAR = 10**9


def _bid(x, rows, q, holder):
    """One double push of row x on zero costs at eps = 1; the row left without a column, or None."""
    values = sorted((q[y], y) for y in rows[x])
    w = values[0][1]
    q[w] = (values[1][0] if len(values) > 1 else values[0][0]) + 1
    out, holder[w] = holder[w], x
    return None if out < 0 else out


def _distances(n, rows, q, holder):
    """Least residual length from each column to a free column (Bellman-Ford)."""
    D = [FAR if holder[y] >= 0 else 0 for y in range(n)]
    while True:
        moved = False
        for y in range(n):
            for z in rows[holder[y]] if holder[y] >= 0 else ():
                if z != y and D[z] < FAR:
                    length = q[z] - q[y] + 1
                    assert length >= 0, "the matched row is not eps-optimal"
                    if D[z] + length < D[y]:
                        D[y], moved = D[z] + length, True
        if not moved:
            return D


def _rounds(n, rows, rng, chain, bids_first, limit=10**4):
    """"ok" or "infeasible": a phase that starts with bids and ends in rounds."""
    q, holder, free = [0] * n, [-1] * n, list(range(n))
    for _ in range(bids_first):
        if not free:
            break
        out = _bid(free.pop(rng.randrange(len(free))), rows, q, holder)
        if out is not None:
            free.append(out)
    for _ in range(limit):
        if not free:
            return "ok"
        D = _distances(n, rows, q, holder)
        need = [min(q[z] + D[z] for z in rows[x]) - min(q[z] for z in rows[x]) for x in free]
        K = max(need)
        if K > FAR // 2:
            return "infeasible"
        q = [v + min(d, K) for v, d in zip(q, D)]
        rng.shuffle(free)
        left = []
        for x in free:
            for _ in range(chain):
                x = _bid(x, rows, q, holder)
                if x is None:
                    break
            if x is not None:
                left.append(x)
        free = left
    raise AssertionError("the rounds do not end")


def test_reachability_decides():
    rng = random.Random(7)
    counts = {True: 0, False: 0}
    for trial in range(1200):
        n = rng.randint(2, 10)
        rows = [sorted(set(r)) for r in _random_graph(rng, n, rng.randint(1, 4))]
        feasible = _feasible(n, rows)
        counts[feasible] += 1
        for s in range(3):
            r = random.Random(10 * trial + s)
            result = _rounds(n, rows, r, chain=r.choice((1, 2, 8)), bids_first=r.randrange(3 * n))
            assert result == ("ok" if feasible else "infeasible"), (n, rows)
    assert counts[True] > 250 and counts[False] > 250
