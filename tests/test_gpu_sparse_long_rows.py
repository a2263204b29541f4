"""Sparse graphs with rows far longer than the others: rows on both sides of
the length from which whole warps read them, a few full rows in an otherwise
sparse graph, more long rows than a CTA lists, and more columns per CTA than
it keeps records of. Parallel arcs come with the random columns. Costs equal
the oracle's, or the returned prices certify the matching; all whole numbers."""

import numpy as np
import pytest

import oracle
from paper_1110_6231_gb300 import synth

from test_gpu_sparse import expect_same, gpu_solve, la  # noqa: F401

pytestmark = pytest.mark.gpu


def with_long_rows(n, degree, count, arcs, seed, hi=10_000):
    """synth.sparse_uniform with `arcs` arcs in each of `count` rows."""
    rng = np.random.default_rng(seed)
    rp, cols, costs = synth.sparse_uniform(n, degree, seed)
    parts, at = [], 0
    lengths = np.diff(rp).astype(np.int64)
    for x in np.sort(rng.choice(n, count, replace=False)):
        extra = arcs - int(lengths[x])
        end = int(rp[x + 1])
        parts.append((cols[at:end], costs[at:end]))
        parts.append((rng.integers(0, n, extra), rng.integers(0, hi + 1, extra)))
        lengths[x], at = arcs, end
    parts.append((cols[at:], costs[at:]))
    c, w = (np.concatenate([p[i] for p in parts]).astype(np.int32) for i in (0, 1))
    return np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32), c, w


def certified(la, g):
    sol = gpu_solve(la, *g, want_prices=True)
    assert sol.stats["status"] == la.LA_OK
    assert sol.stats["price_updates"] > 1
    match = sol.match.cpu().numpy()
    assert oracle.sparse_check_matching(*g, match, sol.cost) == 0
    assert oracle.sparse_check_eps_cs(*g, match, sol.prices.cpu().numpy(), 1) == 0


@pytest.mark.parametrize("arcs", [511, 512, 513, 1025, 5000])
def test_rows_around_the_length_read_by_warps(la, arcs):  # noqa: F811
    assert expect_same(la, *with_long_rows(700, 8, 12, arcs, arcs)) is not None


@pytest.mark.parametrize("n,count,arcs", [(16384, 1, 70_000), (20_000, 150, 5000), (8192, 400, 8192)])
def test_long_rows_in_a_sparse_graph(la, n, count, arcs):  # noqa: F811
    certified(la, with_long_rows(n, 8, count, arcs, n))


def test_more_long_rows_than_a_cta_lists(la):  # noqa: F811
    """40,960 rows of 520 arcs: some 270 columns for each of 152 CTAs, of which 256 are listed."""
    rng = np.random.default_rng(3)
    n, d = 40_960, 520
    cols = rng.integers(0, n, (n, d), dtype=np.int32)
    cols[:, 0] = rng.permutation(n)
    certified(la, (np.arange(n + 1, dtype=np.int32) * d, cols.ravel(), rng.integers(0, 10_001, n * d, dtype=np.int32)))


def test_more_columns_than_a_cta_records(la):  # noqa: F811
    """Over 4,096 columns per CTA, long rows among them on both sides of that line."""
    certified(la, with_long_rows(700_000, 3, 60, 3000, 11))
