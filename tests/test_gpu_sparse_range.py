"""Sparse graphs whose scaled costs come near the top of the price field.

la_solve_sparse accepts every graph with (n + 1)(max C - min C) < 2^40. On
graphs whose residual paths are long, a price update's distances are many
times that range: it must not use up the 2^44 price field, so that such a
graph ends in its optimum, as with bids alone, and not in LA_ERR_OVERFLOW. Whole numbers: every comparison is exact."""

import numpy as np
import pytest

import oracle
from paper_1110_6231_gb300 import synth

from test_gpu_sparse import expect_same, gpu_solve, la  # noqa: F401

pytestmark = pytest.mark.gpu


def band(n, hi, seed, width=4):
    """Row x has arcs to columns x .. x + width - 1 (mod n), costs uniform on [0, hi]."""
    rng = np.random.default_rng(seed)
    cols = (np.arange(n)[:, None] + np.arange(width)) % n
    return np.arange(n + 1) * width, cols.ravel(), rng.integers(0, hi + 1, n * width)


@pytest.mark.parametrize("seed", [1, 2, 3])
@pytest.mark.parametrize("n,hi", [(3000, 10**8), (3000, 360_000_000), (6000, 3 * 10**7)])
def test_long_paths_near_the_top_of_the_range(la, n, hi, seed):  # noqa: F811
    rp, cols, costs = band(n, hi, seed)
    assert (n + 1) * int(costs.max() - costs.min()) < 1 << 40
    assert expect_same(la, rp, cols, costs) is not None


def test_the_scan_budget_holds_when_a_solve_starts_again(la):  # noqa: F811
    """At this range the updates are given up and the solve starts again with
    bids alone; it still stops at the budget, and the next call is clean."""
    g = band(3000, 360_000_000, 4)
    need = gpu_solve(la, *g).stats["scans"]
    got = gpu_solve(la, *g, scan_budget=need // 8)
    assert got.stats["status"] == la.LA_ERR_ITER_LIMIT
    assert got.stats["scans"] < need
    assert expect_same(la, *g) is not None


@pytest.mark.parametrize("width,hi", [(2, 1000), (4, 10_000), (8, 1000)])
def test_long_paths_take_few_rounds(la, width, hi):  # noqa: F811
    """Residual paths of thousands of columns: a round's chains must follow
    them to their end, not a fixed number of columns a round (then one update
    for every 256 columns of path, hundreds in all). The prices certify the
    matching."""
    rp, cols, costs = band(30_000, hi, 5, width)
    sol = gpu_solve(la, rp, cols, costs, want_prices=True)
    assert sol.stats["status"] == la.LA_OK
    match = sol.match.cpu().numpy()
    assert oracle.sparse_check_matching(rp, cols, costs, match, sol.cost) == 0
    assert oracle.sparse_check_eps_cs(rp, cols, costs, match, sol.prices.cpu().numpy(), 1) == 0
    assert sol.stats["price_updates"] <= 5 * (sol.stats["phases"] + 1)


@pytest.mark.parametrize("n", [511, 512, 513])
@pytest.mark.parametrize("degree", [1, 2, 8])
def test_both_sides_of_the_line_for_bids_alone(la, n, degree):  # noqa: F811
    """Up to 512 rows, and up to five arcs for two rows, the cost phases run
    without updates; one row or one arc more and they have them."""
    rp, cols, costs = synth.sparse_uniform(n, degree, n)
    sol = expect_same(la, rp, cols, costs)
    updates = n > 512 and 2 * cols.size > 5 * n
    assert sol.stats["refine_launches"] == (2 if updates else 1) * (sol.stats["phases"] + 1) + (not updates)


@pytest.mark.parametrize("kind", ["geometric", "uniform"])
def test_a_missing_matching_is_found_by_one_update(la, kind):  # noqa: F811
    """12 rows that reach only 11 columns, in a large graph: one update shows it,
    not a price war of 4n steps (more than 40 scans a row)."""
    n = 40_000
    rp, cols, costs = synth.sparse_geometric(n, 4) if kind == "geometric" else synth.sparse_uniform(n, 3, 4)
    keep = np.ones(cols.size, dtype=bool)
    keep[:rp[12]] = False
    hall = np.tile(np.arange(11), 12)
    g = (np.concatenate([np.arange(12) * 11, rp[12:] - rp[12] + 132]), np.concatenate([hall, cols[keep]]),
         np.concatenate([np.full(132, 5), costs[keep]]))
    missing = np.setdiff1d(np.arange(n), g[1])     # columns that only the 12 rows had: row n - 1 takes them
    g = (np.concatenate([g[0][:-1], [g[0][-1] + missing.size]]), np.concatenate([g[1], missing]),
         np.concatenate([g[2], np.zeros(missing.size, dtype=g[2].dtype)]))
    sol = gpu_solve(la, *g)
    assert sol.stats["status"] == la.LA_ERR_INFEASIBLE
    assert sol.stats["price_updates"] >= 1
    assert sol.stats["scans"] < 10 * n
