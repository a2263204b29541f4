"""The end-of-phase kernel of the sparse solver (k_sp_finish) at the sizes
where its tiling can go wrong: fewer columns than one 16-column chunk and one
more than it, rows that find no room in a CTA's shared memory, augmenting
paths through the whole graph, parallel arcs, and graphs without a perfect
matching. Costs are compared with the oracle or certified by the returned
prices; everything is whole numbers, so every comparison is exact."""

import numpy as np
import pytest

import oracle
from paper_1110_6231_gb300 import synth

from test_gpu_sparse import expect_same, gpu_solve, la  # noqa: F401
from test_oracle_sparse import to_csr

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 15, 16, 17, 33, 129, 1031])
@pytest.mark.parametrize("degree", [1, 7, 40])
def test_sizes_around_a_chunk(la, n, degree):  # noqa: F811
    expect_same(la, *synth.sparse_uniform(n, min(degree, n), 100 + n))


@pytest.mark.parametrize("n", [40, 700])
def test_paths_through_the_whole_graph(la, n):  # noqa: F811
    """Row x reaches columns x and x + 1 only, row n - 1 columns n - 1 and 0:
    the cheap cycle and the dear diagonal, with every augmenting path long."""
    rng = np.random.default_rng(n)
    arcs = []
    for x in range(n):
        arcs.append((x, x, int(rng.integers(0, 1000))))
        arcs.append((x, (x + 1) % n, int(rng.integers(0, 1000))))
        arcs.append((x, x, int(rng.integers(0, 1000))))       # a parallel arc
    expect_same(la, *to_csr(n, arcs))


def test_rows_beyond_the_shared_memory(la):  # noqa: F811
    """A complete graph of 2,000 rows: 32,000 arcs per 16-column chunk, more
    than a CTA keeps. The prices certify the matching."""
    n = 2000
    C = synth.uniform_costs(n, 0, 10_000, 5)
    rp = (np.arange(n + 1) * n).astype(np.int32)
    cols = np.tile(np.arange(n, dtype=np.int32), n)
    sol = gpu_solve(la, rp, cols, C.ravel(), want_prices=True)
    assert sol.stats["status"] == la.LA_OK
    match = sol.match.cpu().numpy()
    assert oracle.sparse_check_matching(rp, cols, C.ravel(), match, sol.cost) == 0
    assert oracle.sparse_check_eps_cs(rp, cols, C.ravel(), match, sol.prices.cpu().numpy(), 1) == 0


@pytest.mark.parametrize("n", [18, 300])
def test_no_augmenting_path_is_infeasible(la, n):  # noqa: F811
    """Rows 0 and 1 share their only column; the rest has a perfect matching."""
    arcs = [(0, 0, 3), (1, 0, 4)]
    for x in range(2, n):
        arcs += [(x, x, 1), (x, x - 1, 2)]
    rp, cols, costs = to_csr(n, arcs)
    assert gpu_solve(la, rp, cols, costs).stats["status"] == la.LA_ERR_INFEASIBLE


@pytest.mark.parametrize("n", [1, 2, 31, 33, 130, 513, 1026])
def test_certificate_is_the_largest_potential(la, n):  # noqa: F811
    """la_dual_certificate equals plain Bellman-Ford on the residual graph
    (a unique fixed point), for widths with and without 16-byte rows."""
    import torch
    C = synth.geometric_costs(n, 3 + n)
    t = torch.from_numpy(C).cuda()
    match = la.solve(t).match
    u, v = (a.cpu().numpy() for a in la.dual_certificate(t, match))
    m = match.cpu().numpy()
    c, on = C.astype(np.int64), C[np.arange(n), m].astype(np.int64)
    want = np.zeros(n, np.int64)
    for _ in range(n + 2):
        new = np.minimum(want, (c + (want[m] - on)[:, None]).min(0))
        if np.array_equal(new, want):
            break
        want = new
    np.testing.assert_array_equal(v, want)
    np.testing.assert_array_equal(u, on - want[m])


@pytest.mark.parametrize("n", [300, 1001, 2000])
def test_certificate_of_long_chains_and_of_no_optimum(la, n):  # noqa: F811
    """Residual paths through all columns take more sweeps than the epochs with
    several each: row x costs 1 on its own column and 0 on the next, so that
    v(y) = -y. Two rows swapped are no optimum, which n + 2 epochs show."""
    import torch
    C = torch.full((n, n), 2 * n, dtype=torch.int32, device="cuda")
    i = torch.arange(n, device="cuda")
    C[i, i] = 1
    C[i[:-1], i[1:]] = 0
    match = i.to(torch.int32)
    u, v = la.dual_certificate(C, match)
    assert torch.equal(v, -i)
    assert torch.equal(u, 1 + i)
    match[:2] = match[:2].flip(0)
    out = torch.zeros(n, dtype=torch.int64, device="cuda")
    assert la.la_dual_certificate(C, n, match, None, None, out) == la.LA_ERR_INTERNAL
