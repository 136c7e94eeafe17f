"""PageRank stopped by its limit on the iterations, on a graph that has not
converged by then: limits right after a regular check of the L1 change (two
checks in a row), right before one, and on one. Every CTA has to stop at the
limit, so the count is the limit itself and pi the iterate of that number.

Tolerance: pi to 1e-12 of its largest entry (64-bit sums in another order and
another normalisation; with alpha = 1 their rounding is carried along, 1e-16
an iteration at most).
"""
import numpy as np
import pytest

from paper_2003_04930_gb300 import QprError, Solver, graphs
from paper_2003_04930_gb300 import qpr as Q

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [9, 700])
@pytest.mark.parametrize("limit", [1, 7, 8, 9, 15, 17, 1001, 4097])
def test_stops_at_the_limit(n, limit):
    # a path walked both ways: bipartite, so the iterate alternates for good
    i = np.arange(n - 1)
    src, dst = np.concatenate([i, i + 1]), np.concatenate([i + 1, i])
    w = np.random.default_rng(n).lognormal(0.0, 1.0, 2 * (n - 1))
    g = graphs.EdgeList(n, src, dst, w)
    a = np.zeros((n, n))
    a[dst, src] = w
    s = a / a.sum(0)
    ref = np.full(n, 1.0 / n)
    for _ in range(limit):
        ref = s @ ref
        ref /= ref.sum()
    pi = np.zeros(n)
    with Solver.from_edges(g, alpha=1.0, omega=0.8, backend=Q.QPR_BACKEND_SPARSE, precision=Q.QPR_FP64) as sv:
        for _ in range(20 if limit < 100 else 3):
            with pytest.raises(QprError) as e:
                sv.pagerank(tol=1e-14, max_iter=limit, out=pi)
            assert e.value.status == Q.QPR_E_NOT_CONVERGED
            assert np.abs(pi - ref).max() <= 1e-12 * ref.max()
