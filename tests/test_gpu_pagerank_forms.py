"""PageRank of graphs with many links a node, short rows, a few rows of nearly
all nodes, and out-degrees that overflow, on both sides of the line between its
one-cluster and its grid form, against power iteration in numpy.

Tolerance: pi to 1e-13 of its largest entry, as for the sparse graphs.
"""
import numpy as np
import pytest

from paper_2003_04930_gb300 import QprError, Solver, graphs
from paper_2003_04930_gb300 import qpr as Q

pytestmark = pytest.mark.gpu


def _check(g, dangling=0):
    n = g.n
    a = np.zeros((n, n))
    keep = g.src != g.dst
    np.add.at(a, (g.dst[keep], g.src[keep]), g.w[keep])
    with np.errstate(over="ignore"):
        out = a.sum(0)
    s = a / np.where(out > 0, out, 1.0)
    with Solver.from_edges(g, alpha=0.85, omega=1.0, dangling=dangling, backend=Q.QPR_BACKEND_SPARSE,
                           precision=Q.QPR_FP64) as sv:
        pi = sv.pagerank()
        iters = sv.last_pagerank_iters
    ref = np.full(n, 1.0 / n)
    for _ in range(iters):
        d = ref[out == 0].sum()
        new = s @ ref + ((d - np.where(out == 0, ref, 0.0)) / (n - 1) if dangling == 0 else d / n)
        ref = 0.85 * new + 0.15 * (ref.sum() - ref) / (n - 1)
        ref /= ref.sum()
    assert np.abs(pi - ref).max() <= 1e-13 * ref.max()


@pytest.mark.parametrize("n,p", [(300, 0.25), (700, 0.25), (900, 0.25), (1000, 0.25), (2000, 0.25), (2001, 0.02),
                                 (2000, 0.05)])
def test_links_of_equal_rate(n, p):
    g = graphs.erdos_renyi(n, p, 1)
    _check(graphs.EdgeList(n, g.src, g.dst, np.random.default_rng(2).lognormal(0.0, 1.0, g.m)))


@pytest.mark.parametrize("dangling", [0, 1])
@pytest.mark.parametrize("hubs", [3, 60])
def test_rows_of_nearly_all_nodes(hubs, dangling):
    n = 1501
    g = graphs.heavy_tailed(n, 1)
    src = np.concatenate([g.src] + [np.arange(hubs, n - 100)] * hubs)
    dst = np.concatenate([g.dst] + [np.full(n - 100 - hubs, k) for k in range(hubs)])
    _check(graphs.EdgeList(n, src, dst, np.ones(len(src))), dangling)


def test_out_degrees_that_overflow():
    # such a column of S is zero, G loses weight at every iteration, and the
    # change of an iteration (before the division by the sum) stays above tol
    n = 60
    g = graphs.erdos_renyi(n, 0.3, 4)
    w = np.ones(g.m)
    w[g.src < 20] = 1e308
    s = np.zeros((n, n))
    s[g.dst, g.src] = 1.0
    s /= s.sum(0)
    s[:, :20] = 0.0
    ref = np.full(n, 1.0 / n)
    for _ in range(40):
        ref = 0.85 * (s @ ref) + 0.15 * (ref.sum() - ref) / (n - 1)
        ref /= ref.sum()
    pi = np.zeros(n)
    with Solver.from_edges(graphs.EdgeList(n, g.src, g.dst, w), alpha=0.85, omega=1.0,
                           backend=Q.QPR_BACKEND_SPARSE, precision=Q.QPR_FP64) as sv:
        with pytest.raises(QprError) as e:
            sv.pagerank(max_iter=40, out=pi)
    assert e.value.status == Q.QPR_E_NOT_CONVERGED
    assert np.abs(pi - ref).max() <= 1e-13 * ref.max()
