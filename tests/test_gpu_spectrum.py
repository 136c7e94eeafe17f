"""The spectral spread of H formed on the device (from 8000 nonzeros in a
single problem, 500 in a batch): against numpy's eigenvalues, with rows around
the length a warp takes, the printed diagonal, a weight scale outside the
device form's range; and a batch whose problems stop at different steps (its
lists shrink under one captured graph) against single solves.

Tolerance: 400 power iterations leave the estimate within the 2% margin it
carries above the eigenvalues' distance (never below it by more than 0.5%).
Batch against single solves: bitwise, as in the batch's own tests.
"""
import numpy as np
import pytest
import torch

from paper_2003_04930_gb300 import Solver, graphs
from paper_2003_04930_gb300 import qpr as Q

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,h_diag,scale", [(130, 0, 1.0), (700, 0, 1.0), (700, 1, 1.0), (1001, 0, 1e20)])
def test_spread(n, h_diag, scale):
    g = graphs.erdos_renyi(n, 0.5 if n == 130 else 30.0 / n, 3)
    w = np.random.default_rng(1).lognormal(0.0, 1.0, g.m) * scale
    hub = np.arange(1, 60)
    src, dst = np.concatenate([g.src, hub]), np.concatenate([g.dst, np.zeros(59, dtype=np.int64)])
    g = graphs.EdgeList(n, src, dst, np.concatenate([w, np.full(59, scale)]))
    a = np.zeros((n, n))
    np.add.at(a, (dst, src), g.w)
    np.fill_diagonal(a, 0.0)
    h = -np.maximum(a, a.T)
    if h_diag:
        h -= np.diag(a.sum(0))
    ev = np.linalg.eigvalsh(h)
    with Solver.from_edges(g, alpha=0.85, omega=0.9, h_diag=h_diag, precision=Q.QPR_MIXED,
                           backend=Q.QPR_BACKEND_SPARSE) as s:
        assert np.count_nonzero(h) >= 8000
        r = s.h_spread / (ev[-1] - ev[0])
    assert 0.995 <= r <= 1.03, r


def test_batch_lists_shrink():
    ns = [40, 90, 300, 555, 33, 160, 47]
    omegas = [0.95, 0.5, 0.9, 0.7, 0.6, 0.8, 0.92]
    gs = [graphs.heavy_tailed(n, 20 + k) for k, n in enumerate(ns)]
    rhos = [torch.from_numpy(graphs.maximally_mixed(n)).to("cuda:0") for n in ns]
    _, stats = Q.batch_steady_state(list(zip(gs, omegas, rhos)), tol=1e-6)
    assert len({s["steps"] // 32 for s in stats}) >= 4
    for g, om, rho, st in zip(gs, omegas, rhos, stats):
        with Solver.from_edges(g, alpha=0.85, omega=om, precision=Q.QPR_MIXED, backend=Q.QPR_BACKEND_SPARSE,
                               sparse_form=Q.QPR_SPARSE_FORM_COLUMNS) as s:
            d = torch.from_numpy(graphs.maximally_mixed(g.n)).to("cuda:0")
            one = s.steady_state(d, 0.01, 1e-6, 400000)
        assert one["steps"] == st["steps"] and one["residual"] == st["residual"]
        assert torch.equal(d, rho)
