"""The FP64 dense stage by exact digit products on the tensor cores, against
the CPU oracle: sizes around its tiles (128 rows, 32 columns, 64 along k),
unit weights (one digit of H), lognormal weights (every digit of H, each width
of digit by size), the printed diagonal of H (integers of hundreds), a state
whose columns span many orders, non-finite states, and weights no plan covers
(the FP64 tensor kernel serves then).

Tolerances: the product is exact to 2^-64 of a column's largest entry and
rounded once, so one f(rho) agrees with the oracle's to the oracle's own
rounding, nnz(row) ulps of the largest term at most: 1e-13 max|f| for n <=
160 and n / 16 times that beyond, the bounds of the other FP64 forms;
trajectories 1e-11.
"""
import numpy as np
import pytest
import torch

from oracle import Oracle
from paper_2003_04930_gb300 import QprError, Solver, graphs
from paper_2003_04930_gb300 import qpr as Q

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
KW = dict(alpha=0.85, omega=0.6)


def _weighted(n, p, seed):
    g = graphs.erdos_renyi(n, p, seed)
    return graphs.EdgeList(n, g.src, g.dst, np.random.default_rng(seed).lognormal(0.0, 1.0, g.m))


def _rhs(s, rho):
    out = torch.zeros_like(torch.from_numpy(rho)).to(DEV)
    s.rhs(torch.from_numpy(rho).to(DEV), out)
    return out.cpu().numpy()


@pytest.mark.parametrize("n", [2, 31, 45, 63, 64, 65, 96, 127, 128, 129, 160, 257, 500])
@pytest.mark.parametrize("graph", ["unit", "diagonal", "weights"])
def test_rhs(n, graph):
    g = _weighted(n, 0.4, n) if graph == "weights" else graphs.erdos_renyi(n, 0.4, n)
    kw = dict(KW, h_diag=1 if graph == "diagonal" else 0)
    rho = graphs.random_hermitian(n, 7)
    ref = Oracle.from_edges(g, **kw).rhs(rho)
    with Solver.from_edges(g, backend=Q.QPR_BACKEND_DENSE, **kw) as s:
        f = _rhs(s, rho)
        r = s.residual(torch.from_numpy(rho).to(DEV))
    assert np.abs(f - ref).max() <= 1e-13 * max(1.0, np.abs(ref).max()) * max(1, n / 16)
    assert np.abs(f - f.conj().T).max() == 0.0
    assert abs(r - np.linalg.norm(ref)) <= 1e-12 * np.linalg.norm(ref)


@pytest.mark.parametrize("n,graph", [(50, "unit"), (130, "weights"), (300, "unit")])
def test_trajectory(n, graph):
    g = _weighted(n, 0.3, 1) if graph == "weights" else graphs.erdos_renyi(n, 0.3, 1)
    rho0 = graphs.random_density(n, 3, rank=2)
    with Solver.from_edges(g, **KW) as s:
        dt = min(0.01, 0.9 * s.max_stable_dt)
        d = torch.from_numpy(rho0.copy()).to(DEV)
        s.evolve(d, dt, 100)
        got = d.cpu().numpy()
    ref = Oracle.from_edges(g, **KW).evolve(rho0, dt, 100)
    assert np.abs(got - got.conj().T).max() == 0.0
    assert np.linalg.norm(got - ref) <= 1e-11


def test_wide_range_and_small_columns():
    # populations over 12 orders, coherences to match: every column is exact to its own largest entry
    n = 96
    g = graphs.erdos_renyi(n, 0.4, 3)
    d = 10.0 ** -np.linspace(0, 12, n)
    rho = graphs.random_hermitian(n, 2) * np.sqrt(np.outer(d, d))
    rho /= np.trace(rho).real
    ref = Oracle.from_edges(g, **KW).rhs(rho)
    with Solver.from_edges(g, backend=Q.QPR_BACKEND_DENSE, **KW) as s:
        f = _rhs(s, rho)
    assert np.abs(f - ref).max() <= 1e-13 * np.abs(ref).max()
    # the far corner: its sums reach no large entry of the state only through H
    col = np.abs(rho).max(0)
    assert (np.abs(f - ref) <= 1e-13 * n * (col[None, :] + col[:, None])).all()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_state(bad):
    rho = graphs.maximally_mixed(70)
    rho[3, 2] = rho[2, 3] = bad
    with Solver.from_edges(graphs.erdos_renyi(70, 0.4, 1), **KW) as s:
        with pytest.raises(QprError) as e:
            s.evolve(torch.from_numpy(rho).to(DEV), 0.005, 10)
    assert e.value.status == Q.QPR_E_NONFINITE


def test_weights_without_a_plan():
    g = graphs.erdos_renyi(80, 0.4, 1)
    w = g.w.copy()
    w[::7] = 1e-250
    g = graphs.EdgeList(g.n, g.src, g.dst, w)
    rho = graphs.random_hermitian(80, 7)
    ref = Oracle.from_edges(g, **KW).rhs(rho)
    with Solver.from_edges(g, backend=Q.QPR_BACKEND_DENSE, **KW) as s:
        f = _rhs(s, rho)
    assert np.abs(f - ref).max() <= 5e-13 * max(1.0, np.abs(ref).max())
