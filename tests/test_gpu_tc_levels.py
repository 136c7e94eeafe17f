"""The dense mixed form's product with one, two and three BF16 planes of H
(unit weights, weights of 10 bits, lognormal weights), at sizes around its 128
x 128 tiles and with fewer and more tiles than SMs, against the oracle.

Tolerance: the trajectory bound of the mixed forms, ||drho||_F <= 1e-6; the
states exactly Hermitian.
"""
import numpy as np
import pytest
import torch

from oracle import Oracle
from paper_2003_04930_gb300 import Solver, graphs
from paper_2003_04930_gb300 import qpr as Q

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,steps", [(2, 40), (127, 40), (128, 40), (129, 40), (300, 40), (1153, 6)])
@pytest.mark.parametrize("levels", [1, 2, 3])
def test_trajectory(n, steps, levels):
    g = graphs.erdos_renyi(n, 0.5 if n < 10 else 0.25, n)
    rng = np.random.default_rng(n)
    w = {1: g.w, 2: 1.0 + rng.integers(0, 1024, g.m) / 1024.0, 3: rng.lognormal(0.0, 1.0, g.m)}[levels]
    g = graphs.EdgeList(n, g.src, g.dst, w)
    rho0 = graphs.random_density(n, 3, rank=min(2, n))
    with Solver.from_edges(g, alpha=0.85, omega=0.7, precision=Q.QPR_MIXED, backend=Q.QPR_BACKEND_DENSE,
                           ref_refresh=16) as s:
        dt = min(0.01, 0.9 * s.max_stable_dt)
        d = torch.from_numpy(rho0.copy()).to("cuda:0")
        s.evolve(d, dt, steps)
        got = d.cpu().numpy()
    ref = Oracle.from_edges(g, alpha=0.85, omega=0.7).evolve(rho0, dt, steps)
    assert np.abs(got - got.conj().T).max() == 0.0
    assert np.linalg.norm(got - ref) <= 1e-6


@pytest.mark.parametrize("n", [50, 129])
@pytest.mark.parametrize("weights", ["unit", "lognormal", "wide"])
def test_rhs_and_steady_state_of_a_mixed_context(n, weights):
    # f(rho) is exact FP64 whatever the precision, by whichever FP64 stage the weights allow
    g = graphs.erdos_renyi(n, 0.4, n)
    rng = np.random.default_rng(n)
    w = {"unit": g.w, "lognormal": rng.lognormal(0.0, 1.0, g.m), "wide": np.where(np.arange(g.m) % 7 == 0, 1e-250, 1.0)}[weights]
    g = graphs.EdgeList(n, g.src, g.dst, w)
    o = Oracle.from_edges(g, alpha=0.85, omega=0.8)
    rho = graphs.random_hermitian(n, 7)
    ref = o.rhs(rho)
    with Solver.from_edges(g, alpha=0.85, omega=0.8, precision=Q.QPR_MIXED, backend=Q.QPR_BACKEND_DENSE) as s:
        out = torch.zeros((n, n), dtype=torch.complex128, device="cuda:0")
        s.rhs(torch.from_numpy(rho).to("cuda:0"), out)
        assert np.abs(out.cpu().numpy() - ref).max() <= 1e-13 * max(1.0, np.abs(ref).max()) * max(1, n / 16)
        d = torch.from_numpy(graphs.maximally_mixed(n)).to("cuda:0")
        st = s.steady_state(d, 0.01, 1e-8, 100000)
        assert st["converged"] == 1 and st["residual"] < 1e-8
        assert abs(s.residual(d) - st["residual"]) <= 1e-6 * st["residual"]
    rref, steps, _, _ = o.steady_state(graphs.maximally_mixed(n), 0.01, 1e-8, 100000)
    assert abs(st["steps"] - steps) <= 1
    p, pr = np.real(np.diag(d.cpu().numpy())), np.real(np.diag(rref))
    assert np.abs(p - pr).max() <= 1e-7 * pr.max()
