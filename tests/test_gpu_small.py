"""FP64 RK4 of small problems (one cluster, a block of steps per launch)
against the CPU oracle, at the sizes where it can go wrong: fewer elements
than a warp's octets, one and two nodes per lane in the trace, the largest
size of the form and the first beyond it; both diagonal and dangling modes;
more steps than one launch runs.

Tolerance: FP64 on both sides, other summation orders only; 1e-11 in the
Frobenius norm over 150 steps, the bound the FP64 forms are held to for
degenerate cases, and 1e-10 over 2100 steps.
"""
import numpy as np
import pytest
import torch

from oracle import Oracle
from paper_2003_04930_gb300 import QprError, Solver, graphs
from paper_2003_04930_gb300 import qpr as Q

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _graph(n):
    return graphs.heavy_tailed(n, n) if n > 8 else graphs.erdos_renyi(n, 0.6, 2)


def _evolve(s, rho0, dt, steps):
    d = torch.from_numpy(rho0.copy()).to(DEV)
    s.evolve(d, dt, steps)
    return d.cpu().numpy()


@pytest.mark.parametrize("n", [2, 3, 7, 8, 9, 31, 32, 33, 43, 44, 45])
@pytest.mark.parametrize("h_diag,dangling", [(0, 0), (1, 1)])
def test_trajectory(n, h_diag, dangling):
    kw = dict(alpha=0.85, omega=0.6, h_diag=h_diag, dangling=dangling)
    g = _graph(n)
    rho0 = graphs.random_density(n, 3)
    with Solver.from_edges(g, **kw) as s:
        dt = min(0.01, 0.9 * s.max_stable_dt)
        got = _evolve(s, rho0, dt, 150)
    ref = Oracle.from_edges(g, **kw).evolve(rho0, dt, 150)
    assert np.abs(got - got.conj().T).max() == 0.0
    assert abs(np.trace(got).real - 1.0) < 1e-13
    assert np.linalg.norm(got - ref) <= 1e-11


@pytest.mark.parametrize("steps", [0, 1, 1024, 1025, 2100])
def test_blocks_of_steps(steps):
    g = graphs.erdos_renyi(9, 0.4, 1)
    rho0 = graphs.random_density(9, 3)
    with Solver.from_edges(g, alpha=0.85, omega=0.5) as s:
        got = _evolve(s, rho0, 0.01, steps)
    ref = Oracle.from_edges(g, alpha=0.85, omega=0.5).evolve(rho0, 0.01, steps)
    assert np.linalg.norm(got - ref) <= 1e-10


@pytest.mark.parametrize("n", [16, 44])
def test_steady_state_and_limits(n):
    g = graphs.heavy_tailed(n, 5)
    ref, steps, _, _ = Oracle.from_edges(g, alpha=0.85, omega=0.8).steady_state(graphs.maximally_mixed(n), 0.01, 1e-8, 100000)
    with Solver.from_edges(g, alpha=0.85, omega=0.8) as s:
        d = torch.from_numpy(graphs.maximally_mixed(n)).to(DEV)
        st = s.steady_state(d, 0.01, 1e-8, 100000)
        assert st["converged"] == 1 and st["residual"] < 1e-8 and abs(st["steps"] - steps) <= 1
        assert np.linalg.norm(d.cpu().numpy() - ref) <= 1e-9
        r = s.residual(d)
        assert abs(r - st["residual"]) <= 1e-6 * r
        d = torch.from_numpy(graphs.maximally_mixed(n)).to(DEV)
        st = s.steady_state(d, 0.01, 1e-8, 7, check=False)
        assert st["status"] == Q.QPR_E_NOT_CONVERGED and st["steps"] == 7
        bad = graphs.maximally_mixed(n)
        bad[1, 0] = bad[0, 1] = np.nan
        with pytest.raises(QprError) as e:
            s.evolve(torch.from_numpy(bad).to(DEV), 0.01, 10)
        assert e.value.status == Q.QPR_E_NONFINITE
