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
