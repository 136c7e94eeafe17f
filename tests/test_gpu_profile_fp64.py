"""qpr_profile_step times what a solve of an FP64 context launches: the digit
products' three launches a stage without a gain kernel beside them, the gain and
stage kernels where no plan of digits covers the weights, and for a small
problem the one launch that runs many steps. rho is left alone.
"""
import numpy as np
import pytest
import torch

from paper_2003_04930_gb300 import Solver, graphs
from paper_2003_04930_gb300 import qpr as Q

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,weights,steps,launches,gain", [
    (130, "unit", 3, 12, False), (130, "wide", 3, 8, True), (45, "unit", 1, 12, False), (16, "unit", 1, 0, False),
    (16, "unit", 1025, 0, False), (44, "unit", 3, 0, False)])
def test_launches(n, weights, steps, launches, gain):
    g = graphs.erdos_renyi(n, 0.5, 1)
    if weights == "wide":
        w = g.w.copy()
        w[::7] = 1e-250
        g = graphs.EdgeList(n, g.src, g.dst, w)
    rho = torch.from_numpy(graphs.maximally_mixed(n)).to("cuda:0")
    before = rho.clone()
    with Solver.from_edges(g, alpha=0.85, omega=0.8, backend=Q.QPR_BACKEND_DENSE) as s:
        dt = min(0.01, s.max_stable_dt)
        p = s.profile_step(rho, dt, steps)
        s.evolve(rho, dt, 3)
        ref = before.clone()
        s.evolve(ref, dt, 3)
    assert torch.equal(rho, ref)  # evolve from an unchanged rho
    assert p["launches_per_step"] == launches and (p["gain_ms"] > 0) == gain
    assert p["product_ms"] > 0 and p["epilogue_ms"] == 0 and p["refresh_ms"] == 0
    per_step = p["product_ms"] if n <= 44 else 4 * (p["product_ms"] + p["gain_ms"])
    np.testing.assert_allclose(p["step_ms"], per_step, rtol=1e-9)
