"""The substeps of a problem in a batch are those it takes alone, also where dt
is an exact multiple of the largest stable step, or the next number above one:
there any difference in the last bit of the spectral spread changes the number
of substeps, and with it every bit of the result. Graphs on both sides of the
sizes where the spread is formed on the device, in batches small and large.
"""
import numpy as np
import pytest
import torch

from paper_2003_04930_gb300 import Solver, graphs
from paper_2003_04930_gb300 import qpr as Q

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,copies", [(16, 6), (60, 6), (150, 6), (250, 5), (250, 4), (400, 40), (700, 5)])
def test_substeps_at_the_boundary(n, copies):
    g = graphs.heavy_tailed(n, n)
    with Solver.from_edges(g, alpha=0.85, omega=0.9, precision=Q.QPR_MIXED, backend=Q.QPR_BACKEND_SPARSE,
                           sparse_form=Q.QPR_SPARSE_FORM_COLUMNS) as s:
        for dt in (2 * s.max_stable_dt, np.nextafter(2 * s.max_stable_dt, np.inf)):
            one = torch.from_numpy(graphs.maximally_mixed(n)).to("cuda:0")
            st = s.steady_state(one, dt, 1e-4, 100000)
            rhos = [torch.from_numpy(graphs.maximally_mixed(n)).to("cuda:0") for _ in range(copies)]
            _, stats = Q.batch_steady_state([(g, 0.9, r) for r in rhos], dt=dt, tol=1e-4)
            assert st["substeps_m"] == (2 if dt == 2 * s.max_stable_dt else 3)
            for r, b in zip(rhos, stats):
                assert b["substeps_m"] == st["substeps_m"] and b["steps"] == st["steps"]
                assert torch.equal(r, one)
