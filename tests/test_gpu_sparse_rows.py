"""The FP64 sparse stage at the row lengths where its work is dealt out
differently (rows of at most 96 nonzeros to single warps, longer ones to a
whole CTA; 32 entries at a time, four to a batch), against the oracle: a hub
of exactly `links` links among nodes of a few, two hubs in one tile, rows
without entries.

Tolerance: one f(rho) to 1e-13 max|f| n / 16, as for the other FP64 forms
(summation order only).
"""
import numpy as np
import pytest
import torch

from oracle import Oracle
from paper_2003_04930_gb300 import Solver, graphs
from paper_2003_04930_gb300 import qpr as Q

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("links", [1, 3, 4, 5, 31, 32, 33, 95, 96, 97, 128, 200])
@pytest.mark.parametrize("hubs", [1, 2])
def test_hub_rows(links, hubs):
    n = 230
    rng = np.random.default_rng(links)
    src, dst = [], []
    for h in range(hubs):
        to = rng.permutation(np.arange(hubs, n))[:links]
        src += [h] * links
        dst += list(to)
    src += [150, 151, 152]
    dst += [151, 152, 153]
    g = graphs.EdgeList(n, np.array(src), np.array(dst), rng.lognormal(0.0, 1.0, len(src)))
    kw = dict(alpha=0.85, omega=0.6)
    rho = graphs.random_hermitian(n, 7)
    ref = Oracle.from_edges(g, **kw).rhs(rho)
    with Solver.from_edges(g, backend=Q.QPR_BACKEND_SPARSE, **kw) as s:
        out = torch.zeros((n, n), dtype=torch.complex128, device="cuda:0")
        s.rhs(torch.from_numpy(rho).to("cuda:0"), out)
        f = out.cpu().numpy()
    assert np.abs(f - ref).max() <= 1e-13 * max(1.0, np.abs(ref).max()) * n / 16
    assert np.abs(f - f.conj().T).max() == 0.0
