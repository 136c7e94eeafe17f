"""Mini-batches of more graphs than one group of launches takes: the workspace
stays within its bound (320 MiB and the graphs themselves), and the step is that
of the graphs' gradients.

Tolerance: Adam's first step is lr g / (|g| + eps), redone from loss_grad's
gradients; 4000 additions in FP32 leave g to 4000 x 6e-8 of the sum of |g|, so
entries below a hundredth of the largest are left out, the others agree to 1e-3.
"""
import numpy as np
import pytest
import torch

from paper_2003_04930_gb300 import graphs
from paper_2003_04930_gb300 import qpr as Q

pytestmark = pytest.mark.gpu


def test_many_small_graphs():
    rng = np.random.default_rng(1)
    kinds = []
    for k in range(4):
        p = rng.random(16)
        kinds.append((graphs.erdos_renyi(16, 0.3, k), 0.6, p / p.sum()))
    net = Q.Gnn(seed=2)
    grads = [net.loss_grad(*d)[1].astype(np.float64) for d in kinds]
    losses = [net.loss_grad(*d)[0] for d in kinds]
    th0 = net.get_params()
    torch.cuda.synchronize()
    free0, _ = torch.cuda.mem_get_info()
    got = net.train(kinds * 1000, epochs=1, batch=4000, lr=1e-3)
    free1, _ = torch.cuda.mem_get_info()
    assert free0 - free1 <= 400 << 20
    step = th0 - net.get_params()
    g = sum(grads) / 4
    big = np.abs(g) > 1e-2 * np.abs(g).max()
    np.testing.assert_allclose(step[big], 1e-3 * g[big] / (np.abs(g[big]) + 1e-8), rtol=1e-3, atol=1e-6)
    assert abs(got[0] - np.mean(losses)) <= 1e-6 * abs(got[0])
