"""PageRank by one cluster: graphs with fewer nodes than CTAs, rows around the
length from which a warp takes them, dangling nodes in both modes, the largest
size of the form and the first beyond it, against power iteration in numpy; a
limit on the iterations; and the network's PageRank feature formed on either
side of the host's range, through p_hat against the oracle's network.

Tolerance: pi to 1e-13 relative to its largest entry (64-bit sums in another
order; the iteration contracts every error but the sum's, which is normalised).
p_hat to 2e-5, the bound of the network's tests.
"""
import numpy as np
import pytest

from oracle import gnn as ognn
from paper_2003_04930_gb300 import QprError, Solver, graphs
from paper_2003_04930_gb300 import qpr as Q

pytestmark = pytest.mark.gpu


def _reference(g, alpha, dangling, iters):
    n = g.n
    keep = (g.src != g.dst) & (g.w != 0)
    src, dst, w = g.src[keep], g.dst[keep], g.w[keep]
    out = np.bincount(src, w, n)
    pi = np.full(n, 1.0 / n)
    for _ in range(iters):
        s = np.bincount(dst, w / out[src] * pi[src], n)
        d = pi[out == 0].sum()
        s += (d - np.where(out == 0, pi, 0.0)) / (n - 1) if dangling == 0 else d / n
        pi = alpha * s + (1 - alpha) * (pi.sum() - pi) / (n - 1)
        pi /= pi.sum()
    return pi


@pytest.mark.parametrize("n", [2, 3, 7, 9, 33, 200, 922, 8192, 8193])
@pytest.mark.parametrize("dangling", [0, 1])
def test_pagerank(n, dangling):
    rng = np.random.default_rng(n)
    m = 1 if n == 2 else 4 * n
    src, dst = rng.integers(0, max(1, n - n // 4), m), rng.integers(0, n, m)
    src[0], dst[0] = 0, n - 1
    for k, links in enumerate((47, 48, 49, 150)):  # rows of about these lengths
        if n >= 200:
            src = np.concatenate([src, rng.permutation(n - n // 4)[:links]])
            dst = np.concatenate([dst, np.full(links, 60 + k)])
    g = graphs.EdgeList(n, src.astype(np.int64), dst.astype(np.int64), rng.lognormal(0.0, 1.0, len(src)))
    with Solver.from_edges(g, alpha=0.85, dangling=dangling, backend=Q.QPR_BACKEND_SPARSE,
                           precision=Q.QPR_FP64) as s:
        pi = s.pagerank()
        iters = s.last_pagerank_iters
        assert iters % 8 == 0 and abs(pi.sum() - 1.0) < 1e-13
        ref = _reference(g, 0.85, dangling, iters)
        assert np.abs(pi - ref).max() <= 1e-13 * ref.max()
        if n > 3:  # (two or three nodes are at their fixed point after three iterations)
            with pytest.raises(QprError) as e:
                s.pagerank(tol=1e-14, max_iter=3)
            assert e.value.status == Q.QPR_E_NOT_CONVERGED


@pytest.mark.parametrize("n", [20, 150, 219, 260, 700])
def test_feature(n):
    g = graphs.heavy_tailed(n, 5)
    net = Q.Gnn(seed=3)
    p = np.random.default_rng(n).random(n)
    p /= p.sum()
    _, _, ref = ognn.loss_and_grad(net.get_params().astype(np.float64), n, g.src, g.dst, g.w, 0.7, 0.85, p)
    np.testing.assert_allclose(net.predict(g, 0.7), ref, rtol=2e-5, atol=0)


@pytest.mark.parametrize("count,batch", [(1, 1), (5, 5), (6, 4)])
def test_training_step_is_the_sum_of_the_graphs_gradients(count, batch):
    # one epoch of uneven graphs in mini-batches, Adam redone from loss_grad's
    # gradients (order of the graphs: the sums differ in rounding only, so
    # entries whose gradient is rounding are left out)
    rng = np.random.default_rng(count)
    data = []
    for k in range(count):
        g = graphs.heavy_tailed([9, 130, 257, 40, 128, 511][k], k) if k else graphs.erdos_renyi(9, 0.4, 1)
        p = rng.random(g.n)
        data.append((g, 0.6, p / p.sum()))
    net = Q.Gnn(seed=2)
    th0 = net.get_params()
    if count == batch:
        grads = [net.loss_grad(*d)[1].astype(np.float64) for d in data]
        losses = [net.loss_grad(*d)[0] for d in data]
        g = sum(grads) / count
        got_loss = net.train(data, epochs=1, batch=batch, lr=1e-3)
        step = th0 - net.get_params()
        big = np.abs(g) > 1e-3 * np.abs(g).max()
        np.testing.assert_allclose(step[big], 1e-3 * g[big] / (np.abs(g[big]) + 1e-8), rtol=1e-3, atol=1e-6)
        assert abs(got_loss[0] - np.mean(losses)) <= 1e-6 * abs(got_loss[0])
    else:
        a = net.train(data, epochs=3, batch=batch, lr=1e-3, seed=4)
        th1 = net.get_params()
        net.set_params(th0)
        b = net.train(data, epochs=3, batch=batch, lr=1e-3, seed=4)
        assert np.array_equal(a, b) and np.array_equal(th1, net.get_params()) and a[-1] < a[0]
