"""The FP64 dense stage by digit products, entry by entry: states whose
coherences are far below their populations, and every width of digit that a
plan can take (12, 11, 10, 8, 7, 6, 5 bits; which one a graph gets is worked out
here from the planner's rule), one f(rho) against extended precision.

Bound of an entry (u = 2^-53): the commutator part to 8 u of
(1 - omega) [ sum_{k != b} |H_ak Y_kb| + sum_{k != a} |H_bk Y_ka| + |H_ab| |Y_bb - Y_aa| ]
(a product rounds once, then four operations), the dissipator and the gain to
(n + 8) u of their terms (c and the gain are sums), and what the digits leave
out: 5 S 2^(-S b) <= 65 2^-64 for each entry of a row, of the largest entry of
H's row and of Y's column off the diagonal, for both products.
"""
import math

import numpy as np
import pytest
import torch

from paper_2003_04930_gb300 import Solver, graphs
from paper_2003_04930_gb300 import qpr as Q

pytestmark = pytest.mark.gpu
U = 2.0 ** -53
ALPHA, OMEGA = 0.85, 0.6
WIDTHS = [(12, 6), (11, 6), (10, 7), (8, 8), (7, 10), (6, 11), (5, 13)]


def _rows(g):
    """Rows of A and of H as {column: value}."""
    a = [dict() for _ in range(g.n)]
    for j, i, w in zip(g.src.tolist(), g.dst.tolist(), g.w.tolist()):
        if i != j and w:
            a[i][j] = a[i].get(j, 0.0) + w
    h = [dict() for _ in range(g.n)]
    for i, row in enumerate(a):
        for j, w in row.items():
            v = -max(w, a[j].get(i, 0.0))
            h[i][j] = h[j][i] = v
    return a, h


def _width(h):
    """Bits of a digit for these rows of H."""
    vals = [list(r.values()) for r in h]
    units, tops = [], []
    for v in vals:
        for x in v:
            num, den = abs(x).as_integer_ratio()
            units.append((num & -num).bit_length() - 1 - (den.bit_length() - 1))
        tops.append(max((math.frexp(abs(x))[1] for x in v), default=0))
    one = max(t for t, v in zip(tops, vals) if v) - min(units) <= 11
    for b, s in WIDTHS:
        if not one and b > 8:
            continue
        sh, worst = (1 if one else s), 0
        for v, top in zip(vals, tops):
            last = min(units) if one else top - (b - 1) - b * (sh - 1)
            l1 = 0
            for x in v:
                m, e = math.frexp(x)
                n, sft = int(m * 2 ** 53), e - 53 - last
                n = n << sft if sft >= 0 else ((abs(n) + (1 << (-sft - 1))) >> -sft) * (1 if n > 0 else -1)
                for _ in range(sh - 1):
                    n += 1 << (b - 1)
                    l1 += abs((n & ((1 << b) - 1)) - (1 << (b - 1)))
                    n >>= b
                l1 += abs(n)
            worst = max(worst, l1)
        if worst * 2 ** (b - 1) <= 2 ** 24:
            return b
    return 0


def _check(g, rho):
    n = g.n
    a, h = _rows(g)
    with Solver.from_edges(g, alpha=ALPHA, omega=OMEGA, backend=Q.QPR_BACKEND_DENSE) as s:
        out = torch.zeros(n, n, dtype=torch.complex128, device="cuda:0")
        s.rhs(torch.from_numpy(rho).to("cuda:0"), out)
        got = out.cpu().numpy()
    ld = np.longdouble
    re, im = rho.real.astype(ld), rho.imag.astype(ld)
    off = np.abs(rho)
    np.fill_diagonal(off, 0.0)
    p = np.diagonal(rho).real.astype(ld)
    xr, xi, m, drop = np.zeros((n, n), ld), np.zeros((n, n), ld), np.zeros((n, n)), np.zeros((n, n))
    col = off.max(0)
    for i, row in enumerate(h):
        if not row:
            continue
        k, v = np.array(list(row)), np.array(list(row.values()))
        xr[i], xi[i] = v.astype(ld) @ re[k], v.astype(ld) @ im[k]
        m[i] = np.abs(v) @ off[k]
        drop[i] = 65 * 2.0 ** -64 * len(v) * np.abs(v).max() * col
        m[i, k] += np.abs(v) * np.abs(p[k] - p[i]).astype(float) / 2
    out_deg = np.zeros(n)
    for row in a:
        for j, w in row.items():
            out_deg[j] += w
    gain = np.zeros(n, ld)
    dang = out_deg == 0
    for i, row in enumerate(a):
        sp = sum((ld(w) / ld(out_deg[j]) * p[j] for j, w in row.items()), ld(0))
        sp += (p[dang].sum() - (p[i] if dang[i] else 0)) / (n - 1)
        gain[i] = ALPHA * sp + (1 - ld(ALPHA)) * (p.sum() - p[i]) / (n - 1)
    cm = 1 - ld(OMEGA)
    # -i (1 - omega) (X - X^+) + omega (gain - rho), X = H rho
    fr = cm * (xi + xi.T) - ld(OMEGA) * re
    fi = -cm * (xr - xr.T) - ld(OMEGA) * im
    fr[np.diag_indices(n)] += ld(OMEGA) * gain
    bound = float(cm) * (8 * U * (m + m.T) + drop + drop.T) + (n + 8) * U * OMEGA * np.abs(rho)
    bound[np.diag_indices(n)] += (n + 8) * U * OMEGA * np.abs(gain).astype(float)
    assert (np.abs(got.real - fr) <= bound).all()
    assert (np.abs(got.imag - fi) <= bound).all()


def _state(n, scale, seed):
    """Populations of order 1/n, coherences `scale` of that."""
    rho = graphs.random_hermitian(n, seed) * scale / n
    rho[np.diag_indices(n)] = np.random.default_rng(seed).random(n) * 2 / n
    return rho


def _weighted(g, w):
    return graphs.EdgeList(g.n, g.src, g.dst, w)


@pytest.mark.parametrize("scale", [1.0, 1e-5, 1e-8, 1e-14])
@pytest.mark.parametrize("n", [45, 65, 130])
@pytest.mark.parametrize("weights", ["unit", "eighths", "lognormal"])
def test_small_coherences(n, weights, scale):
    g = graphs.erdos_renyi(n, 0.4, n)
    if weights == "lognormal":
        g = _weighted(g, np.random.default_rng(n).lognormal(0.0, 1.0, g.m))
    if weights == "eighths":
        g = _weighted(g, np.random.default_rng(n).integers(1, 30, g.m) / 8)
    _check(g, _state(n, scale, 7))


@pytest.mark.parametrize("bits,n,top", [(12, 130, 1), (11, 130, 150), (10, 130, 300), (8, 161, 900)])
def test_widths_with_whole_weights(bits, n, top):
    g = graphs.erdos_renyi(n, 1.0, 1)
    g = _weighted(g, np.random.default_rng(2).integers(1, top + 1, g.m).astype(float))
    assert _width(_rows(g)[1]) == bits
    _check(g, _state(n, 1e-3, 5))


@pytest.mark.parametrize("bits,n", [(8, 70), (7, 700), (6, 1300), (5, 1951)])
def test_widths_with_a_long_row(bits, n):
    # the last node is linked to all, the others to a few
    g = graphs.heavy_tailed(n, 3)
    keep = (g.src != n - 1) & (g.dst != n - 1)
    rng = np.random.default_rng(4)
    w = rng.lognormal(0.0, 1.0, n - 1)
    if bits == 5:  # digits near their largest: 0.111110111110... in binary
        w[:] = sum(31.0 * 64.0 ** -k for k in range(9)) / 32
    g = graphs.EdgeList(n, np.concatenate([g.src[keep], np.arange(n - 1)]),
                        np.concatenate([g.dst[keep], np.full(n - 1, n - 1)]), np.concatenate([g.w[keep], w]))
    assert _width(_rows(g)[1]) == bits
    _check(g, _state(n, 1e-3, 6))
