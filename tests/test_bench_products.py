"""bench.bf16_products: the products that the split-BF16 stage forms, by the BF16
planes of H that are not zero.
"""
import numpy as np
import pytest

import bench
from paper_2003_04930_gb300 import graphs


@pytest.mark.parametrize("weights,products", [("unit", 3), ("none", 3), ("bytes", 3), ("words", 5), ("lognormal", 6), ("sums", 5)])
def test_products(weights, products):
    g = graphs.erdos_renyi(40, 0.4, 1)
    rng = np.random.default_rng(2)
    w = {"unit": g.w, "none": None, "bytes": rng.integers(1, 256, g.m) * 1.0, "words": rng.integers(1, 1 << 16, g.m) * 1.0,
         "lognormal": rng.lognormal(0.0, 1.0, g.m), "sums": np.full(g.m, 255.0)}[weights]
    src, dst = g.src, g.dst
    if weights == "sums":  # two links of the same nodes: 255 + 258
        src, dst, w = np.append(src, src[0]), np.append(dst, dst[0]), np.append(w, 258.0)
    assert bench.bf16_products(graphs.EdgeList(g.n, src, dst, w)) == products
