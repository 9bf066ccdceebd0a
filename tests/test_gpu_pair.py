"""The projection on pairs of SMs (large FP32 batches) against the single-SM
kernels of small ones: the same rows give the same projected values, norms,
bytes and factors, as every kernel adds the same products in the same order."""
import numpy as np
import pytest
import torch

import paper_2509_12086_gb300 as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,plan,n", [
    (64, [(0, 64, 4)], 153 * 128),                        # two K blocks, an odd number of row tiles
    (100, [(0, 96, 3), (96, 4, 0)], 20_001),              # a ragged K block and last row
    (20, [(0, 10, 6), (10, 10, 2)], 152 * 128 + 1),       # one K block; a tile of one row
    (328, [(0, 200, 2), (200, 120, 5), (320, 8, 0)], 30_007),  # column passes, the last one ragged
    (776, [(0, 384, 8), (384, 384, 1), (768, 8, 0)], 10_113)])
def test_pairs_equal_single_tiles(d, plan, n):
    rng = np.random.default_rng(d)
    dk = sum(l for _, l, b in plan if b > 0)
    W = np.linalg.qr(rng.standard_normal((d, d)))[0][:dk].copy()
    mean = (rng.standard_normal(d) * 0.1).astype(np.float32).astype(np.float64)
    m = P.saq_model_create(d, mean, W, plan, rounds=2)
    g = torch.Generator(device="cuda").manual_seed(d)
    X = torch.randn(n, d, generator=g, device="cuda") * torch.linspace(1, 0.1, d, device="cuda")
    O, norms = m.project(X)
    codes, factors = m.encode(X)
    m.check_device()
    for a in (0, 128, n // 2 // 128 * 128, (n - 1) // 128 * 128):
        b = min(n, a + 300)
        Y = X[a:b].clone()
        o, nr = m.project(Y)
        c, f = m.encode(Y)
        assert torch.equal(o, O[a:b]) and torch.equal(nr, norms[a:b]), (a, b)
        assert torch.equal(c, codes[a:b]) and torch.equal(f, factors[a:b]), (a, b)
    m.check_device()
