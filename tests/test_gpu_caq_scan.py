"""The warp-per-vector scan of small batches against the lane-per-vector
kernel of large ones: the same rows give the same bytes and factors."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2509_12086_gb300 as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rounds", [0, 1, 6])
@pytest.mark.parametrize("d,plan,n", [
    (200, [(0, 64, 8), (64, 72, 3), (136, 32, 1), (168, 32, 0)], 20_000),
    (132, [(0, 31, 2), (31, 33, 6), (64, 64, 4), (128, 4, 5)], 30_000),
    (700, [(0, 700, 8)], 40_000),       # |u|^2 beyond 2^24: its rounding order counts
    (1000, [(0, 900, 7), (900, 100, 1)], 33_000)])
def test_small_batches_equal_large_ones(d, plan, n, rounds):
    rng = np.random.default_rng(d)
    dk = sum(l for _, l, b in plan if b > 0)
    W = np.linalg.qr(rng.standard_normal((d, d)))[0][:dk].copy()
    mean = (rng.standard_normal(d) * 0.1).astype(np.float32).astype(np.float64)
    m = P.saq_model_create(d, mean, W, plan, rounds=rounds)
    g = torch.Generator(device="cuda").manual_seed(d)
    X = torch.randn(n, d, generator=g, device="cuda") * torch.linspace(1, 0.1, d, device="cuda")
    X[::11] = torch.from_numpy(mean.astype(np.float32)).cuda()  # all-zero segments
    codes, factors = m.encode(X)
    for a, b in ((0, 1), (1, 32), (32, 65), (100, 1100)):
        # rows start at a 16-byte boundary: d % 4 == 0
        c, f = m.encode(X[a:b].clone())
        assert torch.equal(c, codes[a:b]) and torch.equal(f, factors[a:b]), (a, b)
    m.check_device()
