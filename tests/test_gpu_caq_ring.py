"""The lane-per-vector quantizer's batches, slots and code stores at their
edges: segments shorter than, as long as and longer than a batch (8), a slot
(16) and the ring, with codes in shared memory and in the global scratch.  The
warp-per-vector scan of the same rows in small pieces gives the same bytes."""
import numpy as np
import pytest
import torch

import paper_2509_12086_gb300 as P

pytestmark = pytest.mark.gpu

# (length, bits); the 1,160-long segment's codes do not fit in shared memory
SHORT = [(1, 1), (7, 2), (8, 3), (9, 4), (15, 5), (16, 6), (17, 7), (31, 8), (32, 1), (33, 2),
         (40, 3), (47, 5), (48, 8), (63, 4), (65, 6), (68, 1)]


@pytest.mark.parametrize("rounds", [0, 1, 2, 7])
@pytest.mark.parametrize("segments,n", [(SHORT, 40_007), (SHORT + [(1160, 8)], 20_003)])
def test_lane_kernel_equals_scan_at_the_edges(segments, n, rounds):
    plan, at = [], 0
    for length, bits in segments:
        plan.append((at, length, bits))
        at += length
    d = at + (-at % 4)
    if d > at:
        plan.append((at, d - at, 0))
    rng = np.random.default_rng(len(segments))
    W = np.linalg.qr(rng.standard_normal((d, d)))[0][:at].copy()
    mean = (rng.standard_normal(d) * 0.1).astype(np.float32).astype(np.float64)
    m = P.saq_model_create(d, mean, W, plan, rounds=rounds)
    g = torch.Generator(device="cuda").manual_seed(d)
    X = torch.randn(n, d, generator=g, device="cuda") * torch.linspace(1, 0.1, d, device="cuda")
    X[::13] = torch.from_numpy(mean.astype(np.float32)).cuda()  # all-zero segments
    codes, factors = m.encode(X)
    for a, b in ((0, 97), (n - 100, n)):
        c, f = m.encode(X[a:b].clone())
        assert torch.equal(c, codes[a:b]) and torch.equal(f, factors[a:b]), (a, b)
    m.check_device()
