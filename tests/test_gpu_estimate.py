"""The estimator's kernels at the sizes where their forms change, against the
FP64 oracle: numbers of queries around a pass's columns, segments that end
inside a word, every bit width and prefix, records that are staged in shared
memory, that are not, and rows too wide for the queries to be."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2509_12086_gb300 as P

pytestmark = pytest.mark.gpu


def _case(d, plan, n, nq, seed=0, eye=False):
    rng = np.random.default_rng(seed)
    dk = sum(l for _, l, b in plan if b > 0)
    if eye:
        W = np.eye(dk, d)
    else:
        W = np.linalg.qr(rng.standard_normal((d, d)))[0][:dk].copy()
    mean = (rng.standard_normal(d) * 0.1).astype(np.float32).astype(np.float64)
    mo = O.Model(d=d, mean=mean, W=W, plan=plan)
    codes = np.concatenate([rng.integers(0, 1 << b, (n, l)) for _, l, b in mo.kept], axis=1).astype(np.uint8)
    nk = len(mo.kept)
    fac = np.empty((n, 1 + 2 * nk), dtype=np.float32)
    fac[:, 1::2] = rng.uniform(0.5, 1.5, (n, nk))
    fac[:, 2::2] = rng.uniform(0.8, 1.0, (n, nk))
    fac[::7, 1] = 0.0  # an all-zero segment
    fac[:, 0] = (fac[:, 1::2] ** 2).sum(1)
    Q = (mean + rng.standard_normal((nq, d)) / np.sqrt(d)).astype(np.float32)
    return mo, codes, fac, Q


def _tolerance(mo, fac, Q):
    """FP32 bound on |error| of a distance: gamma = (d / 32 + 8) 2^-24 bounds the
    relative error of a lane-split sum of d products, so each rotated query
    coordinate is within gamma |q - c|, the inner products within
    gamma (sqrt(dk) + 2) |o| |q - c| / 0.8, and |o| |q - c| is at most half the
    sum of squares; twice that for the final sums."""
    gamma = (mo.d / 32 + 8) * 2.0 ** -24
    dk = sum(l for _, l, b in mo.plan if b > 0)
    q2 = ((Q.astype(np.float64) - mo.mean) ** 2).sum(1)
    nk = len(mo.kept)
    return 2 * gamma * (np.sqrt(dk * nk) + 2) * (fac[:, 0].astype(np.float64)[None] + q2[:, None])


ODD = [(0, 64, 8), (64, 72, 3), (136, 32, 1), (168, 130, 5), (298, 257, 2), (555, 9, 0), (564, 36, 4)]


@pytest.mark.parametrize("n,nq", [(1, 1), (15, 4), (16, 5), (17, 16), (1000, 17), (333, 32), (100, 33), (5000, 3), (40, 140)])
def test_odd_segments_and_query_counts(n, nq):
    mo, codes, fac, Q = _case(600, ODD, n, nq, seed=n + nq)
    m = P.saq_model_create(mo.d, mo.mean, mo.W, mo.plan, precision="fp32_simt")
    cd, fd = torch.from_numpy(O.pack(codes, mo)).cuda(), torch.from_numpy(fac).cuda()
    Qd = torch.from_numpy(Q).cuda()
    tol = _tolerance(mo, fac, Q)
    for b in (0, 1, 3, 5):
        got = m.estimate_dist(cd, fd, Qd, prefix_bits=b).cpu().numpy().astype(np.float64)
        ref = O.estimate(mo, codes, fac.astype(np.float64), Q, prefix_bits=b)
        assert np.all(np.abs(got - ref) <= tol), b


@pytest.mark.parametrize("bits", [1, 2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("d", [67, 192, 448, 1000])
def test_every_width(bits, d):
    mo, codes, fac, Q = _case(d, [(0, d, bits)], 50, 6, seed=bits)
    m = P.saq_model_create(mo.d, mo.mean, mo.W, mo.plan, precision="fp32_simt")
    got = m.estimate_dist(torch.from_numpy(O.pack(codes, mo)).cuda(), torch.from_numpy(fac).cuda(),
                          torch.from_numpy(Q).cuda()).cpu().numpy().astype(np.float64)
    ref = O.estimate(mo, codes, fac.astype(np.float64), Q)
    assert np.all(np.abs(got - ref) <= _tolerance(mo, fac, Q))


@pytest.mark.parametrize("nq", [2, 9, 31])
@pytest.mark.parametrize("d", [2100, 2500])
def test_records_too_wide_to_stage(d, nq):
    mo, codes, fac, Q = _case(d, [(0, 1024, 8), (1024, d - 1024, 7)], 37, nq, seed=nq)
    m = P.saq_model_create(mo.d, mo.mean, mo.W, mo.plan, precision="fp32_simt")
    got = m.estimate_dist(torch.from_numpy(O.pack(codes, mo)).cuda(), torch.from_numpy(fac).cuda(),
                          torch.from_numpy(Q).cuda()).cpu().numpy().astype(np.float64)
    ref = O.estimate(mo, codes, fac.astype(np.float64), Q)
    assert np.all(np.abs(got - ref) <= _tolerance(mo, fac, Q))


def test_queries_too_wide_for_shared_memory():
    d = 14_400
    mo, codes, fac, Q = _case(d, [(0, 14_000, 1), (14_000, 400, 2)], 20, 5, eye=True)
    m = P.saq_model_create(mo.d, mo.mean, mo.W, mo.plan, precision="fp32_simt")
    got = m.estimate_dist(torch.from_numpy(O.pack(codes, mo)).cuda(), torch.from_numpy(fac).cuda(),
                          torch.from_numpy(Q).cuda()).cpu().numpy().astype(np.float64)
    ref = O.estimate(mo, codes, fac.astype(np.float64), Q)
    assert np.all(np.abs(got - ref) <= _tolerance(mo, fac, Q))


def test_extreme_queries():
    """Scales far from one, a zero query, and a query that is not finite."""
    mo, codes, fac, Q = _case(600, ODD, 64, 6)
    m = P.saq_model_create(mo.d, mo.mean * 0, mo.W, mo.plan, precision="fp32_simt")
    mo.mean = mo.mean * 0
    Q[0] *= 1e15
    Q[1] *= 1e-18
    Q[2] = 0
    Q[3, 5] = np.inf
    Q[4, 7] = np.nan
    got = m.estimate_dist(torch.from_numpy(O.pack(codes, mo)).cuda(), torch.from_numpy(fac).cuda(),
                          torch.from_numpy(Q).cuda()).cpu().numpy().astype(np.float64)
    ref = O.estimate(mo, codes, fac.astype(np.float64), Q)
    ok = [0, 1, 2, 5]
    assert np.all(np.abs(got - ref)[ok] <= _tolerance(mo, fac, Q)[ok])
    assert not np.isfinite(got[3]).any() and not np.isfinite(got[4]).any()
