"""The estimator's inner products against 64 bits for rotated queries whose
coordinates share a sign, lie along the codes, hold one large value or decay,
at every bit width and in every form of the kernel.  W is the identity, so that
the rotated query is the query, and |o| is 2^20, so that the rounding of the
squared norms does not hide an error.

The tolerance is an FP32 sum's: half a unit in the last place of |o| |q| for the
query's own representation (its 24 bits), and twelve of the estimate for the
additions of the windows, the scale's square root, product and quotient and the
final sums.  It fails for queries held in 12 bits, for coordinates held to 23
bits below the largest one of the query, and for sums truncated at 24 bits.
"""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2509_12086_gb300 as P

pytestmark = pytest.mark.gpu

NORM = 2.0 ** 20
MIXED = [(0, 64, 8), (64, 200, 6), (264, 129, 5), (393, 448, 4), (841, 31, 7), (872, 128, 1)]


def _queries(kind, rng, nq, d, U):
    z = rng.standard_normal((nq, d))
    if kind == "one sign":
        return rng.uniform(0.5, 1, (nq, d)) * rng.choice([-1.0, 1.0], (nq, 1))
    if kind == "along":
        return U[rng.integers(0, len(U), nq)]
    if kind == "spike":
        z[np.arange(nq), rng.integers(0, d, nq)] = 1000
    if kind == "decay":
        z *= np.exp(-np.arange(d) / (d / 16))
    return z


def _check(plan, d, n, nq, kind, prefix, seed):
    rng = np.random.default_rng([seed, d, nq])
    mo = O.Model(d=d, mean=np.zeros(d), W=np.eye(d), plan=plan)
    codes = np.concatenate([rng.integers(0, 1 << b, (n, l)) for _, l, b in plan], axis=1).astype(np.uint8)
    used = [min(b, prefix) if prefix else b for _, _, b in plan]
    U = np.concatenate([2.0 * (codes[:, s:s + l] >> (b - k)) - ((1 << k) - 1)
                        for (s, l, b), k in zip(plan, used)], axis=1)
    Q = _queries(kind, rng, nq, d, U)
    Q = (Q / np.linalg.norm(Q, axis=1, keepdims=True)).astype(np.float32)
    fac = np.zeros((n, 1 + 2 * len(plan)), np.float32)
    fac[:, 1::2], fac[:, 2::2] = NORM, 1
    m = P.saq_model_create(d, mo.mean, mo.W, plan, precision="fp32_simt")
    got = m.estimate_dist(torch.from_numpy(O.pack(codes, mo)).cuda(), torch.from_numpy(fac).cuda(),
                          torch.from_numpy(Q).cuda(), prefix_bits=prefix).cpu().numpy()
    ref = O.estimate(mo, codes, fac.astype(np.float64), Q, prefix_bits=prefix)
    tol = np.zeros((nq, n))
    for s, l, _ in plan:
        u, q = U[:, s:s + l], Q[:, s:s + l].astype(np.float64)
        est = np.abs(q @ u.T) / np.linalg.norm(u, axis=1)
        tol += 2.0 ** -24 * (np.linalg.norm(q, axis=1)[:, None] + 12 * est)
    err = np.abs(got.astype(np.float64) - ref) / (2 * NORM)
    assert np.all(err <= tol), (kind, prefix, float((err / tol).max()))


KINDS = ["random", "one sign", "along", "spike", "decay"]


# one, four and eight queries to a B tile; records staged and, at the last
# width, too wide to be
@pytest.mark.parametrize("nq", [2, 13, 40])
@pytest.mark.parametrize("bits,d", [(8, 128), (8, 129), (8, 448), (8, 960), (7, 300), (7, 1000), (6, 640),
                                    (5, 1090), (4, 448), (4, 1536), (3, 960), (1, 1024), (8, 3072)])
def test_one_segment(bits, d, nq):
    for kind in KINDS:
        _check([(0, d, bits)], d, 70, nq, kind, 0, bits)


@pytest.mark.parametrize("prefix", [0, 1, 3, 5, 7])
def test_segments_and_prefixes(prefix):
    for nq in (1, 18):
        for kind in KINDS:
            _check(MIXED, 1000, 50, nq, kind, prefix, prefix)


def test_queries_too_wide_for_shared_memory():
    for kind in KINDS:
        _check([(0, 12_000, 1), (12_000, 2400, 8)], 14_400, 20, 5, kind, 0, 5)
