"""The projection on pairs of SMs at the edges of the rule that selects it (more
tiles than SMs, ten K blocks of 32 dimensions): on both sides of either line the
projected rows, norms, codes and factors are those of the same rows in small
batches, which run on single SMs."""
import numpy as np
import pytest
import torch

import paper_2509_12086_gb300 as P

pytestmark = pytest.mark.gpu


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def _model(d, dk, bits, seed=0, mean=0.1, **kw):
    rng = np.random.default_rng([seed, d])
    W = np.linalg.qr(rng.standard_normal((d, d)))[0][:dk].copy()
    c = (rng.standard_normal(d) * mean).astype(np.float32).astype(np.float64)
    return P.saq_model_create(d, c, W, [(0, dk, bits)] + ([(dk, d - dk, 0)] if dk < d else []), **kw)


@pytest.mark.parametrize("d,dk,bits", [(288, 64, 3), (292, 64, 3), (320, 192, 4), (352, 160, 2)])
@pytest.mark.parametrize("tiles,extra", [(0, 0), (0, 1), (1, 0), (65, -127), (305, 5)])
def test_pairs_equal_single_tiles_at_the_line(d, dk, bits, tiles, extra):
    m = _model(d, dk, bits, rounds=1)
    n = (_sms() + tiles) * 128 + extra  # one column pass: a tile per 128 rows
    g = torch.Generator(device="cuda").manual_seed(d)
    X = torch.randn(n, d, generator=g, device="cuda")
    O, norms = m.project(X)
    codes, factors = m.encode(X)
    m.check_device()
    for a in (0, n // 2 // 128 * 128, (n - 1) // 128 * 128):
        Y = X[a:a + 300].clone()
        b = a + Y.shape[0]
        o, nr = m.project(Y)
        c, f = m.encode(Y)
        assert torch.equal(o, O[a:b]) and torch.equal(nr, norms[a:b]), a
        assert torch.equal(c, codes[a:b]) and torch.equal(f, factors[a:b]), a
    m.check_device()


# ---- failures, as in test_gpu_failure.py, where the pair kernel runs
N_TILES = 40  # beyond the SMs


@pytest.fixture(scope="module")
def batch():
    m = _model(320, 320, 4, mean=0.0, rounds=2)
    n = (_sms() + N_TILES) * 128 - 27
    g = torch.Generator(device="cuda").manual_seed(1)
    X = torch.randn(n, 320, generator=g, device="cuda")
    codes, factors = m.encode(X)
    m.check_device()
    return m, X, codes.clone(), factors.clone()


def _encode_equals(m, X, codes, factors):
    c, f = m.encode(X)
    m.check_device()
    assert torch.equal(c, codes) and torch.equal(f, factors)


def test_wait_timeout_is_reported_and_the_next_encode_is_correct(batch):
    m, X, codes, factors = batch
    P.saq_set_wait_limit(1)
    try:
        for _ in range(3):
            m.encode(X)
            with pytest.raises(P.SaqError, match="timed out"):
                m.check_device()
        with pytest.raises(P.SaqError, match="timed out"):
            m.encode_host(X.cpu().pin_memory())
        m.project(X)
        with pytest.raises(P.SaqError, match="timed out"):
            m.check_device()
    finally:
        P.saq_set_wait_limit(0)
    m.check_device()  # the flag was cleared by the reports
    _encode_equals(m, X, codes, factors)


# a row of the first CTA's half of a tile, of the second's, of the last, ragged tile
@pytest.mark.parametrize("row", [5, 128 + 77, -1])
@pytest.mark.parametrize("bad", ["large", "nan", "inf"])
def test_bad_rows_are_reported(batch, row, bad):
    m, X, codes, factors = batch
    Y = X.clone()
    if bad == "large":
        Y[row] *= 3e4  # beyond the FP16 split's range
    else:
        Y[row, 319] = float(bad)
    m.encode(Y)
    with pytest.raises(P.SaqError, match="out of range"):
        m.check_device()
    m.check_device()
    Y[row] = X[row]
    _encode_equals(m, Y, codes, factors)
