"""The query rotation at the edges of what it stages (1,024 coordinates at a
time, eight queries to a block), through the estimator, against the oracle."""
import pytest
import torch

import oracle as O
import paper_2509_12086_gb300 as P
from tests.test_gpu_estimate import _case, _tolerance

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nq", [1, 2, 3, 8, 9, 23])
@pytest.mark.parametrize("d", [1, 4, 31, 36, 64, 257, 1020, 1023, 1024, 1025, 1028, 2049, 2052])
def test_rotation_at_the_edges_of_a_stage(d, nq):
    mo, codes, fac, Q = _case(d, [(0, d, 2)], 5, nq, seed=d + nq)
    m = P.saq_model_create(mo.d, mo.mean, mo.W, mo.plan, precision="fp32_simt")
    got = m.estimate_dist(torch.from_numpy(O.pack(codes, mo)).cuda(), torch.from_numpy(fac).cuda(),
                          torch.from_numpy(Q).cuda()).cpu().numpy()
    ref = O.estimate(mo, codes, fac.astype("f8"), Q)
    assert (abs(got - ref) <= _tolerance(mo, fac, Q)).all()
