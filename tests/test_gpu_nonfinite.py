"""Queries with a NaN or an infinity: their rows' outputs and lse are NaN, whether
the pair lies within one CTA's range or is split over many (there the merge combines
partials whose lse is NaN); the other rows are those of the finite call."""
import math

import pytest
import torch

from tests.device_util import Call, assert_rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kf8,vf8", [(False, False), (True, False), (True, True), (False, True)])
@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("G,T", [(1, 8), (4, 6), (4, 15)])
@pytest.mark.parametrize("P", [[300, 70, 0, 129], [45000, 70, 0, 129]], ids=["short", "long"])
def test_rows_with_nan_and_infinite_queries(kf8, vf8, D, G, T, P):
    c = Call(P, [T] * 4, G, 2, D, kf8, vf8, 70000 if P[0] > 300 else None, seed=3)
    c.kb[:, 0, :, D - 1] = 1.0  # so that an infinite query has a score of +infinity
    ref = c.reference()
    bad = torch.zeros(c.q.shape[:3], dtype=torch.bool, device="cuda")
    for b in range(4):
        c.q[b, 1, 0, 5], c.q[b, 3, -1, D - 1] = math.nan, math.inf
        bad[b, 1, 0], bad[b, 3, -1] = True, True
    out, lse = c.run()
    torch.cuda.synchronize()
    assert c.status() == 0
    assert bool(out[bad].isnan().all()), "a bad row's output is not NaN"
    assert bool(lse.permute(0, 2, 1)[bad].isnan().all()), "a bad row's lse is not NaN"
    assert_rows(out, lse, ref, keep=~bad)
