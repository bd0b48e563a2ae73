"""The rms that scales the learned warm start's features and targets (one
cluster of eight CTAs), at sizes about its CTAs' first rows (1024 each) and
its first full pass (8192): a recorded target is the solved update with each
component over its rms, so its mean square is 1 per component and the loss of
a network that predicts zero (a fresh one) is 0.5 (1 + 1).  A partial sum
that was lost makes it larger.  Bar 1e-5: the targets are FP32 (2^-24 each),
their squares are added in FP32 in blocks of 256.
"""
import pytest

import paper_1701_06254_gb300 as R
from paper_1701_06254_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1, 1), (3, 1, 1), (33, 31, 1), (32, 32, 1), (41, 25, 1), (64, 32, 4), (2731, 3, 1),
                                   (37, 29, 11)],
                         ids=["1", "3", "1023", "1024", "1025", "8192", "8193", "11803"])
def test_recorded_targets_have_unit_rms(shape):
    c = I.small_case(*shape, seed=31)
    p0, s0, pb0 = I.random_state(c, 500)
    p1, s1, pb1 = I.random_state(c, 501)
    ws = R.WarmStart(seed=1)
    g = R.Sim(c)
    g.record_to(ws)
    g.set_state(p0, s0, pb0)
    g.begin_step(1.0)
    g.set_state(p1, s1, pb1)
    for k in range(4):
        g.assemble()
        g.linear_solve(1e-6)
        assert ws.dataset_size() == k + 1
    assert ws.eval() == pytest.approx(1.0, rel=1e-5)
