"""The wait limit of a batch covers a step of the cases a team waits for, not a whole advance (GPU required)."""
import numpy as np
import pytest

import lapcase
from paper_2507_18268_gb300 import binding as B
from paper_2507_18268_gb300.batch import Batch

pytestmark = pytest.mark.gpu

STEPS = 64


@pytest.mark.parametrize("use_graph", [True, False])
def test_a_team_waits_for_the_steps_of_the_jobs_before_it(use_graph):
    # teams of 432 CTAs each: no launch holds two at once, so the second one is partly staffed while the
    # first runs 64 steps of at least 25 iterations (some 20 ms); one step takes about 0.3 ms
    cases = [lapcase.plain_box(48).with_(DT_uniform=4e-3, dt=0.05, min_iter=25, T0=300.0 + k) for k in range(2)]
    fields = []
    for limit in (10_000_000_000, 3_000_000):
        with Batch() as bt:
            ids = [bt.add_case(c) for c in cases]
            bt.set_launch(256, (1, 1, 1))
            B.lfm_batch_set_barrier_timeout(bt.handle, limit)
            assert bt.advance(STEPS, use_graph=use_graph) == B.LFM_OK
            assert 432 <= B.lfm_batch_get_launch(bt.handle)[0] < 864
            fields.append([bt.field(i).copy() for i in ids])
    for a, b in zip(*fields):
        assert np.array_equal(a, b)
