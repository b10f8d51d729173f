"""Jobs that one CTA runs in turn on meshes of equal slot words and different neighbour distances (GPU
required): every job has to look its distances up in its own case's table."""
import numpy as np
import pytest

import lapcase
from paper_2507_18268_gb300 import Solver
from paper_2507_18268_gb300 import binding as B
from paper_2507_18268_gb300.batch import Batch

pytestmark = pytest.mark.gpu


def cases(prec, n):
    # boxes of (a, b, 4): every one has the distances -ab, -a, -1, 0, 1, a, ab, in this order
    return [lapcase.random_small_case(k, 3 + k % 9, 5 + k % 4, 4, permute=False, face_dt=False).with_(
        tol=1e-10, dt=0.2, precision=prec)
            for k in range(n)]


@pytest.mark.parametrize("prec", [B.LFM_FP64, B.LFM_DF64, B.LFM_MIXED])
def test_each_job_uses_its_own_distances(prec):
    members = cases(prec, 700)  # teams of one CTA, more of them than a launch has CTAs
    fields = []
    for on in (True, False):
        with Batch() as bt:
            ids = []
            for c in members:
                s = Solver.from_box_case(c, layout=prec)
                assert B.lfm_debug_pack_slots(s.ctx, on) == 7
                ids.append(bt.add(s))
            bt.set_launch(256, (4, 4, 4))
            assert bt.advance(2) == B.LFM_OK
            assert B.lfm_batch_get_launch(bt.handle)[0] < len(members)
            fields.append([bt.field(i).copy() for i in ids])
    for a, b in zip(*fields):
        assert np.array_equal(a, b)
