"""Many mixed steps in one launch, each starting from the rows that the verification pass of the step before left
(GPU required): no barrier of the team lies between a step's last decision and the next one's first, so the
threads of a CTA have to agree on both; fields and records equal those of shorter launches bit for bit."""
import numpy as np
import pytest

import lapcase
from paper_2507_18268_gb300 import Solver
from paper_2507_18268_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("on", [True, False])
@pytest.mark.parametrize("dims,launch", [((20, 20, 20), (0, 0)), ((64, 64, 60), (0, 0)), ((31, 30, 29), (60, 512)),
                                         ((24, 23, 22), (12, 1024))])
def test_long_launches_of_seeded_steps(dims, launch, on):
    case = lapcase.random_small_case(sum(dims), *dims, permute=False).with_(tol=1e-7, dt=0.05)
    out = []
    for cuts in ((400,), (150, 250), (100,) * 4):
        with Solver.from_case(case) as s:
            s.set_solver(case.tol, 0.0, 1000, 0, B.LFM_MIXED)
            B.lfm_debug_stage_rows(s.ctx, on)
            if launch[0]:
                s.set_launch(*launch)
            st = []
            for n in cuts:
                st += s.advance(n)
            out.append((s.field().copy(), st))
    for T, st in out[1:]:
        assert np.array_equal(T, out[0][0]) and st == out[0][1]
