"""Packed slot words that the device box builder writes (GPU required): seven distances wherever a box has
six slots, and runs on the words equal runs on the slot rows and on the uploaded mesh's own words bit for bit."""
import numpy as np
import pytest

import lapcase
from paper_2507_18268_gb300 import Solver
from paper_2507_18268_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [B.LFM_FP64, B.LFM_MIXED, B.LFM_DF64])
@pytest.mark.parametrize("dims", [(3, 3, 3), (3, 5, 4), (9, 3, 7), (16, 9, 5), (33, 31, 29), (2, 5, 4), (12, 9, 1)])
def test_box_words_equal_slot_rows_and_uploaded_words(dims, prec):
    case = lapcase.random_small_case(sum(dims), *dims, permute=False, face_dt=False).with_(tol=1e-10, dt=0.2)
    packs = min(dims) >= 3
    out = []
    for make, on in ((Solver.from_box_case, True), (Solver.from_box_case, False), (Solver.from_case, True)):
        with make(case) as s:
            n = B.lfm_debug_pack_slots(s.ctx, on)
            assert n == (7 if packs else 0)
            s.set_solver(case.tol, 0.0, 1000, 0, prec)
            out.append((s.advance(2) + s.advance(1), s.field().copy()))
    for st, T in out[1:]:
        assert st == out[0][0] and np.array_equal(T, out[0][1])


@pytest.mark.parametrize("on", [True, False])
def test_switch_before_a_second_upload(on):
    # the switch of a context holds for a box uploaded after it
    case = lapcase.random_small_case(5, 6, 5, 4, permute=False, face_dt=False).with_(tol=1e-10, dt=0.2)
    with Solver.from_box_case(case) as s, Solver.from_box_case(case) as t:
        assert B.lfm_debug_pack_slots(s.ctx, on) == 7
        share = Solver.sharing(s, case)
        assert B.lfm_debug_pack_slots(share.ctx, on) == 7
        want = t.advance(2)
        assert share.advance(2) == want and s.advance(2) == want
        assert np.array_equal(share.field(), t.field()) and np.array_equal(s.field(), t.field())
        share.close()
