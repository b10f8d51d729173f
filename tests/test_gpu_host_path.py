"""Host path of a launch (GPU required): the flag writes that a field upload may skip, uploads recorded
into a graph, and pinned buffers that pass between contexts and threads."""
import threading

import numpy as np
import pytest

import lapcase
from paper_2507_18268_gb300 import Solver
from paper_2507_18268_gb300 import binding as B

pytestmark = pytest.mark.gpu

PRECS = [B.LFM_FP64, B.LFM_DF64, B.LFM_MIXED]


def case_of(seed=4):
    return lapcase.random_small_case(seed, 7, 6, 5).with_(tol=1e-10, dt=0.2)


def solver(case, prec, **kw):
    s = Solver.from_case(case, **kw)
    s.set_solver(case.tol, 0.0, 1000, 0, prec)
    return s


@pytest.mark.parametrize("prec", PRECS)
def test_field_uploads_before_and_after_launches_and_a_recorded_upload(prec):
    import torch
    case = case_of()
    side = torch.cuda.Stream()
    with solver(case, prec) as s:
        T0 = s.field().copy()
        s.advance(2)
        want = s.field().copy()
    with solver(case, prec, stream=side) as s:
        T = torch.as_tensor(T0, device="cuda")
        torch.cuda.synchronize()
        for _ in range(2):
            for _ in range(2):  # the second finds the flags clear
                B.lfm_set_field_device(s.ctx, T.data_ptr())
            s.advance(2)
            assert np.array_equal(s.field(), want)
        B.lfm_set_field_device(s.ctx, T.data_ptr())
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            graph.capture_begin(capture_error_mode="thread_local")
            B.lfm_set_field_device(s.ctx, T.data_ptr())
            graph.capture_end()
        for _ in range(3):
            with torch.cuda.stream(side):
                graph.replay()
            s.advance(2)
            assert np.array_equal(s.field(), want)
        del graph


def test_contexts_come_and_go_on_several_threads():
    case = case_of(9)
    with solver(case, B.LFM_MIXED) as s:
        want_st = s.advance(2)
        want = s.field().copy()
    bad = []

    def work():
        for i in range(12):
            with solver(case, B.LFM_MIXED) as a, solver(case, B.LFM_MIXED) as b:
                for s in (a, b):
                    if s.advance(2) != want_st or not np.array_equal(s.field(), want):
                        bad.append(i)

    threads = [threading.Thread(target=work) for _ in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
