"""Advances on a stream that is being captured (GPU required): set-up that is due is never only recorded,
and a recorded advance reads the patches as they are when it is replayed."""
import numpy as np
import pytest
import torch

import lapcase
from paper_2507_18268_gb300 import Solver
from paper_2507_18268_gb300 import binding as B

pytestmark = pytest.mark.gpu

PRECS = [B.LFM_FP64, B.LFM_DF64, B.LFM_MIXED]


def base():
    return lapcase.random_small_case(4, 7, 6, 5, patch_types=[lapcase.FIXED_VALUE] * 6).with_(tol=1e-10, dt=0.2)


def general():
    return lapcase.perturbed_box(lapcase.random_small_case(4, 7, 6, 5, permute=False), amp=0.2).with_(tol=1e-10, dt=0.2)


def solver(case, prec, **kw):
    s = Solver.from_case(case, **kw)
    s.set_solver(case.tol, 0.0, 1000, 0, prec)
    return s


def capture(stream, call):
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    x = torch.zeros(8, device="cuda")
    with torch.cuda.stream(stream):
        graph.capture_begin(capture_error_mode="thread_local")
        try:
            x += 1  # the capture holds work whether or not the call adds any
            call()
        finally:
            graph.capture_end()
    return graph, x


def DT_change(s):
    B.lfm_set_diffusivity(s.ctx, 0.0, 1.7 * s.mesh.DT_faces, 0.4 * s.mesh.DT_bfaces)


def dt_change(s):
    B.lfm_set_time_step(s.ctx, 0.05)


def value_change(s):
    B.lfm_set_patch(s.ctx, 0, lapcase.FIXED_VALUE, None, 411.0)


# what is due when the capture begins: (case, warm-up outside the capture, change before it, precisions)
DUE = {
    "fresh": (base, False, None, PRECS),
    "fresh_general": (general, False, None, PRECS),
    "diffusivity": (base, True, DT_change, PRECS),
    "time_step": (base, True, dt_change, [B.LFM_DF64, B.LFM_MIXED]),
    "patch_general": (general, True, value_change, PRECS),
}


@pytest.mark.parametrize("name,prec", [(n, p) for n, d in DUE.items() for p in d[3]])
def test_due_set_up_is_refused_under_capture_and_runs_later(name, prec):
    make, warm, change, _ = DUE[name]
    case = make()
    out = []
    for captured in (False, True):
        side = torch.cuda.Stream()
        with solver(case, prec, stream=side) as s:
            T0 = s.field().copy()
            if warm:
                s.advance(1)
            if change:
                change(s)
            if captured:
                rc = []
                graph, x = capture(side, lambda: rc.append(B.load().lfm_advance_async(s.ctx, 2)))
                assert rc == [B.LFM_ESTATE]
                with torch.cuda.stream(side):
                    graph.replay()  # the capture stays usable
                torch.cuda.synchronize()
                assert float(x[0]) == 1.0
            s.set_field(T0)
            st = s.advance(2)
            out.append((s.field().copy(), st))
    assert np.array_equal(out[0][0], out[1][0]) and out[0][1] == out[1][1]


@pytest.mark.parametrize("prec", PRECS)
def test_patch_changes_around_a_recorded_advance(prec):
    case = base()

    def fresh(value):
        with solver(case, prec) as s:
            B.lfm_set_patch(s.ctx, 0, lapcase.FIXED_VALUE, None, value)
            s.advance(2)
            return s.field().copy()

    want = {v: fresh(v) for v in (300.0, 350.0, 400.0)}
    side = torch.cuda.Stream()
    with solver(case, prec, stream=side) as s:
        T0 = s.field().copy()
        s.advance(1)
        B.lfm_set_patch(s.ctx, 0, lapcase.FIXED_VALUE, None, 300.0)
        graph, _ = capture(side, lambda: B.lfm_advance_async(s.ctx, 2))
        B.lfm_finish_status(s.ctx, 0)  # nothing of the recorded advance is pending on the stream

        def replayed():
            s.set_field(T0)
            with torch.cuda.stream(side):
                graph.replay()
            torch.cuda.synchronize()
            return s.field().copy()

        def advanced():
            s.set_field(T0)
            s.advance(2)
            return s.field().copy()

        assert np.array_equal(advanced(), want[300.0])  # before any replay
        assert np.array_equal(replayed(), want[300.0])
        for v in (350.0, 400.0):
            B.lfm_set_patch(s.ctx, 0, lapcase.FIXED_VALUE, None, v)
            assert np.array_equal(replayed(), want[v])
            assert np.array_equal(advanced(), want[v])
        del graph
