"""Streamed mixed and df64 solves that update the solution in the direction pass (by default from 5 M and
2.5 M cells on) against the update in the residual's pass (GPU required): the same operations on every value in the same
order, so fields and records agree bit for bit."""
import numpy as np
import pytest

import lapcase
from paper_2507_18268_gb300 import Solver
from paper_2507_18268_gb300 import binding as B
from paper_2507_18268_gb300.batch import Batch

pytestmark = pytest.mark.gpu

PRECS = [B.LFM_MIXED, B.LFM_DF64]
NEVER = 2 ** 31 - 1


def box(dims, permute=False, **kw):
    return lapcase.random_small_case(sum(dims), *dims, permute=permute).with_(tol=1e-8, dt=0.2, **kw)


def general(dims):
    return lapcase.perturbed_box(box(dims), amp=0.2, seed=3)


def run(case, prec, cells, stage, launch, cuts):
    with Solver.from_case(case) as s:
        s.set_solver(case.tol, case.rel_tol, case.max_iter, case.min_iter, prec)
        B.lfm_debug_stage_rows(s.ctx, stage)
        B.lfm_debug_late_cells(s.ctx, cells)
        s.set_launch(*launch)
        st, late, code = [], 0, B.LFM_OK
        for n in cuts:
            B.lfm_advance_async(s.ctx, n)
            code, part = B.lfm_finish_status(s.ctx, n)
            st += [x.as_dict() for x in part]
            late += B.lfm_debug_late_solves(s.ctx)
            if code != B.LFM_OK:
                break
        assert B.lfm_debug_solve_form(s.ctx) == 0
        return s.field().copy(), st, late, code


def check(case, prec, launch, stage, cuts=(2, 1)):
    T, st, late, code = run(case, prec, 1, stage, launch, cuts)
    T0, st0, none, code0 = run(case, prec, NEVER, stage, launch, cuts)
    assert late > 0 and none == 0 and code == code0
    assert np.array_equal(T, T0) and st == st0
    return st, code


# (cells, launch, rows streamed through shared memory): ranges that end inside a tile or a warp, odd numbers of
# rows per thread, one row and less, more CTAs than ranges, N not a multiple of 4, five slots, 1024 threads
SHAPES = [((8, 8, 4), (1, 256), False), ((9, 8, 8), (1, 256), True), ((11, 10, 10), (2, 256), True),
          ((7, 9, 5), (1, 256), False), ((15, 13, 11), (1, 256), True), ((16, 16, 9), (1, 256), True),
          ((11, 10, 10), (40, 256), False), ((20, 20, 13), (1, 512), True), ((23, 17, 13), (3, 512), False),
          ((16, 16, 2), (1, 512), True), ((13, 12, 11), (1, 1024), True), ((3, 3, 3), (7, 512), False)]


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("permute", [False, True])
@pytest.mark.parametrize("dims,launch,stage", SHAPES)
def test_late_equals_early(dims, launch, stage, permute, prec):
    st, _ = check(box(dims, permute), prec, launch, stage)
    assert max(x["iters"] for x in st) >= 3


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("kw", [dict(max_iter=1), dict(max_iter=2), dict(max_iter=3), dict(tol=1e-3, min_iter=5),
                                dict(tol=1e-13), dict(tol=0.0, rel_tol=1e-4), dict(Su=9.0, Sp=-0.3),
                                dict(n_nonorth_corr=2)],
                         ids=["one", "two", "three", "min_iter", "sweeps", "rel_tol", "sources", "passes"])
def test_options(kw, prec):
    case = box((10, 9, 8)).with_(**kw)
    for cuts in ((3,), (1, 1, 1)):
        check(case, prec, (2, 256), False, cuts)


@pytest.mark.parametrize("n_corr", [0, 2])
def test_mixed_on_a_general_mesh(n_corr):
    # the mixed form with FP64 outer passes (df64 general meshes never update late)
    for dims, launch in (((9, 8, 8), (1, 256)), ((11, 10, 9), (4, 256)), ((20, 16, 11), (2, 512))):
        check(general(dims).with_(n_nonorth_corr=n_corr), B.LFM_MIXED, launch, True, (2, 1))


@pytest.mark.parametrize("prec", PRECS)
def test_singular_direction_after_a_late_update(prec):
    # eight equal cells with a uniform field and source: one iteration leaves a residual of exactly zero, the
    # second direction is zero and its product singular
    case = lapcase.RawCase(xs=np.arange(3.0), ys=np.arange(3.0), zs=np.arange(3.0), DT_uniform=1.0, dt=1.0, T0=256.0,
                           patches=((lapcase.ZERO_GRADIENT, 0.0),) * 6, Su=64.0, tol=1e-12, min_iter=3, n_steps=1)
    st, code = check(case, prec, (1, 256), False, (1,))
    assert code == B.LFM_ESINGULAR and st[0]["iters"] == 1


def test_late_in_a_batch():
    fields = []
    for cells in (1, NEVER):
        with Batch() as bt:
            ids = [bt.add_case(box(d).with_(precision=B.LFM_MIXED)) for d in ((9, 8, 8), (15, 13, 11), (20, 20, 13))]
            for i in ids:
                B.lfm_debug_late_cells(bt.cases[i].ctx, cells)
            assert bt.advance(2) == B.LFM_OK
            fields.append([(bt.field(i).copy(), bt.stats(i, 2)) for i in ids])
    for (a, sa), (b, sb) in zip(*fields):
        assert np.array_equal(a, b) and sa == sb


@pytest.mark.parametrize("prec,dims,late", [(B.LFM_MIXED, (169, 171, 172), 0), (B.LFM_MIXED, (170, 171, 172), 1),
                                            (B.LFM_DF64, (135, 136, 136), 0), (B.LFM_DF64, (136, 136, 136), 1)])
def test_default_line(prec, dims, late):
    case = lapcase.RawCase(*(lapcase.uniform_axis(n) for n in dims), DT_uniform=4e-5, dt=0.005, n_steps=1,
                           precision=prec)
    with Solver.from_box_case(case, layout=prec) as s:
        assert s.advance(1)[0]["iters"] > 0
        assert (B.lfm_debug_late_solves(s.ctx) > 0) == bool(late)
