"""The mixed form's inner solve kept on chip (matrix rows in shared memory, vectors in registers, the
direction formed inside the product) against the streamed solve (GPU required).

Every value is formed by the same operations and every sum in the same order, so field and
statistics agree bit for bit: at the rows per thread where a kernel for more rows, or the streamed
form, takes over, on ragged meshes (rows loaded without bulk copies), packed and not, with further
sweeps, iteration limits, sources and several launches.
"""
import numpy as np
import pytest

import lapcase
import oracle
from paper_2507_18268_gb300 import Solver
from paper_2507_18268_gb300 import binding as B

pytestmark = pytest.mark.gpu


def case_of(dims, permute=False, **kw):
    c = lapcase.random_small_case(sum(dims), *dims, permute=permute)
    return c.with_(tol=1e-8, dt=0.2, **kw)


def run(case, on, ctas, threads, cuts=(2, 1)):
    with Solver.from_case(case) as s:
        s.set_solver(case.tol, case.rel_tol, case.max_iter, case.min_iter, B.LFM_MIXED)
        B.lfm_debug_stage_rows(s.ctx, on)
        s.set_launch(ctas, threads)
        st = []
        for n in cuts:
            st += s.advance(n)
        return s.field().copy(), st, B.lfm_debug_staged_passes(s.ctx)


# cells, launch: rows per thread 1, 2, 3 (256 threads); 1, 4, 5, 6, 7 (512); ranges that end inside a
# warp; more CTAs than ranges; N not a multiple of 4
SHAPES = [((8, 8, 4), 1, 256), ((8, 8, 8), 1, 256), ((9, 8, 8), 1, 256), ((8, 8, 8), 2, 256),
          ((16, 16, 2), 1, 512), ((16, 16, 8), 1, 512), ((17, 16, 8), 1, 512), ((16, 16, 12), 1, 512),
          ((20, 16, 10), 1, 512), ((20, 16, 10), 3, 512), ((11, 10, 10), 40, 256), ((7, 9, 5), 1, 256),
          ((7, 9, 5), 3, 256), ((3, 3, 3), 1, 512)]


@pytest.mark.parametrize("permute", [False, True])
@pytest.mark.parametrize("dims,ctas,threads", SHAPES)
def test_resident_bitwise_equal_to_streamed(dims, ctas, threads, permute):
    case = case_of(dims, permute)
    T, st, _ = run(case, True, ctas, threads)
    T0, st0, _ = run(case, False, ctas, threads)
    assert np.array_equal(T, T0) and st == st0
    assert max(x["iters"] for x in st) >= 3


@pytest.mark.parametrize("kw", [dict(tol=1e-13), dict(tol=1e-3, min_iter=5), dict(tol=1e-12, max_iter=4),
                                dict(tol=0.0, rel_tol=1e-4), dict(Su=9.0, Sp=-0.3),
                                dict(DT_uniform=0.0, DTx=None, DTy=None, DTz=None)],
                         ids=["sweeps", "min_iter", "max_iter", "rel_tol", "sources", "no_diffusion"])
def test_resident_options_bitwise(kw):
    case = case_of((10, 9, 8)).with_(**kw)
    for cuts in ((3,), (1, 1, 1)):
        T, st, _ = run(case, True, 2, 256, cuts)
        T0, st0, _ = run(case, False, 2, 256, cuts)
        assert np.array_equal(T, T0) and st == st0


def test_resident_against_oracle_and_a_field_that_is_not_finite():
    case = case_of((21, 18, 13)).with_(n_steps=3)
    To, _ = oracle.advance(case)
    with Solver.from_case(case) as s:
        s.set_solver(case.tol, 0.0, 1000, 0, B.LFM_MIXED)
        good = s.field().copy()
        s.advance(3)
        assert np.max(np.abs(s.field() - To) / np.abs(To)) <= 1e-5
        bad = good.copy()
        bad[7] = np.nan
        s.set_field(bad)
        with pytest.raises(B.LfmError) as e:
            s.advance(1)
        assert e.value.code == B.LFM_ENONFINITE
        s.set_field(good)
        s.advance(3)
        assert np.max(np.abs(s.field() - To) / np.abs(To)) <= 1e-5


@pytest.mark.parametrize("prec", [B.LFM_DF64, B.LFM_MIXED])
@pytest.mark.parametrize("spread", [1.0, 1e3])
def test_row_differences_near_and_far(prec, spread):
    # neighbouring values within a factor of two take a shorter exact difference; a field over
    # six decades and both signs takes the general one in nearly every row
    case = case_of((9, 8, 7))
    rng = np.random.default_rng(5)
    T0 = 300.0 * (1 + 1e-3 * rng.standard_normal(case.n_cells)) if spread == 1.0 else \
        rng.choice([-1.0, 1.0], case.n_cells) * np.exp(rng.uniform(-np.log(spread), np.log(spread), case.n_cells))
    case = case.with_(T0=T0, n_steps=2)
    To, _ = oracle.advance(case)
    with Solver.from_case(case) as s:
        s.set_solver(case.tol, 0.0, 1000, 0, prec)
        s.advance(2)
        assert np.max(np.abs(s.field() - To)) <= (1e-10 if prec == B.LFM_DF64 else 1e-5) * np.max(np.abs(To))


def run_as(case, prec, on, ctas, threads, cuts=(2, 1)):
    with Solver.from_case(case) as s:
        s.set_solver(case.tol, case.rel_tol, case.max_iter, case.min_iter, prec)
        B.lfm_debug_stage_rows(s.ctx, on)
        s.set_launch(ctas, threads)
        st = []
        for n in cuts:
            st += s.advance(n)
        return s.field().copy(), st


@pytest.mark.parametrize("prec", [B.LFM_FP64, B.LFM_DF64])
@pytest.mark.parametrize("permute", [False, True])
@pytest.mark.parametrize("dims,ctas,threads", SHAPES)
def test_whole_solve_on_chip_bitwise_equal_to_streamed(dims, ctas, threads, permute, prec):
    case = case_of(dims, permute)
    T, st = run_as(case, prec, True, ctas, threads)
    T0, st0 = run_as(case, prec, False, ctas, threads)
    assert np.array_equal(T, T0) and st == st0
    assert max(x["iters"] for x in st) >= 3


@pytest.mark.parametrize("prec", [B.LFM_FP64, B.LFM_DF64])
@pytest.mark.parametrize("kw", [dict(tol=1e-13), dict(tol=1e-3, min_iter=5), dict(tol=1e-12, max_iter=4),
                                dict(tol=0.0, rel_tol=1e-4), dict(Su=9.0, Sp=-0.3), dict(n_nonorth_corr=2),
                                dict(DT_uniform=0.0, DTx=None, DTy=None, DTz=None)],
                         ids=["tight", "min_iter", "max_iter", "rel_tol", "sources", "passes", "no_diffusion"])
def test_whole_solve_on_chip_options(kw, prec):
    case = case_of((10, 9, 8)).with_(**kw)
    for cuts in ((3,), (1, 1, 1)):
        for launch in ((2, 256), (1, 512)):
            T, st = run_as(case, prec, True, *launch, cuts)
            T0, st0 = run_as(case, prec, False, *launch, cuts)
            assert np.array_equal(T, T0) and st == st0


# more than eight rows per thread: the df64 product streams its packed rows through shared memory
@pytest.mark.parametrize("permute", [False, True])
@pytest.mark.parametrize("dims,ctas,threads", [((16, 16, 8), 1, 256), ((16, 16, 9), 1, 256), ((24, 16, 12), 1, 256),
                                               ((20, 20, 13), 2, 256), ((23, 16, 15), 1, 512)])
def test_df64_streamed_rows_by_rows_per_thread(dims, ctas, threads, permute):
    case = case_of(dims, permute)
    out = []
    for on in (True, False):
        with Solver.from_case(case) as s:
            s.set_solver(case.tol, case.rel_tol, case.max_iter, case.min_iter, B.LFM_DF64)
            B.lfm_debug_stage_rows(s.ctx, on)
            s.set_launch(ctas, threads)
            out.append((s.advance(3), s.field().copy(), B.lfm_debug_staged_passes(s.ctx)))
    assert out[0][0] == out[1][0] and np.array_equal(out[0][1], out[1][1])
    rows = -(-(case.n_cells // ctas) // threads)
    assert (out[0][2] > 0) == (not permute and rows > 8 and case.n_cells % 4 == 0) and out[1][2] == 0
