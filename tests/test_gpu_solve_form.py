"""Which solves stay on chip, as the device notes it, and that they equal the streamed ones bit for bit, at the
rows per thread where one form takes over from another and at sizes of the default launch (GPU required)."""
import numpy as np
import pytest

import lapcase
from paper_2507_18268_gb300 import Solver
from paper_2507_18268_gb300 import binding as B

pytestmark = pytest.mark.gpu

PRECS = [B.LFM_FP64, B.LFM_MIXED, B.LFM_DF64]

# six slots; rows per thread 1, 2, 3 of 256 and 1, 4, 5, 6, 7 of 512; N a multiple of 4 and not; several CTAs
SHAPES = [((8, 8, 4), 1, 256), ((8, 8, 8), 1, 256), ((9, 8, 8), 1, 256), ((7, 9, 5), 1, 256), ((11, 10, 10), 3, 256),
          ((11, 10, 10), 40, 256), ((16, 10, 3), 1, 512), ((16, 16, 8), 1, 512), ((17, 16, 8), 1, 512),
          ((16, 16, 12), 1, 512), ((17, 15, 12), 1, 512), ((20, 16, 10), 1, 512), ((15, 13, 11), 1, 512),
          ((31, 13, 11), 3, 512)]


def case_of(dims, permute=False):
    return lapcase.random_small_case(sum(dims), *dims, permute=permute).with_(tol=1e-8, dt=0.2)


def run(case, prec, on, ctas=0, threads=0):
    with Solver.from_case(case) as s:
        s.set_solver(case.tol, 0.0, 1000, 0, prec)
        B.lfm_debug_stage_rows(s.ctx, on)
        packed = B.lfm_debug_pack_slots(s.ctx, True) > 0
        if threads:
            s.set_launch(ctas, threads)
        st = s.advance(2) + s.advance(1)
        return s.field().copy(), st, B.lfm_debug_solve_form(s.ctx), packed, s.launch()


def form(prec, packed, n, ctas, threads):
    """Rows per thread of the kernel that keeps a case's solves on chip (0: none does)."""
    chunk = -(-(-(-n // ctas)) // 32) * 32
    rows = -(-chunk // threads)
    if threads == 256:
        return 2 if rows <= 2 else 0
    held = {B.LFM_FP64: [], B.LFM_MIXED: [4, 6], B.LFM_DF64: [4]}[prec] if packed else []
    return next((r for r in held if rows <= r), 0)


def check(case, prec, want_packed, ctas=0, threads=0):
    T, st, rows, packed, launch = run(case, prec, True, ctas, threads)
    T0, st0, rows0, _, _ = run(case, prec, False, ctas, threads)
    assert packed == want_packed and rows0 == 0
    assert rows == form(prec, packed, case.n_cells, *launch)
    assert max(x["iters"] for x in st) >= 3
    assert np.array_equal(T, T0) and st == st0
    return rows, launch


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("permute", [False, True])
@pytest.mark.parametrize("dims,ctas,threads", SHAPES)
def test_form_by_rows_per_thread(dims, ctas, threads, permute, prec):
    check(case_of(dims, permute), prec, not permute, ctas, threads)


# the default launch on many CTAs: (cells, permuted) -> rows per thread kept on chip in FP64, mixed, df64
DEFAULTS = [((41, 37, 43), False, (2, 2, 2)), ((41, 37, 43), True, (2, 2, 2)), ((64, 64, 60), False, (0, 4, 4)),
            ((63, 65, 61), False, (0, 4, 4)), ((64, 64, 60), True, (0, 0, 0)), ((96, 96, 90), False, (0, 6, 0))]


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("dims,permute,want", DEFAULTS)
def test_default_launches(dims, permute, want, prec):
    rows, launch = check(case_of(dims, permute), prec, not permute)
    assert launch[0] >= 100
    assert rows == want[PRECS.index(prec)]
