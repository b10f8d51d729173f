"""The matrix is assembled in a launch's first pass and its boundary faces' terms are laid out when
the case changes (GPU required): after any change to a case, the next steps equal those of a fresh
context that was given the final settings, bit for bit, and many steps in one launch equal the same
steps in launches of one.
"""
import numpy as np
import pytest

import lapcase
from paper_2507_18268_gb300 import Solver
from paper_2507_18268_gb300 import binding as B

pytestmark = pytest.mark.gpu

PRECS = [B.LFM_FP64, B.LFM_MIXED, B.LFM_DF64]


def base():
    c = lapcase.random_small_case(77, 9, 7, 6, permute=True, patch_types=[0, 0, 1, 0, 1, 1])
    return c.with_(tol=1e-9)


def change_value(s, m):
    B.lfm_set_patch(s.ctx, 0, lapcase.FIXED_VALUE, None, 311.0)


def change_values(s, m):
    n = int(m.patch_size[3])
    B.lfm_set_patch(s.ctx, 3, lapcase.FIXED_VALUE, np.linspace(280.0, 360.0, n), 0.0)


def change_type(s, m):
    B.lfm_set_patch(s.ctx, 0, lapcase.ZERO_GRADIENT, None, 0.0)
    B.lfm_set_patch(s.ctx, 4, lapcase.FIXED_VALUE, None, 290.0)


def change_dt(s, m):
    B.lfm_set_time_step(s.ctx, 0.037)


def change_DT(s, m):
    B.lfm_set_diffusivity(s.ctx, 0.0, 1.7 * m.DT_faces, 0.4 * m.DT_bfaces)


def change_cells(s, m):
    B.lfm_set_diffusivity_cells(s.ctx, np.linspace(1e-3, 2e-2, m.n_cells), m.weights)


def change_source(s, m):
    B.lfm_set_source(s.ctx, np.full(m.n_cells, 12.0), np.full(m.n_cells, -0.2))


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("change", [change_value, change_values, change_type, change_dt, change_DT, change_cells,
                                    change_source])
def test_change_between_advances_equals_fresh_context(change, prec):
    case = base()
    out = []
    for warm in (True, False):
        with Solver.from_case(case) as s:
            s.set_solver(case.tol, 0.0, 1000, 0, prec)
            T0 = s.field().copy()
            if warm:
                s.advance(3)
            change(s, s.mesh)
            s.set_field(T0)
            st = s.advance(2)
            out.append((s.field().copy(), st))
    assert np.array_equal(out[0][0], out[1][0]) and out[0][1] == out[1][1]


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("name", ["plain", "sources", "skew"])
def test_steps_in_one_launch_equal_launches_of_one(name, prec):
    case = {"plain": base, "sources": lambda: base().with_(Su=9.0, Sp=-0.3),
            "skew": lambda: lapcase.skewed_box(9, n_steps=4)}[name]()
    out = []
    for cuts in ((4,), (1, 1, 1, 1), (1, 3)):
        with Solver.from_case(case) as s:
            s.set_solver(case.tol, 0.0, 1000, 0, prec)
            st = []
            for n in cuts:
                st += s.advance(n)
            out.append((s.field().copy(), st))
    for T, st in out[1:]:
        assert np.array_equal(out[0][0], T) and out[0][1] == st
