"""FP64 solves kept on chip on general (non-orthogonal) meshes against the streamed solve (GPU required).

A pass on such a mesh starts with the gradient of T, which gathers neighbours that other threads and
CTAs updated in the solve before, so the solve's last barrier has to order those updates. The two forms
give every value the same operations and every sum the same order: fields and records agree bit for bit,
run after run, over steps and corrector passes of one launch and over several launches.
"""
import numpy as np
import pytest

import lapcase
from paper_2507_18268_gb300 import Solver
from paper_2507_18268_gb300 import binding as B

pytestmark = pytest.mark.gpu


def perturbed(dims):
    return lapcase.perturbed_box(lapcase.random_small_case(sum(dims), *dims, permute=False), amp=0.3, seed=7)


# one CTA; a few; one row per thread and a CTA on most SMs; two rows per thread, N not a multiple of 4
CASES = {
    "perturbed6x5x4": lambda: perturbed((6, 5, 4)),
    "perturbed11x10x9": lambda: perturbed((11, 10, 9)),
    "skewed31": lambda: lapcase.skewed_box(31),
    "perturbed41x37x43": lambda: perturbed((41, 37, 43)),
}


def run(s, T0, cuts, on):
    B.lfm_debug_stage_rows(s.ctx, on)
    s.set_field(T0)
    st = []
    for n in cuts:
        st += s.advance(n)
    return s.field().copy(), st


@pytest.mark.parametrize("n_corr", [0, 2])
@pytest.mark.parametrize("name", list(CASES))
def test_on_chip_equals_streamed_repeatedly(name, n_corr):
    case = CASES[name]().with_(tol=1e-9, dt=0.05, n_nonorth_corr=n_corr)
    with Solver.from_case(case) as s:
        s.set_solver(case.tol, 0.0, case.max_iter, 0, B.LFM_FP64)
        T0 = s.field().copy()
        want, st = run(s, T0, (3,), False)
        assert all(x["iters"] > 0 for x in st)
        for k in range(12):
            T, st1 = run(s, T0, (3,) if k % 3 else (1, 2), True)
            assert np.array_equal(T, want) and st1 == st, k
