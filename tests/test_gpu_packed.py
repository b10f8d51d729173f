"""Packed slots (the neighbours of a six-slot row as one word of four-bit codes) against the slot
rows they replace (GPU required).

A mesh packs when its neighbour distances take at most 16 values. Both readings give every thread
the same cells and every value the same operations in the same order, so fields and statistics must
agree bit for bit, in every form and through batches and shared meshes; meshes that do not pack run
as before.
"""
import numpy as np
import pytest

import lapcase
import oracle
from paper_2507_18268_gb300 import Solver
from paper_2507_18268_gb300 import binding as B
from paper_2507_18268_gb300.batch import Batch

pytestmark = pytest.mark.gpu

PRECS = [B.LFM_FP64, B.LFM_MIXED, B.LFM_DF64]


def case_of(nx, ny, nz, perm=None, **kw):
    c = lapcase.random_small_case(nx + 10 * ny + 100 * nz, nx, ny, nz, permute=False)
    return c.with_(perm=perm, tol=1e-10, **kw)


def block_perm(n, block):
    """Labels in reversed order inside every block of cells: a few more distances than natural order."""
    lab = np.arange(n)
    for a in range(0, n, block):
        lab[a:a + block] = lab[a:a + block][::-1]
    return lab.astype(np.int64)


# (case, whether it packs): the smallest six-slot box, ragged sizes (N not a multiple of 4), sizes
# around one CTA's threads, a box of more CTAs than SMs, reversed numbering, and meshes with too
# many distances or fewer than six slots
CASES = {
    "3x3x3": (lambda: case_of(3, 3, 3), True),
    "7x5x3": (lambda: case_of(7, 5, 3), True),
    "8x8x8": (lambda: case_of(8, 8, 8), True),
    "9x19x3": (lambda: case_of(9, 19, 3), True),
    "41x37x29": (lambda: case_of(41, 37, 29), True),
    "reversed": (lambda: case_of(11, 7, 5, perm=np.arange(385)[::-1].astype(np.int64)), True),
    "blocks4": (lambda: case_of(8, 8, 8, perm=block_perm(512, 4)), True),   # 9 distances
    "blocks5": (lambda: case_of(8, 8, 8, perm=block_perm(512, 5)), False),  # 17: one too many
    "random": (lambda: case_of(9, 8, 7, perm=np.random.default_rng(3).permutation(504).astype(np.int64)), False),
    "flat": (lambda: case_of(16, 9, 1), False),
    "sources": (lambda: case_of(10, 9, 8, Su=20.0, Sp=-0.1), True),
    "skew": (lambda: lapcase.skewed_box(12, n_steps=3), True),
}


def run(case, prec, on, threads=0, ctas=0):
    with Solver.from_case(case) as s:
        n = B.lfm_debug_pack_slots(s.ctx, on)
        s.set_solver(case.tol, case.rel_tol, case.max_iter, case.min_iter, prec)
        if threads:
            s.set_launch(ctas, threads)
        a = s.advance(2)
        a += s.advance(1)
        return n, s.field().copy(), a


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("name", list(CASES))
def test_packed_bitwise_equal_to_slot_rows(name, prec):
    make, packs = CASES[name]
    case = make()
    for threads, ctas in ((0, 0), (256, 3)):
        n, T, st = run(case, prec, True, threads, ctas)
        _, T0, st0 = run(case, prec, False, threads, ctas)
        assert (0 < n <= 16) == packs, n
        assert np.array_equal(T, T0) and st == st0


def test_packed_batch_and_shared_mesh():
    cases = [case_of(9, 8, 7).with_(precision=p, n_steps=3, DTx=None, DTy=None, DTz=None, DT_uniform=2e-2)
             for p in PRECS]
    for form in (cases, cases[:1] * 2, cases[2:] * 2):  # one kernel per precision and the mixed one
        got = []
        for on in (True, False):
            with Batch() as b:
                first = Solver.from_box_case(form[0])
                solvers = [first] + [Solver.sharing(first, c) for c in form[1:]]
                for s in solvers:
                    assert B.lfm_debug_pack_slots(s.ctx, on) > 0
                ids = [b.add(s) for s in solvers]
                b.advance(3)
                got.append([b.field(i).copy() for i in ids])
                for i in reversed(ids):
                    b.remove(i)
        for x, y in zip(*got):
            assert np.array_equal(x, y)


@pytest.mark.parametrize("prec", PRECS)
def test_packed_against_oracle(prec):
    case = case_of(21, 18, 13)
    To, so = oracle.advance(case)
    _, T, st = run(case.with_(n_steps=3), prec, True)
    assert np.max(np.abs(T - To) / np.abs(To)) <= (1e-5 if prec == B.LFM_MIXED else 1e-10)
    if prec != B.LFM_MIXED:
        assert [x["iters"] for x in st] == [x.iters for x in so]
