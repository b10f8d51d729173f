"""A batch's captured launch takes the step count of each advance when it is launched (GPU required):
advances of different lengths through one graph against direct launches, a case that fails midway, and
capped advances, bit for bit with their records."""
import numpy as np
import pytest

import lapcase
from paper_2507_18268_gb300 import binding as B
from paper_2507_18268_gb300.batch import Batch

pytestmark = pytest.mark.gpu


def mixed_cases():
    out = []
    for i, c in enumerate(lapcase.batch_cases(n_cases=6, seed=3, n_min=5, n_max=18, n_steps=3)):
        out.append(c.with_(precision=[lapcase.FP64, lapcase.MIXED, lapcase.DF64][i % 3]))
    return out


@pytest.mark.parametrize("counts", [(1,), (3, 1, 4), (1, 7, 2)])
def test_one_graph_serves_advances_of_any_length(counts):
    runs = []
    for use_graph in (True, False):
        with Batch() as bt:
            ids = [bt.add_case(c) for c in mixed_cases()]
            rec = []
            for n in counts:
                assert bt.advance(n, use_graph=use_graph) == B.LFM_OK
                rec.append([(bt.stats(i, n), bt.results()[i]) for i in ids])
            bt.advance_capped_async(3, {ids[0]: 1, ids[2]: 0}, use_graph)
            assert bt.finish() == B.LFM_OK
            rec.append([bt.results()[i] for i in ids])
            runs.append((rec, [bt.field(i).copy() for i in ids]))
    assert runs[0][0] == runs[1][0]
    assert [r[1] for r in runs[0][0][-1]] == [1, 3, 0, 3, 3, 3]
    for a, b in zip(runs[0][1], runs[1][1]):
        assert np.array_equal(a, b)


def test_a_failing_case_leaves_the_others_and_the_next_advance_unharmed():
    runs = []
    for use_graph in (True, False):
        with Batch() as bt:
            ids = [bt.add_case(c) for c in mixed_cases()]
            good = bt.field(ids[0]).copy()
            bad = good.copy()
            bad[3] = np.nan
            bt.cases[ids[0]].set_field(bad)
            assert bt.advance(4, use_graph=use_graph) == B.LFM_ENONFINITE
            assert bt.status(ids[0]) == B.LFM_ENONFINITE
            rec = [bt.stats(i, 4) for i in ids[1:]]
            bt.cases[ids[0]].set_field(good)
            assert bt.advance(2, use_graph=use_graph) == B.LFM_OK
            rec += [bt.stats(i, 2) for i in ids]
            runs.append((rec, [bt.field(i).copy() for i in ids]))
    assert runs[0][0] == runs[1][0]
    for a, b in zip(runs[0][1], runs[1][1]):
        assert np.array_equal(a, b)
