"""Byte counts of the bench's roofline for launches on packed meshes (CPU): no more than the indexed counts, and
no more than what the arrays' passes move."""
import importlib.util
import os

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def bench():
    spec = importlib.util.spec_from_file_location("bench_packed_under_test", os.path.join(ROOT, "bench.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return mod


@pytest.mark.parametrize("late", [False, True])
@pytest.mark.parametrize("form,b", [("fp64", 8), ("df64", 8), ("mixed", 4)])
def test_packed_counts(bench, form, b, late):
    if form == "fp64" and late:
        pytest.skip("FP64 has no late form")
    N, F = 1000, 2970
    # the passes of one solve of k iterations, array by array
    field = {"fp64": 8, "df64": 12, "mixed": 12}[form]

    def solve(k):
        p = (k - 1) * (5 if late else 3) * b * N - (b * N if late and k > 1 else 0)  # the first update reads no e
        m = k * (4 * N + 4 * b * N - b * N + b * F)
        u = k * (5 if late else 8) * b * N
        if not late and form != "fp64":
            u -= b * N  # the first update writes the correction without reading it
        end = (3 if k > 1 else 2) * b * N if late else 0
        return p + m + u + end

    rest = {"fp64": 8 * N + (8 * 5 + 4) * N + 16 * N - 8 * N + 8 * F,
            "df64": (field * 2 + 8) * N + (field + 4 + 8 + 8 + 16) * N + 8 * F,
            "mixed": (field * 3 + 4) * N + (2 * field + 4 + 8 + 4 + 12) * N + 8 * F}[form]
    for k in (2, 5, 9):
        assert bench.packed_bytes(N, F, k, 1, form, late) == solve(k) + rest
    assert bench.packed_bytes(N, F, 14, 3, form, late) == pytest.approx(solve(5) * 2 + solve(4) + 3 * rest)


@pytest.mark.parametrize("form", ["fp64", "df64", "mixed"])
def test_packed_counts_lie_below_the_indexed_ones(bench, form):
    n = 600
    N, F = n ** 3, 3 * n * n * (n - 1)
    old = bench.algorithmic_bytes(N, F, 283, 20, 1 if form == "mixed" else 0)
    assert bench.packed_bytes(N, F, 283, 20, form, form != "fp64") < 0.9 * old
    assert bench.algorithmic_bytes_corrected(N, F, 10, 2, True) < bench.algorithmic_bytes_corrected(N, F, 10, 2)
