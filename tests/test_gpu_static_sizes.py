"""The allocation-free solve over the sizes at which its launch changes (GPU required): one CTA and
several, one cell per thread and more, full CTAs and ragged ones, systems without faces, cells
without owned faces; each solution against a direct sparse solve.

A is strictly diagonally dominant by at least 1, so |x - x*| <= sum|b - A x| in every cell, which the
solve brings below tol * normFactor (and rounding: 1e-13 of the solution).
"""
import numpy as np
import pytest

from paper_2507_18268_gb300 import binding as B

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 31, 255, 256, 257, 513, 5000, 38911, 38912, 38913, 65535, 65536]


def system(n, reach, rng):
    """Faces c - c + 1 and, every third cell, c - c + reach."""
    pairs = [np.stack([np.arange(n - 1), np.arange(1, n)], 1)]
    if 0 < reach < n:
        own = np.arange(0, n - reach, 3)
        pairs.append(np.stack([own, own + reach], 1))
    p = np.unique(np.concatenate(pairs), axis=0) if n > 1 else np.zeros((0, 2), dtype=np.int64)
    p = p[np.lexsort((p[:, 1], p[:, 0]))]
    upper = -rng.uniform(0.1, 1.0, len(p))
    diag = 1.0 + rng.uniform(0.0, 1.0, n)
    np.add.at(diag, p[:, 0], -upper)
    np.add.at(diag, p[:, 1], -upper)
    return p[:, 0].astype(np.int32), p[:, 1].astype(np.int32), diag, upper


def solve(owner, neighbour, diag, upper, source, x0, tol):
    import torch
    dev = [torch.as_tensor(a, device="cuda") for a in (owner, neighbour, diag, upper, source, x0)]
    rc, st = B.lfm_pcg_solve_static(len(diag), len(owner), *[d.data_ptr() for d in dev], tol)
    assert rc == B.LFM_OK, B.lfm_last_error()
    return dev[-1].cpu().numpy(), st


@pytest.mark.parametrize("faces", [True, False])
@pytest.mark.parametrize("n", SIZES)
def test_static_solve_over_sizes(n, faces):
    sp = pytest.importorskip("scipy.sparse")
    from scipy.sparse.linalg import spsolve
    rng = np.random.default_rng(n)
    owner, neighbour, diag, upper = system(n, 97, rng)
    if not faces:
        owner, neighbour, upper = owner[:0], neighbour[:0], upper[:0]
    source, x0 = rng.uniform(-1.0, 1.0, n), rng.uniform(-1.0, 1.0, n)
    tol = 1e-11
    x, st = solve(owner, neighbour, diag, upper, source, x0, tol)
    A = sp.coo_matrix((np.concatenate([diag, upper, upper]),
                       (np.concatenate([np.arange(n), owner, neighbour]),
                        np.concatenate([np.arange(n), neighbour, owner])))).tocsc()
    want = spsolve(A, source)
    assert st.converged == 1
    assert np.max(np.abs(x - want)) <= tol * st.norm_factor + 1e-13 * np.max(np.abs(want)) * (1 + len(owner) / n)
    again, st2 = solve(owner, neighbour, diag, upper, source, x0, tol)
    assert np.array_equal(again, x) and st2.iters == st.iters
