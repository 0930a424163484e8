"""Blocked single-column band solves (half bandwidths above 32).

A circuit in one part is one direct band solve, so its first answer has the
solver's own accuracy: with a ground of 1 S on every node cond(A) <= 17 and the
FP64 error stays below 17 * 64 u ~ 1.2e-13 (64 covers the growth of rounding
along a row's band and inverse)."""
import numpy as np
import pytest
import scipy.sparse as sp
import scipy.sparse.linalg as sla
import torch

from paper_0910_0663_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _grid(width, length, unsymmetric, nparts=1, seed=0):
    w = wl.grid2d(length, width, length, width, ground=1.0, seed=seed)
    data = w.data.copy()
    if unsymmetric:  # scaled off-diagonals above the diagonal: LU factors
        rows = np.repeat(np.arange(w.n), np.diff(w.indptr))
        data[w.indices > rows] *= 0.8
    part = (np.arange(w.n) * nparts // w.n).astype(np.int32)
    return w, data, part


@pytest.mark.parametrize("unsymmetric", [False, True])
@pytest.mark.parametrize("width,length", [(33, 34), (47, 60), (64, 64), (65, 70), (96, 100), (97, 120), (128, 130),
                                          (129, 140), (200, 203), (256, 260), (257, 258)])
def test_one_part_is_solved_at_once(width, length, unsymmetric):
    from paper_0910_0663_gb300 import vtm
    w, data, part = _grid(width, length, unsymmetric)
    plan = vtm.Plan(w.indptr, w.indices, data, part, 1)
    assert plan.stats()["max_band"] == width
    x, info = plan.solve(torch.from_numpy(w.b[0]).cuda(), tol=1e-10)
    A = w.csr()
    A.data[:] = data
    ref = sla.spsolve(A.tocsc(), w.b[0])
    assert info["outer_steps"] == 1
    assert np.linalg.norm(x.cpu().numpy() - ref) <= 1.2e-13 * np.linalg.norm(ref)


@pytest.mark.parametrize("width", [33, 64, 100, 128, 160])
def test_fp32_sweeps_with_wide_bands(width):
    from paper_0910_0663_gb300 import vtm
    w, data, part = _grid(width, 3 * width, False, nparts=3)
    plan = vtm.Plan(w.indptr, w.indices, data, part, 3, precision="fp32")
    assert plan.stats()["max_band"] >= 33
    x, info = plan.solve(torch.from_numpy(w.b[0]).cuda(), tol=1e-10)
    ref = sla.spsolve(w.csr().tocsc(), w.b[0])
    # cond(A) <= 17 turns the residual bound into one of the error
    assert info["relres"] <= 1e-10
    assert np.linalg.norm(x.cpu().numpy() - ref) <= 17e-10 * np.linalg.norm(ref)


@pytest.mark.parametrize("multiplier", [-1.8, -0.5])
def test_large_multipliers_are_substituted(multiplier):
    """A = L U with a chain of multipliers in L.  Blocks of a chain of -1.8 have a condition
    of 1.8^32 and more: products with their inverses leave a residual near 1e-9
    (1.8^32 u / 16), substitution a few u, and so do the inverses of a chain of -0.5.
    At 1e-10 one direct solve tells them apart."""
    from paper_0910_0663_gb300 import vtm
    rng = np.random.default_rng(1)
    n, bw = 64, 40
    off = np.subtract.outer(np.arange(n), np.arange(n))
    L = np.where((off > 0) & (off <= bw), rng.uniform(-0.01, 0.01, (n, n)), 0.0) + np.eye(n)
    L[off == 1] = multiplier
    U = np.where((off < 0) & (off >= -bw), rng.uniform(-0.01, 0.01, (n, n)), 0.0) + np.eye(n)
    A = sp.csr_matrix(np.where(np.abs(off) <= bw, L @ U, 0.0))
    A.sort_indices()
    x0 = rng.uniform(-1, 1, n)
    b = A @ x0
    plan = vtm.Plan(A.indptr.astype(np.int64), A.indices.astype(np.int32), A.data, np.zeros(n, np.int32), 1)
    assert plan.stats()["max_band"] == bw
    x, info = plan.solve(torch.from_numpy(b).cuda(), tol=1e-10)
    assert info["outer_steps"] == 1
    assert np.linalg.norm(b - A @ x.cpu().numpy()) <= 1e-10 * np.linalg.norm(b)
