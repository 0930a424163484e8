"""Blocked single-column band solves (half bandwidths above 32).

A circuit in one part is one direct band solve, so its first answer has the
solver's own accuracy: with a ground of 1 S on every node cond(A) <= 17 and the
FP64 error stays below 17 * 64 u ~ 1.2e-13 (64 covers the growth of rounding
along a row's band and inverse)."""
import numpy as np
import pytest
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
