"""Panel factorisation of the bands: ends of panels and windows, one tile.

A circuit in one part is one factorisation and one direct solve; with a ground
of 1 S on every node cond(A) <= 17, so its FP64 error stays below
17 * 64 u ~ 1.2e-13 (as in the blocked band solves' test)."""
import numpy as np
import pytest
import scipy.sparse.linalg as sla
import torch

from paper_0910_0663_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("unsymmetric", [False, True])
@pytest.mark.parametrize("width,length", [(1, 2), (1, 17), (2, 8), (3, 5), (7, 9), (8, 8), (15, 16), (16, 16), (16, 31),
                                          (17, 40), (31, 33), (32, 32), (48, 49), (49, 60), (101, 110), (102, 110),
                                          (103, 110), (140, 150), (141, 150), (150, 155)])
def test_one_part(width, length, unsymmetric):
    from paper_0910_0663_gb300 import vtm
    w = wl.grid2d(length, width, length, width, ground=1.0, seed=width)
    data = w.data.copy()
    if unsymmetric:
        rows = np.repeat(np.arange(w.n), np.diff(w.indptr))
        data[w.indices > rows] *= 0.8
    plan = vtm.Plan(w.indptr, w.indices, data, w.partition, 1)
    x, info = plan.solve(torch.from_numpy(w.b[0]).cuda(), tol=1e-10)
    A = w.csr()
    A.data[:] = data
    ref = sla.spsolve(A.tocsc(), w.b[0])
    assert info["outer_steps"] == 1
    assert np.linalg.norm(x.cpu().numpy() - ref) <= 1.2e-13 * np.linalg.norm(ref)


@pytest.mark.parametrize("width", [8, 32, 64])
def test_a_bad_pivot_is_reported(width):
    from paper_0910_0663_gb300 import vtm
    w = wl.grid2d(3 * width, width, width, width, ground=1.0)
    data = w.data.copy()
    rows = np.repeat(np.arange(w.n), np.diff(w.indptr))
    k = width * width + width * width // 2  # a node inside the second tile
    data[(rows == k) & (w.indices == k)] = -50.0
    with pytest.raises(vtm.VTMError, match="bad pivot in sub-circuit 1"):
        vtm.Plan(w.indptr, w.indices, data, w.partition, w.nparts)


@pytest.mark.parametrize("unsymmetric", [False, True])
@pytest.mark.parametrize("kind", ["checkerboard", "scattered", "mixed"])
def test_tiles_without_inner_branches(kind, unsymmetric):
    """Half bandwidth 0: nothing lies below a panel, its columns are refilled all the
    same.  With a ground of 1 S (cond(A) <= 17) a residual of 1e-12 bounds the error
    by 17e-12."""
    from paper_0910_0663_gb300 import vtm
    ny, nx = 23, 31
    w = wl.grid2d(ny, nx, ny, nx, ground=1.0, seed=3)
    r, c = np.divmod(np.arange(w.n), nx)
    if kind == "checkerboard":
        part = (r + c) % 2
    elif kind == "scattered":  # eight tiles, no two nodes of one adjacent
        part = (2 * r + c) % 8
    else:  # a tile of half bandwidth 23 beside two of half bandwidth 0
        part = np.where(c < 16, 0, 1 + (r + c) % 2)
    data = w.data.copy()
    if unsymmetric:  # (the branches across the cut stay lines)
        rows = np.repeat(np.arange(w.n), np.diff(w.indptr))
        if kind == "mixed":
            data[(w.indices > rows) & (part[rows] == part[w.indices])] *= 0.8
        else:
            data[w.indices > rows] *= 0.8
    plan = vtm.Plan(w.indptr, w.indices, data, part.astype(np.int32), int(part.max()) + 1)
    x, info = plan.solve(torch.from_numpy(w.b[0]).cuda(), tol=1e-12)
    A = w.csr()
    A.data[:] = data
    ref = sla.spsolve(A.tocsc(), w.b[0])
    assert np.linalg.norm(x.cpu().numpy() - ref) <= 17e-12 * np.linalg.norm(ref)
