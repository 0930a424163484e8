"""The FP64 batched sweep on the tensor cores against the FP64 CUDA-core sweep.

Both compute the same iterate to FP64 accuracy: digits exact to 2^-63 of a row's and
a column's largest entry, one FP64 rounding per 256 inputs, against one per input.
After K sweeps and the recovery each is within K 8 u cond(K_P) of the exact iterate
(K_P here: diagonals of at least 7, off-diagonals summing to at most 12: cond <= 24;
the reflections do not expand errors), so they differ by at most 2 * 12 * 8 * 24 u
~ 5.2e-13 of the largest value of the column."""
import numpy as np
import pytest
import torch

from oracle import vtm_oracle as O
from paper_0910_0663_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _pair(w, b, data=None, **kw):
    from paper_0910_0663_gb300 import vtm
    out = []
    for bk in (0, 1):
        plan = vtm.Plan(w.indptr, w.indices, w.data if data is None else data, w.partition, w.nparts, Zc=w.Zc,
                        batch_kernel=bk, **kw)
        x, info = plan.solve(torch.from_numpy(b).cuda(), tol=1e-300, check=False)
        assert plan.stats()["batch_kernel"] == (1 if bk else 2)
        out.append((x.cpu().numpy(), info["sweeps"]))
    assert out[0][1] == out[1][1] == kw["max_sweeps"]
    return out[0][0], out[1][0]


@pytest.mark.parametrize("nrhs", [2, 7, 8, 9, 16, 17, 24, 25, 32, 33, 48, 64])
def test_same_iterates_as_the_cuda_cores(nrhs):
    # boxes of up to 400 ports: several chunks of 256 inputs, ragged last blocks
    w = wl.thermal3d(8, 24, 24, 6, nrhs=nrhs, seed=nrhs, min_box=20, max_box=2600)
    x, ref = _pair(w, w.b, max_sweeps=12)
    assert (np.abs(x - ref).max(1) <= 5.2e-13 * np.abs(ref).max(1)).all()


@pytest.mark.parametrize("sweeps", [1, 2, 3])
def test_columns_of_any_size_and_an_unsymmetric_matrix(sweeps):
    # columns from 1e-140 to 1e140 (their squares must fit), a zero column, one that decays over 1e-30 of
    # its largest value; LU factors inside the boxes (the cut stays symmetric)
    w = wl.thermal3d(6, 12, 13, 5, nrhs=9, seed=2, min_box=20, max_box=900)
    rows = np.repeat(np.arange(w.n), np.diff(w.indptr))
    data = w.data.copy()
    data[(w.indices > rows) & (w.partition[rows] == w.partition[w.indices])] *= 0.8
    b = w.b * np.array([1e-140, 1e140, 1.0, 0.0, 1e-30, 1e30, -1.0, 1e100, 1.0])[:, None]
    b[8] *= 10.0 ** -np.linspace(0, 30, w.n)
    x, ref = _pair(w, b, data, max_sweeps=sweeps)
    assert (np.abs(x - ref).max(1) <= 5.2e-13 * np.abs(ref).max(1)).all()
    assert (x[3] == 0).all()


def test_tiles_without_ports_and_non_finite_columns():
    from paper_0910_0663_gb300 import vtm
    w = wl.grid2d(10, 30, 10, 10, ground=0.5, nrhs=3)
    cut = (w.partition[np.repeat(np.arange(w.n), np.diff(w.indptr))] == 2) != (w.partition[w.indices] == 2)
    data = np.where(cut, 0.0, w.data)  # the last tile stands alone
    plan = vtm.Plan(w.indptr, w.indices, data, w.partition, w.nparts)
    x, info = plan.solve(torch.from_numpy(w.b).cuda())
    A = w.csr()
    A.data[:] = data
    assert O.residual_norms(A, x.cpu().numpy(), w.b).max() <= 1e-10
    bad = w.b.copy()
    bad[1, 5] = np.nan
    with pytest.raises(vtm.VTMError, match="diverged"):
        plan.solve(torch.from_numpy(bad).cuda())
    y, _ = plan.solve(torch.from_numpy(w.b).cuda())
    assert torch.equal(x, y)


@pytest.mark.parametrize("nrhs", [2, 6, 33])
def test_columns_with_one_hot_node(nrhs):
    """A column that decays by 1e-20 and more across its boxes keeps its small entries:
    each within 1e-9 of itself of the CUDA cores' (45 sweeps of sums of up to 2000
    products whose waves cancel to 1/64 at a place: 45 * 2000 * 64 u = 6e-10).  Columns
    of random entries lie between them in the same groups of eight."""
    w = wl.thermal3d(8, 24, 24, 8, nrhs=nrhs, seed=1, min_box=20, max_box=2600)
    b = w.b.copy()
    hot = np.random.default_rng(0).integers(0, w.n, nrhs)
    for r in range(0, nrhs, 2):
        b[r] = 0.0
        b[r, hot[r]] = 1.0
    x, ref = _pair(w, b, max_sweeps=45)
    assert (np.abs(ref[0]).max() / np.abs(ref[0]).min()) > 1e20
    assert (np.abs(x - ref)[::2] <= 1e-9 * np.abs(ref[::2])).all()
    assert (np.abs(x - ref).max(1) <= 45 / 12 * 5.2e-13 * np.abs(ref).max(1)).all()
