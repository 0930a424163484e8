"""Channel-form sweeps (lagged couplings, block Jacobi) in their two forms.

Up to 768 output pairs per CTA every sweep runs in one launch (equal ranges of
output pairs, several tiles or parts of one per CTA); larger plans launch one
kernel per sweep.  Small cases are compared with the
oracle's history; the iterate that is returned and the history must belong
together in both forms, whatever sweep the run ends with.
"""
import numpy as np
import pytest
import torch

from oracle import vtm_oracle as O
from paper_0910_0663_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vtm():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_0910_0663_gb300 import build
    build.build()
    from paper_0910_0663_gb300 import vtm as V
    return V


# one CTA; ragged tiles of 1 to 9 rows (odd output counts, tiles of a few
# channels); tiles shared by several CTAs and streamed elements
@pytest.mark.parametrize("n,ty,tx,method", [(6, 3, 3, "vtm"), (31, 7, 9, "vtm"), (31, 3, 31, "bj"),
                                            (160, 80, 54, "vtm"), (96, 12, 12, "bj")])
def test_history_matches_oracle(vtm, n, ty, tx, method):
    w = wl.vccs_grid(n, n, ty, tx, seed=11)
    A = w.csr()
    plan = vtm.Plan(w.indptr, w.indices, w.data, w.partition, w.nparts, Zc=1.0, method=method)
    plan.set_options(history_len=30, max_sweeps=30)
    plan.solve(torch.from_numpy(w.b).cuda(), tol=1e-13, check=False)
    if method == "vtm":
        ref = O.vtm_midpoint(A, w.partition, w.nparts, w.b, W=1.0, tol=0, max_sweeps=30).history[:, 0]
    else:
        ref = O.block_jacobi(A, w.partition, w.nparts, w.b, tol=0, max_sweeps=30)[3][:, 0]
    h = np.asarray(plan.history)
    m = h > 0  # entries past convergence stay zero
    assert m.sum() >= min(20, (ref > 1e-12).sum())
    assert np.allclose(h[m], ref[:len(h)][m], rtol=1e-9, atol=1e-13)


# residual of the returned iterate against the history entry of that sweep: both are
# sums of products of size |b| in FP64, so 1e-12 of ||b|| apart at most
@pytest.mark.parametrize("n,tile", [(48, 12), (200, 50), (1024, 8)])
@pytest.mark.parametrize("sweeps", [1, 2, 3, 9])
def test_returned_iterate_is_the_sweep_asked_for(vtm, n, tile, sweeps):
    w = wl.vccs_grid(n, n, tile, tile, seed=12)
    A = w.csr()
    plan = vtm.Plan(w.indptr, w.indices, w.data, w.partition, w.nparts, Zc=1.0)
    plan.set_options(history_len=12, max_sweeps=12)
    b = torch.from_numpy(w.b).cuda()
    plan.solve(b, tol=1e-15, check=False)
    h = np.array(plan.history)
    plan.set_options(history_len=12, max_sweeps=sweeps)
    x, info = plan.solve(b, tol=1e-15, check=False)
    assert info["sweeps"] == sweeps
    r = O.residual_norms(A, x.cpu().numpy().reshape(w.b.shape), w.b).max()
    assert abs(r - h[sweeps - 1]) <= 1e-12 + 1e-9 * r
    tol = float(h[4] * 1.0000001)  # converges at the sweep the history gives
    k = int(np.argmax(h <= tol)) + 1
    plan.set_options(history_len=12, max_sweeps=12)
    x, info = plan.solve(b, tol=tol, check=False)
    assert info["sweeps"] == k
    r = O.residual_norms(A, x.cpu().numpy().reshape(w.b.shape), w.b).max()
    assert abs(r - h[k - 1]) <= 1e-12 + 1e-9 * r


@pytest.mark.parametrize("limit", [1 << 30, (1 << 31) - 1])
def test_a_sweep_limit_above_what_the_barrier_counts(vtm, limit):
    """Up to 2^31 arrivals of all CTAs together run in one launch, more take a launch
    per sweep."""
    w = wl.vccs_grid(200, 200, 50, 50, seed=12)
    plan = vtm.Plan(w.indptr, w.indices, w.data, w.partition, w.nparts, Zc=1.0)
    b = torch.from_numpy(w.b).cuda()
    x, info = plan.solve(b, tol=1e-9)
    assert info["kernel_launches"] < info["sweeps"]
    plan.set_options(max_sweeps=limit)
    y, many = plan.solve(b, tol=1e-9)
    assert many["kernel_launches"] > many["sweeps"]
    assert abs(many["sweeps"] - info["sweeps"]) <= 1  # (sums in another order)
    assert O.residual_norms(w.csr(), y.cpu().numpy().reshape(w.b.shape), w.b).max() <= 1e-9


def test_wait_polls_bounds_the_channel_form_too(vtm):
    w = wl.vccs_grid(200, 200, 50, 50, seed=12)
    plan = vtm.Plan(w.indptr, w.indices, w.data, w.partition, w.nparts, Zc=1.0)
    b = torch.from_numpy(w.b).cuda()
    x, _ = plan.solve(b)
    plan.set_options(wait_polls=1)  # the first poll that finds the barrier open gives up
    with pytest.raises(vtm.VTMError, match="timed out"):
        plan.solve(b)
    plan.set_options(wait_polls=0)
    y, _ = plan.solve(b)
    assert torch.equal(x, y)
