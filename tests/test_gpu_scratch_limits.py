"""Workspaces that only make a call faster do not make it fail: with the device's
memory nearly taken the kernels that need none of them serve.

The bars are those of the same solves with memory to spare (1e-10 of ||b|| asked for)."""
import numpy as np
import pytest
import torch

from paper_0910_0663_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


class _Full:
    """Takes the device's free memory but for `left` bytes."""

    def __init__(self, left):
        torch.cuda.empty_cache()
        free, _ = torch.cuda.mem_get_info()
        self.block = torch.empty(max(free - left, 0), dtype=torch.uint8, device="cuda") if free > left else None

    def release(self):
        self.block = None
        torch.cuda.empty_cache()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_factor_and_solve_without_room_for_the_inverses(precision):
    from paper_0910_0663_gb300 import vtm
    # 537 MB of inverses (FP32 sweeps: 805), 118 MB of T_P; FP32 sweeps 545 MB of factors
    w = wl.grid2d(1024, 1024, 64, 64, ground=0.1, seed=1)
    b = torch.from_numpy(w.b[0]).cuda()
    plan = vtm.Plan(w.indptr, w.indices, w.data, w.partition, w.nparts, precision=precision, factor=False)
    torch.cuda.synchronize()
    full = _Full(480 << 20 if precision == "fp64" else 1000 << 20)
    try:
        plan.factor()
        x, info = plan.solve(b, tol=1e-10)
    finally:
        full.release()
    plan.factor()  # with room again
    y, again = plan.solve(b, tol=1e-10)
    assert info["relres"] <= 1e-10 and again["relres"] <= 1e-10


def test_batched_solve_where_the_digits_would_take_the_rest():
    """Room for the digits of T_P (18 bytes per entry) or for the columns' buffers, not
    for both: the FP64 sweep on the CUDA cores serves, and the digits again with room."""
    from paper_0910_0663_gb300 import vtm
    w = wl.thermal3d(16, 48, 48, 20, nrhs=64, seed=4, min_box=200, max_box=4000)
    b = torch.from_numpy(w.b).cuda()
    plan = vtm.Plan(w.indptr, w.indices, w.data, w.partition, w.nparts)
    p = np.bincount(plan.ports()[2], minlength=w.nparts)
    digits = int(((p + 15) // 16 * ((p + 7) // 8) * 9 * 256).sum())
    torch.cuda.synchronize()
    full = _Full(digits + (120 << 20))
    try:
        x, info = plan.solve(b, tol=1e-10)
        assert plan.stats()["batch_kernel"] in (1, 3)  # the CUDA cores, by whichever grid is faster
    finally:
        full.release()
    y, again = plan.solve(b, tol=1e-10)
    assert plan.stats()["batch_kernel"] == 2
    assert info["relres"] <= 1e-10 and again["relres"] <= 1e-10


def test_a_call_that_ran_out_of_memory_leaves_the_next_one_alone():
    from paper_0910_0663_gb300 import vtm
    w = wl.grid2d(1024, 1024, 64, 64, ground=0.1, seed=1)
    arrays = [torch.from_numpy(a).cuda() for a in (w.indptr, w.indices, w.data, w.partition)]
    small = wl.grid2d(24, 24, 8, 8, ground=0.1, seed=2)
    torch.cuda.synchronize()
    full = _Full(64 << 20)
    try:
        with pytest.raises(vtm.VTMError, match="out of memory"):
            vtm.Plan(*arrays, w.nparts)
        plan = vtm.Plan(small.indptr, small.indices, small.data, small.partition, small.nparts)
    finally:
        full.release()
    x, info = plan.solve(torch.from_numpy(small.b[0]).cuda())
    assert info["relres"] <= 1e-10


def test_new_values_without_room_for_a_second_copy():
    from paper_0910_0663_gb300 import vtm
    w = wl.grid2d(1536, 1536, 32, 32, ground=0.1, seed=1)  # 94 MB of values
    new = torch.from_numpy(w.data * 1.5).cuda()
    bad = new.clone()
    bad[7] = float("nan")
    b = torch.from_numpy(w.b[0]).cuda()
    plan = vtm.Plan(w.indptr, w.indices, w.data, w.partition, w.nparts)
    x0, _ = plan.solve(b)
    full = _Full(90 << 20)
    try:
        with pytest.raises(vtm.VTMError, match="non-finite"):
            plan.set_values(bad)
        y, _ = plan.solve(b)  # still factored, the old values
        plan.set_values(new)
        plan.factor()
        x, _ = plan.solve(b)
    finally:
        full.release()
    assert torch.equal(x0, y)
    ref, _ = vtm.Plan(w.indptr, w.indices, w.data * 1.5, w.partition, w.nparts, sweep_kernel=12).solve(b)
    assert np.linalg.norm((x - ref).cpu().numpy()) <= 1e-7 * np.linalg.norm(ref.cpu().numpy())
