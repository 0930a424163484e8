"""Sweeps of an inner solve in one launch (the resident form the autotuner picks
for plans of few sub-circuits; it reports as kernel 8): one SM and a grid barrier.

Bars as for the other sweep kernels: FP64 histories within 1e-8 of the oracle's
(1e-13 absolute), low precision within the rounding of the stored T_P, iterates
after k sweeps within 1e-12.  A residual term is a difference of FP32 waves in the
low precisions: six roundings (u = 2^-24) of at most (1 + g/W) 4 |w|, g/W <= 2, and
|w| <= (W + 2 g) |x| 2 <= 10 |x|, so a history entry carries up to
720 u |x|_max sqrt(ports) / |b| on top."""
import numpy as np
import pytest
import torch

from oracle import vtm_oracle as O
from paper_0910_0663_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

# (grid, tile): one SM -- 2 tiles, 16 tiles of 32 ports, 7 tiles of 33..64 ports;
# grid barrier -- 9 and 25 ragged tiles, 6 tiles of up to 256 ports (streamed
# blocks), 400 tiles (several per SM)
ONE = [((1, 6), (1, 3)), ((32, 32), (8, 8)), ((17, 119), (17, 17))]
GRID = [((50, 50), (17, 19)), ((90, 90), (18, 18)), ((128, 192), (64, 64)), ((240, 240), (12, 12))]


def _plan(shape, precision, **kw):
    from paper_0910_0663_gb300 import vtm
    (ny, nx), (th, tw) = shape
    w = wl.grid2d(ny, nx, th, tw, ground=0.05, seed=7)
    return w, vtm.Plan(w.indptr, w.indices, w.data, w.partition, w.nparts, precision=precision, **kw)


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16", "bf16"])
@pytest.mark.parametrize("shape", ONE + GRID)
def test_histories_follow_the_oracle(shape, precision):
    w, plan = _plan(shape, precision)
    A = w.csr()
    b = torch.from_numpy(w.b[0]).cuda()
    plan.set_options(history_len=40)
    x, _ = plan.solve(b, tol=1e-10)
    h = plan.history
    x2, _ = plan.solve(b, tol=1e-10)
    assert torch.equal(x, x2) and np.array_equal(h, plan.history)  # fixed order of every sum
    assert O.residual_norms(A, x.cpu().numpy()[None], w.b[:1]).max() <= 1e-10
    if precision == "fp64":  # only the resident form reports 8 on an FP64 plan
        assert plan.stats()["sweep_kernel"] == 8
    ref = O.vtm_midpoint(A, w.partition, w.nparts, w.b[:1], W=1 / w.Zc, tol=0, max_sweeps=40)
    href = ref.history[:, 0]
    rtol, floor, kmax = {"fp64": (1e-8, 1e-9, 40), "fp32": (1e-3, 1e-4, 40), "fp16": (2e-2, 5e-3, 20),
                         "bf16": (5e-2, 2e-2, 15)}[precision]
    k = min(kmax, int(np.count_nonzero((h > 0) & (href[: len(h)] > floor))))
    assert k >= 1
    u32 = 720 * 2.0 ** -24 * float(x.abs().max()) * plan.stats()["nports"] ** 0.5 / np.linalg.norm(w.b[0])
    assert np.allclose(h[:k], href[:k], rtol=rtol, atol=1e-13 if precision == "fp64" else u32)


@pytest.mark.parametrize("shape", [ONE[1], GRID[1]])
@pytest.mark.parametrize("k", [1, 2, 3, 10])
def test_iterate_after_k_sweeps(shape, k):
    w, plan = _plan(shape, "fp64", max_sweeps=k)
    x, info = plan.solve(torch.from_numpy(w.b[0]).cuda(), tol=1e-300, check=False)
    assert info["sweeps"] == k and plan.stats()["sweep_kernel"] == 8
    _, its = O.vtm_midpoint(w.csr(), w.partition, w.nparts, w.b[:1], W=1 / w.Zc, tol=0, max_sweeps=k,
                            keep_iterates=True)
    ref = its[k - 1][0]
    assert np.abs(x.cpu().numpy() - ref).max() <= 1e-12 * np.abs(ref).max()


def test_a_barrier_that_runs_out_is_reported_and_the_plan_recovers():
    from paper_0910_0663_gb300 import vtm
    w, plan = _plan(GRID[1], "fp64")
    b = torch.from_numpy(w.b[0]).cuda()
    x, _ = plan.solve(b)
    plan.set_options(wait_polls=1)  # the first poll that finds the barrier open gives up
    with pytest.raises(vtm.VTMError, match="timed out"):
        plan.solve(b)
    plan.set_options(wait_polls=0)
    x2, _ = plan.solve(b)
    assert torch.equal(x, x2)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_one_sm_with_several_warps_per_tile_ends_every_warp_at_one_sweep(precision):
    """Tiles of 33..64 ports take two warps each, which meet at a barrier of their own
    in every sweep; the runs end by tolerance and by the sweep limit, at odd and even
    sweeps, with the same bits each time."""
    w, plan = _plan(ONE[2], precision)
    b = torch.from_numpy(w.b[0]).cuda()
    for limit in (1, 2, 3, 4, 17, 18, 200000):
        plan.set_options(max_sweeps=limit)
        x, info = plan.solve(b, check=False)
        assert info["sweeps"] == limit or info["relres"] <= 1e-10
        for _ in range(20):
            y, again = plan.solve(b, check=False)
            assert torch.equal(x, y) and again["sweeps"] == info["sweeps"]


@pytest.mark.parametrize("forced", [9, 11])
def test_captured_sweeps_do_not_outlive_their_buffers(forced):
    """A plan with a stream of its own captures its sweeps; a later solve that may take
    the resident form must leave the captured launches a buffer that still exists."""
    from paper_0910_0663_gb300 import vtm
    w = wl.grid2d(240, 240, 12, 12, ground=0.05, seed=7)
    A = w.csr()
    b = torch.from_numpy(w.b[0]).cuda()
    plan = vtm.Plan(w.indptr, w.indices, w.data, w.partition, w.nparts, precision="fp16", stream=torch.cuda.Stream(),
                    sweep_kernel=forced)
    x, _ = plan.solve(b)
    for kernel in (0, forced, 0, 5, forced):
        plan.set_options(sweep_kernel=kernel)
        y, info = plan.solve(b)
        assert O.residual_norms(A, y.cpu().numpy()[None], w.b[:1]).max() <= 1e-10
        if kernel == forced:
            assert torch.equal(x, y)


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16"])
def test_the_choice_follows_what_a_later_solve_allows(precision):
    """The kernel chosen by an earlier solve may not serve a later one: a sweep limit
    that the grid barrier cannot count to, or an FP64 plan that went to FP32 and back
    (its hi + lo copy is gone)."""
    from paper_0910_0663_gb300 import vtm
    w, plan = _plan(GRID[1], precision)
    A = w.csr()
    b = torch.from_numpy(w.b[0]).cuda()

    def solves(**opts):
        plan.set_options(**opts)
        x, info = plan.solve(b)
        assert O.residual_norms(A, x.cpu().numpy()[None], w.b[:1]).max() <= 1e-10
        return x

    x = solves()
    solves(max_sweeps=1 << 30)
    solves(max_sweeps=200000)
    if precision == "fp64":
        plan.set_options(precision="fp32")
        with pytest.raises(vtm.VTMError):
            plan.solve(b)  # not factored for FP32
        plan.factor()
        solves()
        solves(precision="fp64")
        plan.factor()
        solves()


# 9 tiles of up to 128 ports (in one launch, FP64 or double-float by speed) and 6 of up to
# 256 (FP64)
FP64 = [((66, 65), (32, 32)), GRID[2]]


@pytest.mark.parametrize("shape", ONE + GRID + FP64)
def test_fp64_histories_at_the_other_kernels_bar(shape):
    w, plan = _plan(shape, "fp64")
    plan.set_options(history_len=40, max_sweeps=40)
    plan.solve(torch.from_numpy(w.b[0]).cuda(), tol=1e-300, check=False)
    assert plan.stats()["sweep_kernel"] == 8
    ref = O.vtm_midpoint(w.csr(), w.partition, w.nparts, w.b[:1], W=1 / w.Zc, tol=0, max_sweeps=40)
    h, href = plan.history, ref.history[:, 0]
    k = int(np.count_nonzero((h > 0) & (href[: len(h)] > 1e-9)))
    assert k >= 1 and np.allclose(h[:k], href[:k], rtol=1e-9, atol=1e-13)


def test_tiles_above_128_ports_sweep_in_fp64():
    """53 bits and FP64's range: a residual of 1e-14 is reached (double-float ends near
    1e-13), and a power of two on b changes no bit."""
    w, plan = _plan(GRID[2], "fp64", max_sweeps=20000)
    b = torch.from_numpy(w.b[0]).cuda()
    x, info = plan.solve(b, tol=1e-14)
    assert info["relres"] <= 1e-14 and plan.stats()["sweep_kernel"] == 8
    for e in (-400, 400):
        y, scaled = plan.solve(b * 2.0 ** e, tol=1e-14)
        assert scaled["sweeps"] == info["sweeps"] and torch.equal(y, x * 2.0 ** e)


@pytest.mark.parametrize("kind", ["alpha", "wob"])
def test_fp64_in_one_launch_equals_kernel_1_on_odd_and_lone_tiles(kind):
    """Odd port counts (a last pair of outputs half empty), ranges of pairs over several
    tiles, a tile without ports, power waves: the same sums in another order, so
    histories agree like those of any two FP64 kernels (1e-9, 1e-13 absolute)."""
    from paper_0910_0663_gb300 import vtm
    w = wl.grid2d(129, 259, 43, 65, ground=0.3, seed=11)
    rows = np.repeat(np.arange(w.n), np.diff(w.indptr))
    lone = (w.partition[rows] == 5) != (w.partition[w.indices] == 5)
    data = np.where(lone, 0.0, w.data)  # its branches stay on the diagonals: conductances to ground
    b = torch.from_numpy(w.b[0]).cuda()
    out = []
    for kernel in (0, 1):
        plan = vtm.Plan(w.indptr, w.indices, data, w.partition, w.nparts, sweep_kernel=kernel, factor=False)
        plan.set_admittance(kind, alpha=0.8)
        plan.factor()
        st = plan.stats()
        assert 128 < st["max_ports"] <= 256
        plan.set_options(sweep_kernel=kernel, history_len=30)
        x, info = plan.solve(b, tol=1e-12)
        assert kernel or plan.stats()["sweep_kernel"] == 8
        out.append((x, info["sweeps"], plan.history))
    h0, h1 = out[0][2], out[1][2]
    k = int(np.count_nonzero((h0 > 1e-9) & (h1 > 1e-9)))
    assert abs(out[0][1] - out[1][1]) <= 1 and k >= 10
    assert np.allclose(h0[:k], h1[:k], rtol=1e-9, atol=1e-13)
