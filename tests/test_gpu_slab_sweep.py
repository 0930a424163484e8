"""Kernel 1 (slabs of 32, 64 or 128 outputs per work item) against the oracle.

The bars are those of the other sweep kernels: FP64 residual histories within
1e-9 of the oracle's (1e-13 absolute: the residual is a difference of waves), low precision within the rounding of the stored T_P."""
import numpy as np
import pytest
import torch

from oracle import vtm_oracle as O
from paper_0910_0663_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

# uneven boxes with ragged port counts (32-wide slabs), slabs wider than the
# tiles (1024 tiles of up to 32 ports: 128-wide), ragged second slabs (361 tiles
# of up to 72 ports: 64-wide)
PLANS = {"boxes": lambda: wl.thermal3d(8, 24, 24, 12, nrhs=1, seed=3, min_box=100, max_box=1200),
         "wide": lambda: wl.grid2d(256, 256, 8, 8, seed=4, ground=0.1),
         "ragged": lambda: wl.grid2d(342, 342, 18, 18, seed=5, ground=0.1),
         "pair": lambda: wl.grid2d(1, 9, 1, 5, seed=6, ground=0.1)}


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16", "bf16"])
@pytest.mark.parametrize("name", sorted(PLANS))
def test_slab_sweeps_follow_the_oracle(name, precision):
    from paper_0910_0663_gb300 import vtm
    w = PLANS[name]()
    A = w.csr()
    plan = vtm.Plan(w.indptr, w.indices, w.data, w.partition, w.nparts, Zc=w.Zc, precision=precision, sweep_kernel=1)
    plan.set_options(history_len=30)
    x, info = plan.solve(torch.from_numpy(w.b[0]).cuda(), tol=1e-10)
    assert O.residual_norms(A, x.cpu().numpy()[None], w.b[:1]).max() <= 1e-10
    ref = O.vtm_midpoint(A, w.partition, w.nparts, w.b[:1], W=1 / w.Zc, tol=0, max_sweeps=30)
    h, href = plan.history, ref.history[:, 0]
    rtol, floor, kmax = {"fp64": (1e-9, 1e-9, 30), "fp32": (1e-3, 1e-4, 30), "fp16": (2e-2, 5e-3, 20),
                         "bf16": (5e-2, 2e-2, 15)}[precision]
    k = min(kmax, int(np.count_nonzero((h > 0) & (href[: len(h)] > floor))))
    assert k >= 1
    assert np.allclose(h[:k], href[:k], rtol=rtol, atol=1e-13 if precision == "fp64" else 0)


@pytest.mark.parametrize("precision", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("scale", [2.0 ** -60, 2.0 ** -45, 2.0 ** 70])
def test_right_hand_sides_of_any_size(precision, scale):
    """A power of two on b changes no bit of the sweeps or of their residuals while the
    waves stay in FP32's range (entries of b from 1e-18 to 1e21 here; squared residuals leave it)."""
    from paper_0910_0663_gb300 import vtm
    w = PLANS["boxes"]()
    plan = vtm.Plan(w.indptr, w.indices, w.data, w.partition, w.nparts, Zc=w.Zc, precision=precision, sweep_kernel=1)
    b = torch.from_numpy(w.b[0]).cuda()
    x, info = plan.solve(b, tol=1e-8)
    y, scaled = plan.solve(b * scale, tol=1e-8)
    assert scaled["sweeps"] == info["sweeps"] and scaled["outer_steps"] == info["outer_steps"]
    assert torch.equal(y, x * scale)
