"""New values on the device: refused sets leave the plan as it was, accepted
ones give the same operators as a plan made from those values."""
import numpy as np
import pytest
import torch

from paper_0910_0663_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _plan(w, data, **kw):
    from paper_0910_0663_gb300 import vtm
    return vtm.Plan(w.indptr, w.indices, data, w.partition, w.nparts, Zc=w.Zc, **kw)


def _scaled(w, seed):
    """Values of the same pattern: every branch and ground times its own factor."""
    rng = np.random.default_rng(seed)
    return wl.assemble_nodal(w.n, w.edges, w.g * rng.uniform(0.5, 2.0, w.g.shape), w.ground * 1.5)[2]


@pytest.mark.parametrize("kind", ["alpha", "diag", "wob", "sca"])
@pytest.mark.parametrize("side", ["host", "default", "own"])
def test_new_values_equal_a_new_plan(kind, side):
    w = wl.grid2d(37, 45, 9, 11, seed=2, ground=0.1)
    data = _scaled(w, 3)
    stream = torch.cuda.Stream() if side == "own" else None
    plan = _plan(w, w.data, stream=stream, factor=False)
    plan.set_admittance(kind, alpha=0.7, radius=1)
    plan.set_values(data if side == "host" else torch.from_numpy(data).cuda() * 1.0)
    plan.factor()
    ref = _plan(w, data, factor=False)
    ref.set_admittance(kind, alpha=0.7, radius=1)
    assert np.array_equal(plan.admittance(), ref.admittance())
    for t in (0, w.nparts // 2, w.nparts - 1):
        assert np.array_equal(plan.reflection(t), ref.reflection(t))


def test_channel_form_follows_new_values():
    w = wl.vccs_grid(40, 36, 10, 12, seed=4)
    data = w.data * 1.25  # every entry of every row: lines and couplings stay
    plan = _plan(w, w.data)
    plan.set_values(data)
    plan.factor()
    b = torch.from_numpy(w.b[0]).cuda()
    x, info = plan.solve(b)
    y, ref = _plan(w, data).solve(b)
    assert info["sweeps"] == ref["sweeps"] and torch.equal(x, y)


def test_refused_values_leave_the_plan_alone():
    from paper_0910_0663_gb300 import vtm
    w = wl.grid2d(24, 24, 8, 8, seed=5, ground=0.1)
    plan = _plan(w, w.data)
    b = torch.from_numpy(w.b[0]).cuda()
    x0, _ = plan.solve(b)
    rows = np.repeat(np.arange(w.n), np.diff(w.indptr))
    part = w.partition
    inner = np.flatnonzero((rows < w.indices) & (part[rows] == part[w.indices]))[3]
    cut = np.flatnonzero((rows < w.indices) & (part[rows] != part[w.indices]))[5]
    back = int(np.flatnonzero((rows == w.indices[cut]) & (w.indices == rows[cut]))[0])
    for change, why in [({inner: np.nan}, "non-finite"), ({inner: np.inf}, "non-finite"),
                        ({inner: w.data[inner] * 2}, "symmetric"), ({cut: 0.0, back: 0.0}, "torn lines")]:
        bad = w.data.copy()
        for q, v in change.items():
            bad[q] = v
        with pytest.raises(vtm.VTMError, match=why):
            plan.set_values(bad)
        x, _ = plan.solve(b)  # still factored, same values
        assert torch.equal(x, x0)
