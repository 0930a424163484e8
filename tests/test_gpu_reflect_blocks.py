"""Reflection matrices built 32 ports at a time, against sparse LU.

T_P(s, q) = 2 W beta_s beta_q [K_P^-1](l_s, l_q) + [s = q](W - 2 g)/(W + 2 g); with
a ground of 1 S on every node cond(K_P) <= 17, so entries (at most 1 in size) agree
within 17 * 64 u ~ 1.2e-13."""
import numpy as np
import pytest
import scipy.sparse.linalg as sla

from paper_0910_0663_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _reference(w, plan, t):
    node, remote, part, _ = plan.ports()
    sel = np.flatnonzero(part == t)
    A = w.csr()
    nodes = np.flatnonzero(w.partition == t)
    pos = {v: i for i, v in enumerate(nodes)}
    K = A[nodes][:, nodes].tolil()
    W = plan.admittance()[sel]
    g = np.array([-A[node[s], remote[s]] for s in sel])
    loc = np.array([pos[node[s]] for s in sel])
    for a, v in zip(loc, g - 4 * g * g / (2 * g + W)):
        K[a, a] += v
    beta = 2 * g / (2 * g + W)
    E = np.zeros((len(nodes), len(sel)))
    E[loc, np.arange(len(sel))] = 1.0
    G = sla.splu(K.tocsc()).solve(E)[loc]
    return 2 * (W * beta)[:, None] * G * beta[None, :] + np.diag((W - 2 * g) / (W + 2 * g))


@pytest.mark.parametrize("kind", ["alpha", "wob"])
@pytest.mark.parametrize("ny,nx,th,tw", [(1, 9, 1, 3), (6, 6, 2, 3), (24, 24, 8, 8), (33, 66, 31, 33), (64, 64, 32, 32),
                                         (70, 68, 33, 35), (96, 128, 48, 64), (65, 133, 65, 66), (130, 260, 129, 130),
                                         (150, 306, 150, 153)])
def test_reflections_equal_sparse_lu(ny, nx, th, tw, kind):
    from paper_0910_0663_gb300 import vtm
    w = wl.grid2d(ny, nx, th, tw, ground=1.0, seed=ny)
    plan = vtm.Plan(w.indptr, w.indices, w.data, w.partition, w.nparts, Zc=0.7, factor=False)
    plan.set_admittance(kind, alpha=0.6 if kind == "wob" else 1.4)
    tiles = sorted({0, w.nparts // 2, w.nparts - 1}) if min(th, tw) < 100 else [0]
    for t in tiles:
        T = plan.reflection(t)
        assert np.abs(T - _reference(w, plan, t)).max() <= 1.2e-13
