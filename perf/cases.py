"""What the solver is measured on: calls that a circuit simulator makes through
``paper_0910_0663_gb300.vtm``, over the sizes, precisions and options in use.

Every case builds its circuit on the GPU from the seed alone (the recipes of
``paper_0910_0663_gb300.workloads``, drawn with torch), plans and factors it in
``prepare`` as a program does once per circuit, and times the calls that the
program then repeats: a solve, a forward and adjoint pair, a time march, a
gradient step on new conductances, a new corner of the same circuit.  ``exact``
solves the same systems in FP64 by preconditioned Krylov iterations and
refinement, without this repository's code.
"""
import math

import numpy as np
import torch

from paper_0910_0663_gb300 import vtm, workloads

DEV = "cuda"


def listed():
    return [
        # the 32 x 32 worked circuit in the default precision: the smallest call, thousands of tiny sweeps
        dict(name="grid32_fp64", kind="grid", ny=32, nx=32, th=8, tw=8, precision="fp64", nrhs=1, tol=1e-10),
        # the headline: a 2048^2 power grid, 4096 sub-circuits, FP16 sweeps on the caller's own stream
        dict(name="power2048_fp16", kind="power", ny=2048, nx=2048, th=32, tw=32, precision="fp16", nrhs=1,
             tol=1e-10, zc=1.0, own_stream=True),
        # a power grid of odd size with ragged tiles in the default precision (plain FP64 sweeps)
        dict(name="power1000x1500_fp64", kind="power", ny=1000, nx=1500, th=32, tw=32, precision="fp64", nrhs=1,
             tol=1e-10, zc=1.0),
        # a middle-sized power grid in FP32, the right-hand side and the result in host memory
        dict(name="power777x1291_fp32_host", kind="power", ny=777, nx=1291, th=28, tw=30, precision="fp32", nrhs=1,
             tol=1e-10, zc=1.0, host=True, own_stream=True),
        # few large sub-circuits (64 x 64 nodes, up to 256 ports) in the default precision
        dict(name="grid512_tiles64_fp64", kind="grid", ny=512, nx=512, th=64, tw=64, precision="fp64", nrhs=1, tol=1e-10),
        # the RC thermal grid, 400 uneven boxes, 64 current vectors at once, BF16 sweeps
        dict(name="thermal_64rhs_bf16", kind="thermal", nz=32, ny=128, nx=128, boxes=400, precision="bf16", nrhs=64,
             tol=1e-10),
        # a smaller thermal grid with an uneven count of right-hand sides in the default precision
        dict(name="thermal_18rhs_fp64", kind="thermal", nz=32, ny=64, nx=72, boxes=110, precision="fp64", nrhs=18,
             tol=1e-10),
        # backward-Euler transient of a thermal grid, every step warm-started from the one before
        dict(name="march_8steps_fp32", kind="march", nz=24, ny=96, nx=80, boxes=150, precision="fp32", nrhs=8, tol=1e-10),
        # an amplifier-like unsymmetric circuit: forward and adjoint solves (a sensitivity pair), admittances of Sec. VIII
        dict(name="vccs640_pair_fp64", kind="vccs", ny=640, nx=640, th=64, tw=64, precision="fp64", nrhs=1, tol=1e-10,
             admittance="sca"),
        # one step of a conductance optimisation: new values, factorisation, forward and adjoint solve, gradients
        dict(name="gradient1024_fp32", kind="gradient", ny=1024, nx=1024, th=64, tw=64, precision="fp32", nrhs=1, tol=1e-11),
        # another process corner of a power grid: new values, factorisation, one solve
        dict(name="corner512_fp16", kind="corner", ny=512, nx=512, th=32, tw=32, precision="fp16", nrhs=1, tol=1e-10, zc=1.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: a kind of work, then sizes, tiles and options of its range."""
    kind = rng.choice(["grid", "power", "power", "thermal", "thermal", "march", "vccs", "gradient", "corner"])
    c = dict(kind=kind, nrhs=1, tol=1e-10)
    if kind == "grid":
        tile = _log_int(rng, 6, 64)
        # no more than 16 tiles a side: a grid of many small tiles takes tens of thousands of sweeps
        c.update(ny=tile * rng.randint(2, 14) + rng.randint(0, 5), nx=tile * rng.randint(2, 14) + rng.randint(0, 5),
                 th=tile, tw=tile, precision=rng.choice(["fp64", "fp64", "fp32"]))
        c.update(ny=min(c["ny"], 700), nx=min(c["nx"], 700))
    elif kind == "power":
        tile = rng.choice([16, 24, 31, 32, 32, 40])
        c.update(ny=_log_int(rng, 100, 1400), nx=_log_int(rng, 100, 1400), th=tile, tw=tile,
                 precision=rng.choice(["fp64", "fp32", "bf16", "fp16"]), zc=rng.choice([0.5, 1.0, 1.0, 4.0]),
                 own_stream=rng.random() < 0.5, host=rng.random() < 0.2)
    elif kind in ("thermal", "march"):
        nz, ny, nx = rng.randint(8, 32), _log_int(rng, 24, 80), _log_int(rng, 24, 80)
        precision = rng.choice(["fp64", "fp32", "bf16", "fp16"] if kind == "thermal" else ["fp64", "fp32"])
        c.update(nz=nz, ny=ny, nx=nx, boxes=max(8, nz * ny * nx // rng.randint(900, 1500)), precision=precision)
        c["nrhs"] = rng.randint(3, 10) if kind == "march" else _log_int(rng, 2, 12 if precision == "fp64" else 64)
    elif kind == "vccs":
        tile = rng.choice([24, 32, 48, 64])
        c.update(ny=_log_int(rng, 128, 640), nx=_log_int(rng, 128, 640), th=tile, tw=tile, precision="fp64",
                 admittance=rng.choice(["sca", "wob"]))
    elif kind == "gradient":
        tile = rng.choice([32, 48, 64])
        c.update(ny=_log_int(rng, 128, 900), nx=_log_int(rng, 128, 900), th=tile, tw=tile, precision="fp32", tol=1e-11)
    else:
        tile = rng.choice([24, 32, 32, 48])
        c.update(ny=_log_int(rng, 128, 700), nx=_log_int(rng, 128, 700), th=tile, tw=tile,
                 precision=rng.choice(["fp64", "fp32", "bf16", "fp16"]), zc=1.0)
    return c


# ---- circuits ---------------------------------------------------------------

def _stencil(dims, conds, ground):
    """Columns and values (n x (2d + 1), columns ascending, -1 where there is
    no neighbour) of the nodal matrix of a grid: conds[a] holds the branches
    along axis a, ground one value per node."""
    n = math.prod(dims)
    idx = torch.arange(n, device=DEV).reshape(dims)
    d = len(dims)
    cols = torch.full((2 * d + 1, n), -1, dtype=torch.int64, device=DEV)
    vals = torch.zeros((2 * d + 1, n), dtype=torch.float64, device=DEV)
    diag = ground.reshape(dims).clone()
    for a in range(d):
        g, m = conds[a], dims[a]
        lo, hi = (idx.narrow(a, 0, m - 1).reshape(-1), idx.narrow(a, 1, m - 1).reshape(-1))
        cols[a, hi], vals[a, hi] = lo, -g.reshape(-1)
        cols[2 * d - a, lo], vals[2 * d - a, lo] = hi, -g.reshape(-1)
        diag.narrow(a, 0, m - 1).add_(g)
        diag.narrow(a, 1, m - 1).add_(g)
    cols[d], vals[d] = idx.reshape(-1), diag.reshape(-1)
    return cols.t().contiguous(), vals.t().contiguous()


def _csr(cols, vals):
    ok = cols >= 0
    ptr = torch.zeros(cols.shape[0] + 1, dtype=torch.int64, device=DEV)
    ptr[1:] = ok.sum(1).cumsum(0)
    return ptr, cols[ok].to(torch.int32), vals[ok]


def _uniform(gen, lo, hi, *shape):
    return torch.rand(*shape, generator=gen, dtype=torch.float64, device=DEV) * (hi - lo) + lo


def _tiles(ny, nx, th, tw):
    r = torch.arange(ny, device=DEV)[:, None] // th
    c = torch.arange(nx, device=DEV)[None, :] // tw
    return (r * -(-nx // tw) + c).reshape(-1).to(torch.int32), -(-ny // th) * -(-nx // tw)


def _add_sources(gen, cols, vals, ny, nx):
    """Controlled sources at 5% of the rows: a target 1 to 3 branches away,
    a gain of +-0.3 of the row's diagonal, whose size is added to the diagonal."""
    n = ny * nx
    rows = torch.randperm(n, generator=gen, device=DEV)[: n // 20]
    hops = torch.tensor([(a, b) for a in range(-3, 4) for b in range(-3, 4) if 1 <= abs(a) + abs(b) <= 3], device=DEV)
    hop = hops[torch.randint(len(hops), (len(rows),), generator=gen, device=DEV)]
    r, c = rows // nx, rows % nx
    dr = torch.where((r + hop[:, 0] < 0) | (r + hop[:, 0] >= ny), -hop[:, 0], hop[:, 0])
    dc = torch.where((c + hop[:, 1] < 0) | (c + hop[:, 1] >= nx), -hop[:, 1], hop[:, 1])
    target = (r + dr) * nx + c + dc
    gain = _uniform(gen, -0.3, 0.3, len(rows)) * vals[rows, 2]
    vals[rows, 2] += gain.abs()
    cols = torch.cat([cols, torch.full((n, 1), -1, dtype=torch.int64, device=DEV)], 1)
    vals = torch.cat([vals, torch.zeros((n, 1), dtype=torch.float64, device=DEV)], 1)
    same = cols[rows] == target[:, None]  # a neighbour's entry takes the gain; else it is one more entry
    vals[rows] += same * gain[:, None]
    new = ~same.any(1)
    cols[rows[new], 5], vals[rows[new], 5] = target[new], gain[new]
    key, order = torch.where(cols < 0, n, cols).sort(1)
    return torch.where(key == n, -1, key), vals.gather(1, order)


def _circuit(case, seed):
    """The circuit and the right-hand sides of a case, all on the GPU."""
    gen = torch.Generator(DEV).manual_seed(seed * 2 + 1)
    kind = case["kind"]
    w = {}
    if kind in ("thermal", "march"):
        dims = (case["nz"], case["ny"], case["nx"])
        boxes = workloads.random_boxes(np.random.default_rng(seed), dims, case["boxes"])
        part = np.empty(dims, np.int32)
        for k, b in enumerate(boxes):
            part[b[0]:b[1], b[2]:b[3], b[4]:b[5]] = k
        w["part"], w["nparts"] = torch.from_numpy(part.reshape(-1)).to(DEV), len(boxes)
    else:
        dims = (case["ny"], case["nx"])
        w["part"], w["nparts"] = _tiles(*dims, case["th"], case["tw"])
    n = w["n"] = math.prod(dims)
    shapes = [tuple(m - (a == b) for b, m in enumerate(dims)) for a in range(len(dims))]
    if kind in ("power", "corner"):
        conds = [10.0 ** _uniform(gen, -1.0, 1.0, *s) for s in shapes]
        pads = torch.randperm(n, generator=gen, device=DEV)[: round(0.01 * n)]
        ground = torch.zeros(n, dtype=torch.float64, device=DEV)
        ground[pads] = 10.0
        w["b"] = -_uniform(gen, 0.0, 1e-3, n)
        w["b"][pads] = 0.0
        if kind == "corner":  # the branches of another corner: 10% off, each by itself
            corner = [g * _uniform(gen, 0.9, 1.1, *g.shape) for g in conds]
            w["corner"] = _csr(*_stencil(dims, corner, ground))
    else:
        conds = [_uniform(gen, 0.5, 2.0, *s) for s in shapes]
        if kind in ("thermal", "march"):
            ground = _uniform(gen, 1.0, 10.0, n)  # C / h
        else:
            ground = torch.full((n,), 1e-3, dtype=torch.float64, device=DEV)
        w["b"] = _uniform(gen, -1.0, 1.0, *([n] if kind != "thermal" and kind != "march" else [case["nrhs"], n]))
    cols, vals = _stencil(dims, conds, ground)
    if kind == "vccs":
        cols, vals = _add_sources(gen, cols, vals, *dims)
        w["b2"] = _uniform(gen, -1.0, 1.0, n)
    if kind == "gradient":
        idx = torch.arange(n, device=DEV).reshape(dims)
        w["edges"] = torch.cat([torch.stack([idx.narrow(a, 0, dims[a] - 1).reshape(-1),
                                             idx.narrow(a, 1, dims[a] - 1).reshape(-1)], 1) for a in (1, 0)])
        w["g"] = torch.cat([conds[1].reshape(-1), conds[0].reshape(-1)])
        step = [g * _uniform(gen, 0.95, 1.05, *g.shape) for g in conds]  # where the optimiser's step leads
        w["g_next"] = torch.cat([step[1].reshape(-1), step[0].reshape(-1)])
        w["next"] = _csr(*_stencil(dims, step, ground))
    w["ground"] = ground
    w["csr"] = _csr(cols, vals)
    return w


# ---- the calls --------------------------------------------------------------

def prepare(case, seed):
    w = _circuit(case, seed)
    kind = case["kind"]
    stream = torch.cuda.Stream() if case.get("own_stream") else None
    torch.cuda.synchronize()  # the plan reads the arrays on its own stream
    s = {"case": dict(case), "b": w["b"], "w": w}
    if kind == "gradient":
        s["net"] = vtm.Network(w["n"], w["edges"].cpu().numpy(), w["csr"][0], w["csr"][1], w["part"], w["nparts"],
                               precision=case["precision"], g0=w["g"], ground0=w["ground"])
        s["g"] = w["g"].clone().requires_grad_()
        s["ground"] = w["ground"].clone().requires_grad_()
        s["b"] = w["b"].clone().requires_grad_()
        return s
    admittance = case.get("admittance")
    s["plan"] = vtm.Plan(*w["csr"], w["part"], w["nparts"], Zc=case.get("zc", 1.0), precision=case["precision"],
                         stream=stream, factor=admittance is None)
    if admittance:
        s["plan"].set_admittance(admittance, alpha=0.5, radius=1)
    if case.get("host"):
        s["b"] = w["b"].cpu().pin_memory()
    return s


def run(s):
    case, kind, tol = s["case"], s["case"]["kind"], s["case"]["tol"]
    if kind == "gradient":
        with torch.no_grad():
            s["g"].copy_(s["w"]["g_next"])  # the optimiser's update, in place
        x = s["net"].solve(s["g"], s["ground"], s["b"], tol=tol)
        grads = torch.autograd.grad((x * x).sum(), [s["g"], s["ground"], s["b"]])
        return [x.detach(), *grads]
    plan = s["plan"]
    if kind == "march":
        return plan.march(s["w"]["ground"], s["b"], tol=tol)[0]
    if kind == "corner":
        plan.set_values(s["w"]["corner"][2])
        plan.factor()
    x = plan.solve(s["b"], tol=tol)[0]
    if kind == "vccs":
        return [x, plan.adjoint(s["w"]["b2"], tol=tol)[0]]
    return x


# ---- what a pass cannot do without ------------------------------------------

def work(case):
    """Every array that the call is given read once (the matrix in CSR, new
    values where the call brings them, right-hand sides) and its results
    written once; the operations of the residual that confirms each result."""
    kind, r = case["kind"], case["nrhs"]
    n = case["ny"] * case["nx"] * case.get("nz", 1)
    per_row = 7 if kind in ("thermal", "march") else 5
    solves = 2 if kind in ("vccs", "gradient") else 1
    byte = n * (12 * per_row + 8) + 16 * n * r * solves
    if kind == "gradient":
        byte += 8 * 2 * (2 * n) + 8 * 2 * n  # conductances and their gradients; ground and its gradient
    return {"bytes": byte, "flops": 2 * per_row * n * r * solves}


# ---- the same results in 64 bits --------------------------------------------

def _krylov(A, b, dinv, symmetric):
    """Jacobi-preconditioned CG (BiCGStab for an unsymmetric A) on the columns
    of b, to about 1e-9 of each."""
    tiny = 1e-300
    x, r = torch.zeros_like(b), b.clone()
    stop = 1e-9 * b.norm(dim=0)
    dot = lambda u, v: (u * v).sum(0)  # noqa: E731
    if symmetric:
        z = dinv * r
        p, rz = z.clone(), dot(r, z)
        for k in range(20000):
            q = A @ p
            a = rz / (dot(p, q) + tiny)
            x += a * p
            r -= a * q
            if k % 16 == 15 and bool((r.norm(dim=0) <= stop).all()):
                break
            z = dinv * r
            rz, old = dot(r, z), rz
            p = z + rz / (old + tiny) * p
        return x
    r0, p, rho = r.clone(), r.clone(), dot(r, r)
    for k in range(20000):
        y = dinv * p
        v = A @ y
        a = rho / dot(r0, v)
        s = r - a * v
        z = dinv * s
        t = A @ z
        om = dot(t, s) / (dot(t, t) + tiny)
        x += a * y + om * z
        r = s - om * t
        if k % 16 == 15 and bool((r.norm(dim=0) <= stop).all()):
            break
        rho, old = dot(r0, r), rho
        p = r + rho / old * (a / om) * (p - om * v)
    return x


def _solve64(csr, b, symmetric=True, transpose=False):
    """A x = b (rows of b) in FP64: Krylov solves inside refinement."""
    n = csr[0].numel() - 1
    A = torch.sparse_csr_tensor(csr[0], csr[1].to(torch.int64), csr[2], (n, n))
    row = torch.repeat_interleave(torch.arange(n, device=DEV), csr[0][1:] - csr[0][:-1])
    on = row == csr[1]
    dinv = (1.0 / csr[2][on])[:, None]
    if transpose:
        A = torch.sparse_coo_tensor(torch.stack([csr[1].to(torch.int64), row]), csr[2], (n, n)).coalesce().to_sparse_csr()
    rhs = b.reshape(-1, n).t().contiguous()
    x = torch.zeros_like(rhs)
    for _ in range(4):
        x += _krylov(A, rhs - A @ x, dinv, symmetric)
    return x.t().reshape(b.shape).contiguous()


def exact(case, seed):
    kind = case["kind"]
    w = _circuit(case, seed)
    if kind == "march":
        out, x = [], torch.zeros(w["n"], dtype=torch.float64, device=DEV)
        for p in w["b"]:
            x = _solve64(w["csr"], p + w["ground"] * x)
            out.append(x)
        return torch.stack(out)
    if kind == "vccs":
        return [_solve64(w["csr"], w["b"], symmetric=False), _solve64(w["csr"], w["b2"], symmetric=False, transpose=True)]
    if kind == "corner":
        return _solve64(w["corner"], w["b"])
    if kind == "gradient":
        x = _solve64(w["next"], w["b"])
        lam = _solve64(w["next"], 2 * x)
        i, j = w["edges"][:, 0], w["edges"][:, 1]
        return [x, -(lam[i] - lam[j]) * (x[i] - x[j]), -lam * x, lam]
    return _solve64(w["csr"], w["b"])
