"""What the speed of this library is measured on: its calls as a user's program makes them.

A case is a dict of plain values.  listed() gives the cases, draw() more of the
same ranges, prepare() what a program holds before the call, run() one pass
through the public entry points, work() the bytes and operations that the pass
cannot do without, exact() its outputs by plain torch in 64 bits.

The problems are the paper's: P1 diffusion on triangles and tetrahedra with a
strongly anisotropic tensor (a rotated constant one in 2D; the dispersion law
of a vortex velocity, alpha_L / alpha_T = 1e3, elsewhere), Dirichlet data,
bounds 0 <= c (<= 1), steady or backward Euler.  Steady and transient 3D solves
stop at kkt_rel 1e-12, the tolerance of the repository's oracle: there a
solution is known to about 1e-10 and can be compared; 2D solves, whose
attainable residual is higher and whose solutions are known better, stop at the
library's default.
"""
from __future__ import annotations

import math
import random
from types import SimpleNamespace

import numpy as np
import torch

import paper_1506_08435_gb300 as P

DEV = torch.device("cuda" if torch.cuda.is_available() else "cpu")
F64 = torch.float64

SOLVERS = {"gpcg": P.NN_SOLVER_GPCG, "lbfgs": P.NN_SOLVER_LBFGS, "tron": P.NN_SOLVER_TRON}
PRECISIONS = {"fp64": P.NN_PREC_FP64, "mixed": P.NN_PREC_MIXED, "auto": P.NN_PREC_AUTO}
FORMATS = {"sell": P.NN_FMT_SELL, "csr": P.NN_FMT_CSR}
RTOL_2D, RTOL_3D = 1e-10, 1e-12


# ------------------------------------------------------------------ the cases

def _steady2d(nx, ny, field, precision="fp64"):
    return dict(kind="solve", mesh="grid2d", nx=nx, ny=ny, nz=0, field=field, solver="gpcg", precision=precision,
                rtol=RTOL_2D)


def _steady3d(nx, ny, nz, precision):
    return dict(kind="solve", mesh="grid3d", nx=nx, ny=ny, nz=nz, field="rotated", solver="gpcg", precision=precision,
                rtol=RTOL_3D)


def _transient3d(nx, ny, nz, steps, solver, precision):
    return dict(kind="transient", mesh="grid3d", nx=nx, ny=ny, nz=nz, field="vortex", dt=0.01, steps=steps,
                solver=solver, precision=precision, rtol=RTOL_3D)


def _hole(m, tilt, solver, precision):
    return dict(kind="solve", mesh="hole", nx=9 * m, ny=9 * m, nz=9 * m, m=m, tilt=tilt, field="uniform",
                solver=solver, precision=precision, rtol=RTOL_3D)


def _batch(count, nmin, nmax, precision):
    return dict(kind="batch", mesh="grid2d", count=count, nmin=nmin, nmax=nmax, precision=precision, rtol=RTOL_2D)


def _assemble(mesh, nx, ny, nz, field, dt):
    return dict(kind="assemble", mesh=mesh, nx=nx, ny=ny, nz=nz, field=field, dt=dt)


def _spmv(nx, ny, nz, fmt):
    return dict(kind="spmv", mesh="grid3d", nx=nx, ny=ny, nz=nz, field="rotated", format=fmt)


def _serve(count, nodes2d, nodes3d):
    return dict(kind="serve", count=count, nodes2d=nodes2d, nodes3d=nodes3d, precision="auto", rtol=RTOL_2D)


def listed():
    return [
        # the smallest solve a user makes: the 2,601-node square (launches, barriers)
        dict(_steady2d(50, 50, "tensor"), name="steady2d_50x50"),
        # a 2D request near the upper end of the serving range, ragged sides, heterogeneous field
        dict(_steady2d(397, 283, "blocks2d"), name="steady2d_397x283"),
        # the transient benchmark's mesh: warm-started backward-Euler steps with their history
        dict(_transient3d(40, 40, 40, 8, "gpcg", "fp64"), name="transient3d_40"),
        # the same on a ragged mesh with the mixed-precision option
        dict(_transient3d(37, 29, 53, 6, "gpcg", "mixed"), name="transient3d_mixed_37x29x53"),
        # projected L-BFGS, the paper's quasi-Newton solver (BLMVM), on a small transient run
        dict(_transient3d(21, 25, 18, 4, "lbfgs", "fp64"), name="transient3d_lbfgs_21x25x18"),
        # a large steady solve in plain FP64 (the flagship steady problem, sized to a second)
        dict(_steady3d(96, 96, 96, "fp64"), name="steady3d_96"),
        # the largest: AUTO takes FP32 inner solves, the operator streams from HBM
        dict(_steady3d(112, 104, 120, "auto"), name="steady3d_auto_112x104x120"),
        # the paper's own test problem (cube with a hole, explicit mesh) with its solver TRON
        dict(_hole(5, 1.0, "tron", "fp64"), name="cube_hole_tron_m5"),
        # many independent 2D systems of uneven size in one call
        dict(_batch(40, 20, 120, "fp64"), name="batch2d_40"),
        # building a large system: pattern, elements, elimination, SELL and FP32 copies
        dict(_assemble("grid3d", 90, 101, 84, "rotated", 0.0), name="assemble3d_90x101x84"),
        # one matrix-vector product on a large system, the unit of the paper's cost model
        dict(_spmv(96, 88, 104, "sell"), name="spmv_sell_96x88x104"),
        # a burst of requests from host memory through the serving loop
        dict(_serve(8, 30000, 40000), name="serve_8"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _sides3d(rng, lo, hi):
    """Three uneven sides whose geometric mean is log-uniform in [lo, hi]."""
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    a, b = rng.uniform(0.8, 1.25), rng.uniform(0.8, 1.25)
    return max(3, round(n * a)), max(3, round(n * b)), max(3, round(n / (a * b)))


def draw(rng):
    kind = rng.choice(["steady2d", "transient", "lbfgs", "steady3d", "hole", "batch", "assemble", "spmv", "serve"])
    if kind == "steady2d":
        n = _log(rng, 40, 330)
        r = rng.uniform(0.75, 1.33)
        field = "tensor" if n < 100 and rng.random() < 0.5 else "blocks2d"
        return _steady2d(max(8, round(n * r)), max(8, round(n / r)), field)
    if kind == "transient":
        x, y, z = _sides3d(rng, 14, 40)
        return _transient3d(x, y, z, rng.randint(2, 8), "gpcg", rng.choice(["fp64", "fp64", "mixed"]))
    if kind == "lbfgs":
        x, y, z = _sides3d(rng, 10, 22)
        return _transient3d(x, y, z, rng.randint(2, 4), "lbfgs", "fp64")
    if kind == "steady3d":
        x, y, z = _sides3d(rng, 18, 92)
        return _steady3d(x, y, z, rng.choice(["fp64", "auto"]))
    if kind == "hole":
        return _hole(rng.randint(2, 5), round(rng.uniform(0.6, 1.4), 3), rng.choice(["tron", "gpcg"]), "fp64")
    if kind == "batch":
        lo = rng.randint(20, 40)
        return _batch(rng.randint(6, 40), lo, lo + rng.randint(10, 80), rng.choice(["fp64", "fp64", "mixed"]))
    if kind == "assemble":
        if rng.random() < 0.4:
            n = _log(rng, 50, 900)
            return _assemble("grid2d", n, max(8, round(n * rng.uniform(0.6, 1.1))), 0, "blocks2d", 0.0)
        x, y, z = _sides3d(rng, 16, 88)
        dt = rng.choice([0.0, 0.01])
        return _assemble("grid3d", x, y, z, "vortex" if dt else "rotated", dt)
    if kind == "spmv":
        x, y, z = _sides3d(rng, 20, 96)
        return _spmv(x, y, z, rng.choice(["sell", "csr"]))
    return _serve(rng.randint(3, 8), _log(rng, 4000, 30000), _log(rng, 12000, 40000))


# ------------------------------------------------------------------ problems

_PERMS = ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0))


def _host(t):
    return np.ascontiguousarray(t.cpu().numpy())


def _vortex(x, y, px, py):
    x, y = 2 * math.pi * (x + px), 2 * math.pi * (y + py)
    return torch.stack([torch.sin(x) * torch.cos(y), -torch.cos(x) * torch.sin(y), torch.full_like(x, 0.1)], -1)


def _cells(*sizes):
    """Lattice coordinates of the cells, the first index fastest."""
    return [g.reshape(-1) for g in reversed(torch.meshgrid(*[torch.arange(n, device=DEV) for n in reversed(sizes)],
                                                           indexing="ij"))]


def _rotations(g, count):
    q = torch.randn(count, 4, generator=g, device=DEV, dtype=F64)
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    rows = [1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
            2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
            2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]
    return torch.stack(rows, 1).reshape(count, 3, 3)


def _spec(mesh, nx, ny, nz, field, seed, dt=0.0, m=0, tilt=1.0):
    """The problem's data in host memory, with the fields that P.Problem reads."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    r = random.Random(seed)
    s = SimpleNamespace(dim=2 if mesh == "grid2d" else 3, nx=nx, ny=ny, nz=nz, lo=0.0, hi=1.0, dt=dt, f_elem=None,
                        coef_kind=P.NN_COEF_VELOCITY, aL=1.0, aT=1e-3, DM=1e-9, coords=None, conn=None)
    if mesh == "grid2d":
        i, j = _cells(nx, ny)
        # centroids of the two triangles of each square
        x = torch.stack([(3 * i + 2) / (3.0 * nx), (3 * i + 1) / (3.0 * nx)], 1).reshape(-1).double()
        y = torch.stack([(3 * j + 1) / (3.0 * ny), (3 * j + 2) / (3.0 * ny)], 1).reshape(-1).double()
        if field == "tensor":    # constant rotated tensor, c >= 0 only
            th, ratio = r.uniform(0.1, 3.0), 10.0 ** r.uniform(2.0, 3.0)
            a, b = math.cos(th), math.sin(th)
            d = [ratio * a * a + b * b, (ratio - 1.0) * a * b, ratio * b * b + a * a]
            s.coef_kind, s.hi, s.aL, s.aT, s.DM = P.NN_COEF_TENSOR, math.inf, 0.0, 0.0, 0.0
            s.coef = np.tile(np.array(d), (2 * nx * ny, 1))
        else:                    # vortex speed along a random direction per block of 10 x 10 squares
            nbx, nby = -(-nx // 10), -(-ny // 10)
            th = math.pi * torch.rand(nbx * nby, generator=g, device=DEV, dtype=F64)
            th = th[(i // 10 + nbx * (j // 10)).repeat_interleave(2)]
            speed = _vortex(x, y, r.random(), r.random()).norm(dim=1)
            s.coef = _host(torch.stack([speed * torch.cos(th), speed * torch.sin(th)], 1))
        x0, y0 = 0.6 * r.random(), 0.6 * r.random()
        x1, y1 = x0 + r.uniform(0.15, 0.35), y0 + r.uniform(0.15, 0.35)
        s.f_elem = _host(((x >= x0) & (x <= x1) & (y >= y0) & (y <= y1)).double())
        i, j = _cells(nx + 1, ny + 1)
        mask = (i == 0) | (i == nx) | (j == 0) | (j == ny)
        s.dmask, s.dval = _host(mask.to(torch.uint8)), np.zeros(len(mask))
        s.c0 = s.dval.copy()
        return s
    if mesh == "hole":           # the paper's cube with a cubic hole, hexahedron diagonals across the velocity
        i, j, k = _cells(nx, nx, nx)
        keep = ~((i >= 4 * m) & (i < 5 * m) & (j >= 4 * m) & (j < 5 * m) & (k >= 4 * m) & (k < 5 * m))
        base = torch.stack([i, j, k], 1)[keep]
        tets = []
        for p in _PERMS:
            v, at = base.clone(), [base]
            for a in p:
                v = v.clone()
                v[:, a] += 1
                at.append(v)
            tets.append(torch.stack([w[:, 0] + (nx + 1) * (w[:, 1] + (nx + 1) * w[:, 2]) for w in at], 1))
        used, conn = torch.unique(torch.stack(tets, 1).reshape(-1, 4), return_inverse=True)
        i, j, k = used % (nx + 1), used // (nx + 1) % (nx + 1), used // (nx + 1) ** 2
        s.coords = _host(torch.stack([nx - i, j, k], 1).double() / nx)
        s.conn = _host(conn.to(torch.int32))
        v = torch.tensor([1 + r.uniform(-0.2, 0.2), 1 + r.uniform(-0.2, 0.2), tilt], device=DEV, dtype=F64)
        v = v.expand(len(conn), 3).contiguous()
        hole = (i >= 4 * m) & (i <= 5 * m) & (j >= 4 * m) & (j <= 5 * m) & (k >= 4 * m) & (k <= 5 * m)
        mask = hole | (i == 0) | (i == nx) | (j == 0) | (j == nx) | (k == 0) | (k == nx)
        s.coef, s.dmask, s.dval, s.DM = _host(v), _host(mask.to(torch.uint8)), _host(hole.double()), 0.0
        s.c0 = s.dval.copy()
        return s
    i, j, k = _cells(nx, ny, nz)
    off = torch.zeros(6, 3, dtype=torch.int64)
    for p, perm in enumerate(_PERMS):
        for a, w in zip(perm, (3, 2, 1)):
            off[p, a] += w
    off = off.to(DEV)
    x = ((4 * i)[:, None] + off[:, 0]).reshape(-1).double() / (4.0 * nx)
    y = ((4 * j)[:, None] + off[:, 1]).reshape(-1).double() / (4.0 * ny)
    v = _vortex(x, y, r.random(), r.random())
    if field == "rotated":       # a random rotation per block of 10 x 10 x 10 hexahedra
        nb = [-(-n // 10) for n in (nx, ny, nz)]
        q = _rotations(g, nb[0] * nb[1] * nb[2])
        bid = i // 10 + nb[0] * (j // 10 + nb[1] * (k // 10))
        v = torch.einsum("hij,hpj->hpi", q[bid], v.reshape(-1, 6, 3)).reshape(-1, 3)
    s.coef = _host(v)
    i, j, k = _cells(nx + 1, ny + 1, nz + 1)
    patch = (i == 0) & (4 * j >= ny) & (4 * j <= 3 * ny) & (4 * k >= nz) & (4 * k <= 3 * nz)
    s.dmask, s.dval = _host((patch | (i == nx)).to(torch.uint8)), _host(patch.double())
    s.c0 = s.dval.copy()
    return s


def _case_spec(case, seed):
    return _spec(case["mesh"], case["nx"], case["ny"], case["nz"], case["field"], seed, case.get("dt", 0.0),
                 case.get("m", 0), case.get("tilt", 1.0))


def _batch_specs(case, seed):
    r = random.Random(seed)
    # the sizes belong to the case, the data to the seed
    sizes = random.Random(case["count"] * 1000003 + case["nmin"] * 1009 + case["nmax"])
    return [_spec("grid2d", n, n, 0, "tensor", r.randrange(1 << 30))
            for n in (sizes.randint(case["nmin"], case["nmax"]) for _ in range(case["count"]))]


def _serve_shapes(case):
    r = random.Random(case["count"] * 1000003 + case["nodes2d"] * 1009 + case["nodes3d"])
    shapes = []
    for k in range(case["count"]):
        if k % 2 == 0:
            n = round(math.sqrt(math.exp(r.uniform(math.log(1e3), math.log(case["nodes2d"]))))) - 1
            shapes.append(("grid2d", n, n, 0, "blocks2d"))
        else:
            n = round(math.exp(r.uniform(math.log(1e4), math.log(case["nodes3d"]))) ** (1 / 3)) - 1
            shapes.append(("grid3d", n, n, n, "rotated"))
    return shapes


def _counts(mesh, nx, ny, nz, m=0):
    """(dim, nodes, elements, nonzeros) of a mesh, nonzeros to within the boundary."""
    if mesh == "grid2d":
        n = (nx + 1) * (ny + 1)
        return 2, n, 2 * nx * ny, 7 * n
    n = (nx + 1) * (ny + 1) * (nz + 1)
    e = 6 * nx * ny * nz
    if mesh == "hole":
        n, e = n - max(m - 1, 0) ** 3, e - 6 * m ** 3
    return 3, n, e, 15 * n


# ------------------------------------------------------------------ one pass

def _opts(case):
    return P.solve_opts(solver=SOLVERS[case.get("solver", "gpcg")], precision=PRECISIONS[case["precision"]],
                        rtol=case["rtol"])


def _device(a):
    return torch.as_tensor(a, device=DEV)


def prepare(case, seed):
    kind = case["kind"]
    st = dict(kind=kind)
    if kind == "batch":
        specs = _batch_specs(case, seed)
        st["systems"] = [P.nn_assemble(P.Problem(s, device=DEV)) for s in specs]
        st["c0"] = [_device(s.c0) for s in specs]
        st["opts"] = _opts(case)
        return st
    if kind == "serve":
        r = random.Random(seed)
        st["specs"] = [_spec(*shape, r.randrange(1 << 30)) for shape in _serve_shapes(case)]
        st["problems"] = [P.Problem(s) for s in st["specs"]]
        st["server"] = P.nn_serve_create(16 << 30, P.serve_opts(solve=_opts(case)))
        return st
    spec = _case_spec(case, seed)
    st["problem"] = P.Problem(spec, device=DEV)
    if kind == "assemble":
        return st
    st["system"] = P.nn_assemble(st["problem"])
    if kind == "spmv":
        st["format"] = FORMATS[case["format"]]
        n = P.nn_system_describe(st["system"])["n_free"]
        g = torch.Generator(device=DEV).manual_seed(seed + 1)
        st["x"] = torch.rand(n, generator=g, device=DEV, dtype=F64)
        return st
    st["opts"] = _opts(case)
    st["c0"] = _device(spec.c0)
    if kind == "transient":
        st["steps"] = case["steps"]
    return st


def run(st):
    kind = st["kind"]
    if kind == "solve":
        c = st["c0"].clone()
        P.nn_qp_solve(st["system"], c, st["opts"])
        return c
    if kind == "transient":
        c = torch.empty_like(st["c0"])
        hist = torch.empty(st["steps"], len(c), dtype=F64, device=c.device)
        P.nn_transient(st["system"], st["c0"], st["steps"], c, hist, st["opts"])
        return {"final": c, "history": hist}
    if kind == "batch":
        cs = [c.clone() for c in st["c0"]]
        P.nn_batch_solve(st["systems"], cs, st["opts"])
        return cs
    if kind == "spmv":
        return P.nn_spmv(st["system"], st["x"], torch.empty_like(st["x"]), st["format"])
    if kind == "serve":
        ids = [P.nn_serve_submit(st["server"], p) for p in st["problems"]]
        P.nn_serve_drain(st["server"])
        cs = [np.empty_like(s.c0) for s in st["specs"]]
        for i, c in zip(ids, cs):
            P.nn_serve_poll(st["server"], i, c)
        return cs
    system = P.nn_assemble(st["problem"])
    d = P.nn_system_describe(system)
    dev = st["problem"].dval.device
    out = dict(A_rowptr=torch.empty(d["n_free"] + 1, dtype=torch.int64, device=dev),
               A_col=torch.empty(d["nnz_free"], dtype=torch.int32, device=dev),
               A_val=torch.empty(d["nnz_free"], dtype=F64, device=dev),
               b0=torch.empty(d["n_free"], dtype=F64, device=dev))
    for what, dst in out.items():
        P.nn_system_copy_out(system, what, dst)
    return out


def work(case):
    """Inputs read once and outputs written once.  A solve reads the operator
    (value and column of every nonzero), the right-hand side and the start and
    writes the solution; the number of its products depends on the method and
    is not part of this figure."""
    kind = case["kind"]
    if kind in ("batch", "serve"):
        if kind == "batch":
            sizes = random.Random(case["count"] * 1000003 + case["nmin"] * 1009 + case["nmax"])
            shapes = [("grid2d", n, n, 0) for n in (sizes.randint(case["nmin"], case["nmax"])
                                                    for _ in range(case["count"]))]
        else:
            shapes = [s[:4] for s in _serve_shapes(case)]
        b = f = 0
        for s in shapes:
            dim, n, e, nnz = _counts(*s)
            b += 12 * nnz + 24 * n if kind == "batch" else 8 * (dim + 1) * e + 17 * n
            f += 2 * nnz
        return dict(bytes=b, flops=f)
    dim, n, e, nnz = _counts(case["mesh"], case["nx"], case["ny"], case["nz"], case.get("m", 0))
    if kind == "assemble":   # coefficients, sources, Dirichlet data in; CSR of A and b0 out
        return dict(bytes=8 * (dim if dim == 3 else dim + 1) * e + 9 * n + 12 * nnz + 16 * n,
                    flops=(120 if dim == 3 else 50) * e)
    if kind == "spmv":
        return dict(bytes=12 * nnz + 16 * n, flops=2 * nnz)
    steps = case.get("steps", 1)
    return dict(bytes=(20 if steps > 1 else 12) * nnz + (16 + 8 * steps) * n, flops=2 * nnz * steps)


# ------------------------------------------------------------------ plain torch in 64 bits

def _torch_system(s):
    """(A, M, b0, free): the reduced system of a problem as coalesced sparse matrices."""
    dev = DEV
    if s.coords is not None:
        X, conn = _device(s.coords), _device(s.conn).long()
    elif s.dim == 2:
        i, j = _cells(s.nx + 1, s.ny + 1)
        X = torch.stack([i.double() / s.nx, j.double() / s.ny], 1)
        i, j = _cells(s.nx, s.ny)
        v = i + (s.nx + 1) * j
        conn = torch.stack([v, v + 1, v + s.nx + 2, v, v + s.nx + 2, v + s.nx + 1], 1).reshape(-1, 3)
    else:
        i, j, k = _cells(s.nx + 1, s.ny + 1, s.nz + 1)
        X = torch.stack([i.double() / s.nx, j.double() / s.ny, k.double() / s.nz], 1)
        i, j, k = _cells(s.nx, s.ny, s.nz)
        step = (1, s.nx + 1, (s.nx + 1) * (s.ny + 1))
        tets = []
        for p in _PERMS:
            v = [i + step[1] * j + step[2] * k]
            for a in p:
                v.append(v[-1] + step[a])
            tets.append(torch.stack(v, 1))
        conn = torch.stack(tets, 1).reshape(-1, 4)
    dim, nv, N = s.dim, s.dim + 1, len(X)
    J = (X[conn[:, 1:]] - X[conn[:, :1]]).transpose(1, 2)
    det = torch.linalg.det(J)
    vol = det.abs() / (2.0 if dim == 2 else 6.0)
    G = torch.linalg.inv(J)
    G = torch.cat([-G.sum(1, keepdim=True), G], 1)
    coef = _device(s.coef)
    if s.coef_kind == P.NN_COEF_TENSOR:
        at = torch.tensor([0, 1, 1, 2] if dim == 2 else [0, 1, 2, 1, 3, 4, 2, 4, 5], device=dev)
        D = coef[:, at].reshape(-1, dim, dim)
    else:
        speed = coef.norm(dim=1)[:, None, None]
        D = (s.aT * speed + s.DM) * torch.eye(dim, device=dev, dtype=F64)
        D = D + (s.aL - s.aT) * coef[:, :, None] * coef[:, None, :] / speed.clamp_min(1e-300)
    Ke = vol[:, None, None] * torch.einsum("eap,epq,ebq->eab", G, D, G)
    mask, val = _device(s.dmask).bool(), _device(s.dval)
    free = torch.nonzero(~mask).reshape(-1)
    fid = torch.full((N,), -1, device=dev)
    fid[free] = torch.arange(len(free), device=dev)
    b = torch.zeros(N, device=dev, dtype=F64)
    if s.f_elem is not None:
        b.index_add_(0, conn.reshape(-1), (_device(s.f_elem) * vol / nv).repeat_interleave(nv))
    lift = torch.where(mask, val, torch.zeros_like(val))[conn]
    b.index_add_(0, conn.reshape(-1), -torch.einsum("eab,eb->ea", Ke, lift).reshape(-1))
    rows, cols = fid[conn][:, :, None].expand(-1, nv, nv).reshape(-1), fid[conn][:, None, :].expand(-1, nv, nv).reshape(-1)
    on = (rows >= 0) & (cols >= 0)
    at = torch.stack([rows[on], cols[on]])

    def reduced(e):
        return torch.sparse_coo_tensor(at, e.reshape(-1)[on], (len(free), len(free))).coalesce()

    M = None
    if s.dt > 0:
        Me = vol[:, None, None] * (torch.ones(nv, nv, device=dev, dtype=F64) + torch.eye(nv, device=dev, dtype=F64))
        Me = Me / (nv * (nv + 1))
        M, Ke = reduced(Me), Ke + Me / s.dt
    return reduced(Ke), M, b[free], free


def _torch_qp(A, diag, b, lo, hi, x):
    """The box QP's minimiser: MPRGP (Dostal and Schoeberl 2005) on the system
    scaled by its diagonal, then CG on the face it ends on; None where it
    takes too long."""
    sc = diag.rsqrt()
    big = torch.sparse_csr_tensor(A.crow_indices(), A.col_indices(), A.values().abs(), A.shape)
    step = 1.5 / float((sc * (big @ sc)).max())
    low, high, rhs = lo / sc, hi / sc, sc * b
    zero = torch.zeros_like(b)

    def mul(v):
        return sc * (A @ (sc * v))

    def face(y):
        return (y > low) & (y < high)

    y = torch.minimum(torch.maximum(x / sc, low), high)
    g = mul(y) - rhs
    p = torch.where(face(y), g, zero)
    stop = 1e-13 * float(rhs.norm())
    for _ in range(40000):
        free = torch.where(face(y), g, zero)
        chop = torch.where(y <= low, g.clamp_max(0.0), torch.where(y >= high, g.clamp_min(0.0), zero))
        cut = torch.where(free > 0, torch.minimum(free, (y - low) / step), torch.maximum(free, (y - high) / step))
        cc, ff, norm2 = torch.stack([chop @ chop, cut @ free, free @ free + chop @ chop]).tolist()
        if math.sqrt(norm2) <= stop:
            break
        d = p if cc <= ff else chop
        Ad = mul(d)
        most = torch.where(d > 0, (y - low) / d, torch.where(d < 0, (y - high) / d, torch.full_like(d, math.inf))).min()
        gd, dAd, room = torch.stack([g @ d, d @ Ad, most]).tolist()
        if dAd <= 0.0:
            break
        a = min(gd / dAd, room)
        y, g = y - a * d, g - a * Ad
        free = torch.where(face(y), g, zero)
        if cc <= ff and a < room:
            p = free - ((free @ Ad) / dAd) * p
            continue
        if cc <= ff:              # a bound was met: a projected step with the fixed length
            y = torch.minimum(torch.maximum(y - step * free, low), high)
            g = mul(y) - rhs
        p = torch.where(face(y), g, zero)
    else:
        return None
    on = face(y)
    x = torch.where(y <= low, torch.full_like(x, lo), torch.where(y >= high, torch.full_like(x, min(hi, 1e300)), sc * y))
    for _ in range(2):            # each pass starts from the true residual of the one before
        r = torch.where(on, b - A @ x, zero)
        z = r / diag
        p, rz = z, torch.dot(r, z)
        last = 1e-10 * rz
        for k in range(8000):
            if k % 50 == 0 and bool(rz <= last):
                break
            q = torch.where(on, A @ p, zero)
            a = rz / torch.dot(p, q).clamp_min(1e-300)
            x, r = x + a * p, r - a * q
            z = r / diag
            new = torch.dot(r, z)
            p, rz = z + (new / rz.clamp_min(1e-300)) * p, new
    y = x.clamp(lo, hi)
    return y if bool((x - y).norm() <= 1e-13 * x.norm()) else None


def _csr(A):
    return A.to_sparse_csr()


def _diag(A):
    i, j = A.indices()
    return A.values()[i == j]


def _exact_solve(s, steps):
    A, M, b0, free = _torch_system(s)
    diag, A = _diag(A), _csr(A)
    M = _csr(M) if M is not None else None
    c = _device(s.c0)
    out = []
    for _ in range(steps):
        b = b0 if M is None else b0 + (M @ c[free]) / s.dt
        x = _torch_qp(A, diag, b, s.lo, s.hi, c[free])
        if x is None:
            return None
        c = _device(s.dval).clone()
        c[free] = x
        out.append(c)
    return torch.stack(out)


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve":
        return None          # a minute of solves
    if kind == "batch":
        if case["count"] * case["nmax"] > 500:
            return None      # a minute of solves one after another
        got = [_exact_solve(s, 1) for s in _batch_specs(case, seed)]
        return None if any(c is None for c in got) else [c[0] for c in got]
    n = _counts(case["mesh"], case["nx"], case["ny"], case["nz"], case.get("m", 0))[1]
    s = _case_spec(case, seed)
    if kind == "assemble":
        A, _, b0, _ = _torch_system(s)
        ptr = torch.zeros(len(b0) + 1, dtype=torch.int64, device=DEV)
        ptr[1:] = torch.cumsum(torch.bincount(A.indices()[0], minlength=len(b0)), 0)
        return dict(A_rowptr=ptr, A_col=A.indices()[1].to(torch.int32), A_val=A.values(), b0=b0)
    if kind == "spmv":
        A = _torch_system(s)[0]
        g = torch.Generator(device=DEV).manual_seed(seed + 1)
        x = torch.rand(A.shape[0], generator=g, device=DEV, dtype=F64)
        return _csr(A) @ x
    if n > (20000 if case["mesh"] == "grid2d" else 100000):
        return None          # more than 20 seconds of iterations
    if kind == "solve":
        c = _exact_solve(s, 1)
        return None if c is None else c[0]
    hist = _exact_solve(s, case["steps"])
    return None if hist is None else {"final": hist[-1], "history": hist}
