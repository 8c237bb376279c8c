"""The CG phase that keeps its vectors in shared memory (mid-size solves), at
the edges of its layout: one slice per block, partly filled last slices, empty
blocks, 4 / 8 / 12 compute warps with uneven slices per warp, narrow (2D) and
wide (3D) rows, rows of more than 16 entries, FP64 and the FP32 inner solves,
against the oracle and against the same form with its vectors in memory."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import nn_inputs as I
import paper_1506_08435_gb300 as P
from oracle import oracle as O
from tests.gpu_common import compare_solution, oracle_reduced, oracle_solution

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _steady(spec, **opts):
    s = P.nn_assemble(P.Problem(spec, device=torch.device(DEV)))
    c = torch.zeros(spec.n_nodes, dtype=torch.float64, device=DEV)
    info = P.nn_qp_solve(s, c, P.solve_opts(**opts))
    assert info["status"] == 0
    return c.cpu().numpy()


@pytest.mark.parametrize("n,blocks", [(2, 0), (3, 0), (9, 0), (30, 0), (30, 152), (60, 0), (60, 28), (60, 14), (60, 13),
                                      (60, 5), (60, 4), (60, 1)])
def test_2d_layouts(n, blocks):
    spec = I.config1_steady_2d(n=n)
    x = _steady(spec, grid_blocks=blocks)
    red, b, x_ref, _ = oracle_solution(spec)
    if np.abs(b).max() == 0.0:      # no source reaches the free nodes of the coarsest mesh
        assert np.array_equal(x, np.zeros_like(x))
        return
    compare_solution(x[red.free], x_ref, red.A, b, spec.lo, spec.hi)


@pytest.mark.parametrize("n,blocks", [(4, 0), (13, 0), (13, 17), (13, 3), (13, 2)])
def test_3d_layouts(n, blocks):
    spec = I.config3_steady_3d(n=n)
    x = _steady(spec, grid_blocks=blocks)
    red, b, x_ref, _ = oracle_solution(spec)
    compare_solution(x[red.free], x_ref, red.A, b, spec.lo, spec.hi)


def test_rows_of_more_than_sixteen_entries():
    """A fan of triangles: one node with 40 neighbours, the rows of the others
    narrow."""
    m = 40
    a = 2 * np.pi * np.arange(m) / m
    ring = np.stack([np.cos(a), np.sin(a)], 1)
    coords = np.concatenate([[[0.0, 0.0]], ring, 2 * ring])
    j, k = np.arange(m), (np.arange(m) + 1) % m
    conn = np.concatenate([np.stack([np.zeros(m, int), 1 + j, 1 + k], 1),
                           np.stack([1 + j, 1 + m + j, 1 + m + k], 1), np.stack([1 + j, 1 + m + k, 1 + k], 1)])
    mask = np.zeros(len(coords), np.uint8)
    mask[1 + m:] = 1
    E = len(conn)
    spec = I.ProblemSpec("fan", 2, 1, 1, 0, I.KIND_TENSOR, np.tile([2.0, 0.3, 1.0], (E, 1)), np.ones(E), mask,
                         np.zeros(len(coords)), 0.0, 0.4, coords=coords, conn=conn.astype(np.int32))
    x = _steady(spec)
    red, b, x_ref, _ = oracle_solution(spec)
    assert np.diff(red.A.indptr).max() > 17
    compare_solution(x[red.free], x_ref, red.A, b, spec.lo, spec.hi)


@pytest.mark.parametrize("prec", [P.NN_PREC_FP64, P.NN_PREC_MIXED])
@pytest.mark.parametrize("blocks", [0, 11, 9, 3])
def test_transient_layouts(prec, blocks, monkeypatch):
    """Every step is a KKT point by the oracle and equals, to the residual's
    share, the step with the vectors in memory (kkt_rel <= 1e-10 on both)."""
    spec = I.config2_transient_3d(n=12, nsteps=4)
    s = P.nn_assemble(P.Problem(spec, device=torch.device(DEV)))
    out = []
    for warps in (None, "0"):
        if warps is not None:
            monkeypatch.setenv("NNQP_RES_WARPS", warps)
        c0 = torch.tensor(spec.c0, device=DEV)
        hist = torch.zeros(spec.nsteps * spec.n_nodes, dtype=torch.float64, device=DEV)
        infos = P.nn_transient(s, c0, spec.nsteps, torch.zeros_like(c0), hist,
                               P.solve_opts(precision=prec, grid_blocks=blocks))
        assert all(i["status"] == 0 and i["kkt_rel"] <= 1e-10 for i in infos)
        out.append(hist.cpu().numpy().reshape(spec.nsteps, -1))
    asm, red = oracle_reduced(spec)
    prev = spec.c0
    for k in range(spec.nsteps):
        q = O.kkt(red.A, red.rhs(prev), spec.lo, spec.hi, out[0][k][red.free])
        assert q["bounds_ok"] and q["kkt_rel"] <= 1e-8
        prev = out[0][k]
    assert np.abs(out[0] - out[1]).max() <= 1e-6


@pytest.mark.parametrize("case", ["square9", "square60", "cube6", "cube13", "hole", "steps"])
@pytest.mark.parametrize("ksp", [1e-1, 1e-3])
def test_tron_layouts(case, ksp, monkeypatch):
    """TRON with its subspace CG resident: the oracle's KKT test, and the
    solution of the plain kernels (which the KKT tolerance fixes to 1e-6)."""
    spec = dict(square9=lambda: I.config1_steady_2d(n=9), square60=lambda: I.config1_steady_2d(n=60),
                cube6=lambda: I.config3_steady_3d(n=6), cube13=lambda: I.config3_steady_3d(n=13),
                hole=lambda: I.cube_with_hole(1), steps=lambda: I.config2_transient_3d(n=9, nsteps=3))[case]()
    s = P.nn_assemble(P.Problem(spec, device=torch.device(DEV)))
    opts = P.solve_opts(solver=P.NN_SOLVER_TRON, ksp_rtol=ksp)
    out = []
    for warps in (None, "0"):
        if warps is not None:
            monkeypatch.setenv("NNQP_RES_WARPS", warps)
        c = torch.zeros(spec.n_nodes, dtype=torch.float64, device=DEV)
        if spec.dt > 0:
            infos = P.nn_transient(s, torch.tensor(spec.c0, device=DEV), spec.nsteps, c, None, opts)
        else:
            infos = [P.nn_qp_solve(s, c, opts)]
        assert all(i["status"] == 0 and i["kkt_rel"] <= 1e-10 for i in infos)
        out.append(c.cpu().numpy())
    assert np.abs(out[0] - out[1]).max() <= 1e-6 * max(np.abs(out[1]).max(), 1e-300)
    if spec.dt == 0:
        red, b, x_ref, _ = oracle_solution(spec)
        compare_solution(out[0][red.free], x_ref, red.A, b, spec.lo, spec.hi)
