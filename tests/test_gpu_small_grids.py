"""Launch shapes of small systems: 256-thread blocks of four slices up to four
slices per SM, 512-thread blocks above and for fewer blocks by the caller's
choice, at the sizes where they change."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import nn_inputs as I
import paper_1506_08435_gb300 as P

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _solve(s, spec, **opts):
    c = torch.zeros(spec.n_nodes, dtype=torch.float64, device=DEV)
    info = P.nn_qp_solve(s, c, P.solve_opts(**opts))
    k = P.nn_kkt_residual(s, c)
    assert info["status"] == 0 and k["bounds_ok"] and k["kkt_rel"] <= 1e-9, k
    return c.cpu().numpy()


# cells a side: 1, 4, 5 slices; 5 x 76 slices and the next size; 4 x 152 slices and the next size
@pytest.mark.parametrize("n", [6, 12, 13, 110, 112, 140, 141])
@pytest.mark.parametrize("solver", [P.NN_SOLVER_GPCG, P.NN_SOLVER_TRON, P.NN_SOLVER_LBFGS])
def test_shapes_agree(n, solver):
    """The default shape and a caller's blocks: the same solution, to what the
    KKT tolerance leaves open (as in the layout tests of the resident phase)."""
    spec = I.config1_steady_2d(n=n)
    s = P.nn_assemble(P.Problem(spec, device=torch.device(DEV)))
    slices = (P.nn_system_describe(s)["n_free"] + 31) // 32
    ref = _solve(s, spec, solver=solver)
    again = _solve(s, spec, solver=solver)
    assert np.array_equal(ref, again)
    for blocks in {1, max(slices // 5, 1), (slices + 3) // 4, 152, 400}:
        if solver != P.NN_SOLVER_GPCG and blocks not in (152,):
            continue
        x = _solve(s, spec, solver=solver, grid_blocks=blocks)
        assert np.abs(x - ref).max() <= 1e-6 * max(np.abs(ref).max(), 1e-300)


@pytest.mark.parametrize("prec", [P.NN_PREC_FP64, P.NN_PREC_MIXED])
@pytest.mark.parametrize("n", [3, 5, 14, 25, 26])
def test_steps_with_the_operator_outside_are_the_same_bits(n, prec, monkeypatch):
    """256-thread blocks hold the operator in shared memory; read from memory
    (in 512-thread blocks of the same rows) the sums have the same order."""
    spec = I.config2_transient_3d(n=n, nsteps=2)
    s = P.nn_assemble(P.Problem(spec, device=torch.device(DEV)))
    out = []
    for flag in ("1", "0"):
        monkeypatch.setenv("NNQP_SMEM_OP", flag)
        c = torch.zeros(spec.n_nodes, dtype=torch.float64, device=DEV)
        infos = P.nn_transient(s, torch.tensor(spec.c0, device=DEV), spec.nsteps, c, None, P.solve_opts(precision=prec))
        assert all(i["status"] == 0 and i["kkt_rel"] <= 1e-10 for i in infos)
        out.append(c.cpu().numpy())
    assert np.array_equal(out[0], out[1])
