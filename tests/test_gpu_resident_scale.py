"""The scalar step of the resident CG phase at the ends of the number range and
of TRON's subspace tolerance."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import nn_inputs as I
import paper_1506_08435_gb300 as P

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _solve(kind, shift):
    spec = I.config1_steady_2d(n=40)
    spec.f_elem = spec.f_elem * 2.0 ** shift
    s = P.nn_assemble(P.Problem(spec, device=torch.device(DEV)))
    c = torch.zeros(spec.n_nodes, dtype=torch.float64, device=DEV)
    if kind == "batch":
        info = P.nn_batch_solve([s], [c], P.solve_opts())[0]
    else:
        info = P.nn_qp_solve(s, c, P.solve_opts(solver=dict(gpcg=P.NN_SOLVER_GPCG, tron=P.NN_SOLVER_TRON)[kind]))
    assert info["status"] == 0
    return c.cpu().numpy() * 2.0 ** -shift, info["spmv"]


@pytest.mark.parametrize("kind", ["gpcg", "tron", "batch"])
def test_data_scaled_by_powers_of_two_follow_the_same_path(kind):
    """No operation rounds differently, so the iterates are the unscaled ones
    shifted: r'D^-1 r is up to 2^1000 here, its square is not a number."""
    ref, products = _solve(kind, 0)
    for shift in (200, 270, 330, 480, -200, -270, -330):
        x, n = _solve(kind, shift)
        assert n == products, (shift, n, products)
        assert np.array_equal(x, ref), shift


@pytest.mark.parametrize("spec", [lambda: I.config1_steady_2d(n=60), lambda: I.config3_steady_3d(n=13)])
@pytest.mark.parametrize("ksp", [1e-8, 1e-14])
def test_tron_subspace_steps_to_the_last_digits(spec, ksp):
    """A subspace tolerance at or below what the recurrences can reach: every
    step ends and the solve converges."""
    spec = spec()
    s = P.nn_assemble(P.Problem(spec, device=torch.device(DEV)))
    c = torch.zeros(spec.n_nodes, dtype=torch.float64, device=DEV)
    info = P.nn_qp_solve(s, c, P.solve_opts(solver=P.NN_SOLVER_TRON, ksp_rtol=ksp, rtol=1e-12))
    assert info["status"] == 0 and info["kkt_rel"] <= 1e-12
