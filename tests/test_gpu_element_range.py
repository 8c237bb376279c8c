"""Element sums where a quotient by a common reciprocal would leave the range:
infinite, huge and tiny sources, elements of extreme shape."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import nn_inputs as I
import paper_1506_08435_gb300 as P

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _full(spec):
    s = P.nn_assemble(P.Problem(spec, device=torch.device(DEV)), P.assemble_opts(keep_full=1))
    d = P.nn_system_describe(s)
    F = torch.empty(spec.n_nodes, dtype=torch.float64, device=DEV)
    K = torch.empty(d["nnz_full"], dtype=torch.float64, device=DEV)
    P.nn_system_copy_out(s, "F", F)
    P.nn_system_copy_out(s, "K_val", K)
    return F.cpu().numpy(), K.cpu().numpy()


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, 1e308, 1e-308, 5e-324])
@pytest.mark.parametrize("dim", [2, 3])
def test_sources_divide_as_numbers_do(value, dim):
    spec = I.tiny_2d(3, 3) if dim == 2 else I.tiny_3d(2, np.array([1.0, 0, 0, 1.0, 0, 1.0]))
    ref, _ = _full(spec)
    assert np.isfinite(ref).all()
    spec.f_elem = np.zeros_like(spec.f_elem)
    spec.f_elem[0] = value
    F, _ = _full(spec)
    vol = 1.0 / (len(spec.f_elem))
    share = value * vol / (dim + 1)
    got = F[F != 0] if not np.isnan(value) else F[np.isnan(F)]
    if share == 0.0:
        assert len(got) == 0
        return
    assert len(got) == dim + 1
    if np.isfinite(value):
        assert np.all(np.abs(got - share) <= 4e-16 * abs(share) + 5e-324)
    else:
        assert np.array_equal(got, np.full(dim + 1, value), equal_nan=True)


def test_thin_elements():
    """Edges of 1e-130 and 1e+130: the gradients are 1e+-130, their products
    with |e| and D = I representable."""
    for scale in (1.0, 1e130, 1e-130):
        coords = np.array([[0, 0], [1, 0], [1, 1], [0, 1]], float) * [scale, 1.0]
        conn = np.array([[0, 1, 2], [0, 2, 3]], np.int32)
        spec = I.ProblemSpec("thin", 2, 1, 1, 0, I.KIND_TENSOR, np.tile([scale, 0.0, 1 / scale], (2, 1)), np.ones(2),
                             np.array([1, 0, 0, 0], np.uint8), np.zeros(4), 0.0, np.inf, coords=coords, conn=conn)
        _, K = _full(spec)
        if scale == 1.0:
            ref = K
        assert np.all(np.abs(K - ref) <= 4e-15 * np.abs(ref).max())
