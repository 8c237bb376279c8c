"""Assembly at the edges of its per-node lists: fans up to and past the limits
on incidences and neighbours, isolated nodes, inverted elements, nearly
degenerate dispersion tensors, against the oracle; what is refused stays
refused."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import nn_inputs as I
import paper_1506_08435_gb300 as P
from tests.gpu_common import oracle_reduced

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _fan(m, extra=0):
    """m triangles around node 0, the rim on the Dirichlet boundary except one
    node; extra nodes that no element uses."""
    a = 2 * np.pi * np.arange(m) / m
    coords = np.concatenate([[[0.0, 0.0]], np.stack([np.cos(a), np.sin(a)], 1), np.full((extra, 2), 9.0)])
    j, k = np.arange(m), (np.arange(m) + 1) % m
    conn = np.stack([np.zeros(m, int), 1 + j, 1 + k], 1).astype(np.int32)
    conn[::2] = conn[::2][:, [0, 2, 1]]            # every other one clockwise
    mask = np.ones(len(coords), np.uint8)
    mask[[0, 1]] = 0
    return I.ProblemSpec("fan", 2, 1, 1, 0, I.KIND_TENSOR, np.tile([2.0, 0.3, 1.0], (m, 1)), np.linspace(0.5, 1.5, m),
                         mask, np.zeros(len(coords)), 0.0, 1.0, coords=coords, conn=conn)


def _assembled(spec, **kw):
    s = P.nn_assemble(P.Problem(spec, device=torch.device(DEV)), P.assemble_opts(**kw))
    d = P.nn_system_describe(s)
    out = {}
    for what, n, dt in (("A_rowptr", d["n_free"] + 1, np.int64), ("A_col", d["nnz_free"], np.int32),
                        ("A_val", d["nnz_free"], np.float64), ("b0", d["n_free"], np.float64),
                        ("K_col", d["nnz_full"], np.int32), ("K_val", d["nnz_full"], np.float64)):
        out[what] = P.nn_system_copy_out(s, what, np.zeros(n, dt))
    return out


def _against_oracle(spec):
    got = _assembled(spec)
    asm, red = oracle_reduced(spec)
    A = red.A.tocsr()
    A.sort_indices()
    assert np.array_equal(got["A_rowptr"], A.indptr) and np.array_equal(got["A_col"], A.indices)
    assert np.array_equal(got["K_col"], asm.col)
    # entries are sums of at most 64 element terms of a few rounded operations each: 64 eps of the largest
    assert np.abs(got["A_val"] - A.data).max() <= 1e-13 * np.abs(A.data).max()
    assert np.abs(got["b0"] - red.rhs(spec.c0) if spec.dt > 0 else got["b0"] - red.rhs()).max() <= 1e-13 * (
        np.abs(A.data).max() + np.abs(got["b0"]).max())


@pytest.mark.parametrize("m", [3, 7, 8, 9, 62, 63])
def test_fans_up_to_the_limit(m):
    _against_oracle(_fan(m))


@pytest.mark.parametrize("m", [64, 85, 86, 200])
def test_fans_past_the_limits_are_refused(m):
    with pytest.raises(P.NnError) as e:
        _assembled(_fan(m))
    assert e.value.status == P.NN_ERR_INVALID_ARG


def test_isolated_nodes_keep_their_diagonal():
    spec = _fan(12, extra=5)
    got = _assembled(spec)
    assert np.array_equal(got["K_col"][-5:], np.arange(13, 18)) and np.all(got["K_val"][-5:] == 0.0)


@pytest.mark.parametrize("sides", [(1, 1, 1), (2, 1, 3), (5, 4, 3), (7, 7, 7)])
def test_small_boxes(sides):
    nx, ny, nz = sides
    v = I.dispersion_velocities_3d(nx, ny, nz, rotate_seed=3)
    mask, val = I.patch_dirichlet_3d(nx, ny, nz)
    _against_oracle(I.ProblemSpec("box", 3, nx, ny, nz, I.KIND_VELOCITY, v, None, mask, val, 0.0, 1.0, aL=1.0,
                                  aT=1e-3, DM=1e-9))


@pytest.mark.parametrize("aL,aT,DM,scale", [(1.0, 1e-3, 0.0, 1.0), (1.0, 1e-7, 0.0, 1.0), (1e-3, 1.0, 1e-9, 1.0),
                                            (1.0, 1e-3, 1e-9, 0.0), (1.0, 1e-3, 1e-9, 1e-160), (1.0, 0.5, 0.0, 1e30)])
def test_dispersion_tensors(aL, aT, DM, scale):
    """The general path (minors formed), longitudinal below transversal
    dispersivity, no flow, and speeds whose squares leave the range."""
    v = scale * I.dispersion_velocities_3d(4, 4, 4, rotate_seed=5)
    mask, val = I.patch_dirichlet_3d(4, 4, 4)
    _against_oracle(I.ProblemSpec("disp", 3, 4, 4, 4, I.KIND_VELOCITY, v, None, mask, val, 0.0, 1.0, aL=aL, aT=aT,
                                  DM=DM))


@pytest.mark.parametrize("aL,aT,DM", [(1.0, 0.0, 0.0), (1.0, -1e-3, 0.0), (0.0, 0.0, 0.0)])
def test_singular_dispersion_is_refused(aL, aT, DM):
    v = np.tile([1.0, 0.0, 0.0], (6 * 8, 1))
    mask, val = I.patch_dirichlet_3d(2, 2, 2)
    spec = I.ProblemSpec("sing", 3, 2, 2, 2, I.KIND_VELOCITY, v, None, mask, val, 0.0, 1.0, aL=aL, aT=aT, DM=DM)
    with pytest.raises(P.NnError) as e:
        _assembled(spec)
    assert e.value.status == P.NN_ERR_NOT_SPD
