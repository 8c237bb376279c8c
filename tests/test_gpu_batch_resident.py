"""Batched solves with the resident CG phase: every cluster size, the operator
in shared memory and in global memory, instances that do not fit it at all, one
slice per instance, more instances than clusters, both precisions -- against
the oracle, and by the FP64 KKT measure of every instance."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import nn_inputs as I
import paper_1506_08435_gb300 as P
from tests.gpu_common import compare_solution, oracle_solution

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _instance(i, n):
    s = I.config4_instance(i, nmin=n, nmax=n)
    assert s.nx == n
    return s


def _solve(specs, prec):
    systems = [P.nn_assemble(P.Problem(s, device=torch.device(DEV))) for s in specs]
    cs = [torch.zeros(s.n_nodes, dtype=torch.float64, device=DEV) for s in specs]
    infos = P.nn_batch_solve(systems, cs, P.solve_opts(precision=prec, rtol=1e-10))
    assert [i["status"] for i in infos] == [0] * len(specs)
    for s, sy, c in zip(specs, systems, cs):
        k = P.nn_kkt_residual(sy, c)
        assert k["bounds_ok"] and k["kkt_rel"] <= 1e-8, (s.name, k)
    return [c.cpu().numpy() for c in cs]


@pytest.mark.parametrize("prec", [P.NN_PREC_FP64, P.NN_PREC_MIXED])
@pytest.mark.parametrize("shape,sizes", [
    (None, [3, 4, 9, 20, 33, 57, 80, 101]),          # the default: a cluster size for each
    (None, [5]),
    (None, [24] * 40 + [90]),                        # more instances than SMs' worth of clusters
    ("512x2", [12, 30, 55]),
    ("512x4", [30, 100, 130]),                       # the operator outside, and an instance that does not fit
    ("512x8", [64, 110]),
    ("512x16", [8, 129, 200]),
])
def test_batch_sizes(shape, sizes, prec, monkeypatch):
    if shape:
        monkeypatch.setenv("NNQP_BATCH_SHAPE", shape)
    specs = [_instance(i, n) for i, n in enumerate(sizes)]
    xs = _solve(specs, prec)
    for s, x in list(zip(specs, xs))[:6]:
        if s.nx > 60:
            continue                                 # (the oracle takes minutes there; the KKT test covers them)
        red, b, x_ref, _ = oracle_solution(s)
        if np.abs(b).max() > 0.0:
            compare_solution(x[red.free], x_ref, red.A, b, s.lo, s.hi)


def test_batch_on_a_side_stream_repeats_its_bits():
    specs = [_instance(i, n) for i, n in enumerate([15, 40, 90])]
    ref = _solve(specs, P.NN_PREC_FP64)
    with torch.cuda.stream(torch.cuda.Stream()):
        again = _solve(specs, P.NN_PREC_FP64)
    for a, b in zip(ref, again):
        assert np.array_equal(a, b)
