"""Batched solves at the limits of the device: cluster waits that run out."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import nn_inputs as I
import paper_1506_08435_gb300 as P

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _systems(sizes):
    specs = [I.config4_instance(i, nmin=n, nmax=n) for i, n in enumerate(sizes)]
    return specs, [P.nn_assemble(P.Problem(s, device=torch.device(DEV))) for s in specs]


def _solve(specs, systems, allow=(), **opts):
    cs = [torch.zeros(s.n_nodes, dtype=torch.float64, device=DEV) for s in specs]
    infos = P.nn_batch_solve(systems, cs, P.solve_opts(**opts), allow=allow)
    return [c.cpu().numpy() for c in cs], infos


@pytest.mark.parametrize("prec", [P.NN_PREC_FP64, P.NN_PREC_MIXED])
@pytest.mark.parametrize("sizes", [[20], [20, 57, 101], [24] * 200, [130, 24, 24]])
def test_cluster_waits_run_out_with_a_status(sizes, prec, monkeypatch):
    """Every instance reports TIMEOUT, those that no cluster took included, and
    the next call is as if nothing had happened."""
    specs, systems = _systems(sizes)
    ref, infos = _solve(specs, systems, precision=prec)
    assert all(i["status"] == 0 for i in infos)
    monkeypatch.setenv("NNQP_TEST_STALL_BARRIER", "1")
    t = time.time()
    _, infos = _solve(specs, systems, allow=(P.NN_ERR_TIMEOUT,), precision=prec, wait_timeout_s=0.2)
    assert time.time() - t < 20.0
    assert {i["status"] for i in infos} == {P.NN_ERR_TIMEOUT}
    with pytest.raises(P.NnError) as e:
        _solve(specs, systems, precision=prec, wait_timeout_s=0.2)
    assert e.value.status == P.NN_ERR_TIMEOUT
    monkeypatch.delenv("NNQP_TEST_STALL_BARRIER")
    again, infos = _solve(specs, systems, precision=prec)
    assert all(i["status"] == 0 for i in infos)
    for a, b in zip(ref, again):
        assert np.array_equal(a, b)
