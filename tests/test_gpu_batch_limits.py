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


@pytest.mark.parametrize("prec", [P.NN_PREC_FP64, P.NN_PREC_MIXED])
@pytest.mark.parametrize("most", [0, 1, 2, 8])
def test_clusters_that_the_device_does_not_schedule(most, prec, monkeypatch):
    """The next smaller cluster, or a block per instance, solves what a larger
    one would have."""
    specs, systems = _systems([20, 57, 101, 150])
    monkeypatch.setenv("NNQP_TEST_MAX_CLUSTER", str(most))
    xs, infos = _solve(specs, systems, precision=prec)
    assert all(i["status"] == 0 for i in infos)
    for s, sy, x in zip(specs, systems, xs):
        k = P.nn_kkt_residual(sy, torch.tensor(x, device=DEV))
        assert k["bounds_ok"] and k["kkt_rel"] <= 1e-8, (s.name, k)
    # a shape that was asked for by name is still refused, with every c untouched
    monkeypatch.setenv("NNQP_BATCH_SHAPE", "256x16")
    cs = [torch.full((s.n_nodes,), 0.5, dtype=torch.float64, device=DEV) for s in specs]
    with pytest.raises(P.NnError) as e:
        P.nn_batch_solve(systems, cs, P.solve_opts(precision=prec))
    assert e.value.status == P.NN_ERR_INVALID_ARG
    assert all(bool((c == 0.5).all()) for c in cs)
