"""Host threads that solve on one system, each with a stream and a state of its
own, the system's first solves among them: the bits of the same solves one
after the other."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import nn_inputs as I
import paper_1506_08435_gb300 as P

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
THREADS = 8

CASES = dict(step=(lambda: I.config2_transient_3d(n=9, nsteps=1), {}),
             square=(lambda: I.config1_steady_2d(n=30), {}),
             tron=(lambda: I.config1_steady_2d(n=30), dict(solver=P.NN_SOLVER_TRON)),
             ssor=(lambda: I.config1_steady_2d(n=30), dict(precond=P.NN_PC_SSOR)),
             lbfgs=(lambda: I.config2_transient_3d(n=9, nsteps=1), dict(solver=P.NN_SOLVER_LBFGS)))


def _run(system, spec, opts, starts, parallel):
    out = [None] * len(starts)
    errors = []
    streams = [torch.cuda.Stream() for _ in starts]
    gate = threading.Barrier(len(starts) if parallel else 1)

    def one(k):
        try:
            gate.wait()
            with torch.cuda.stream(streams[k]):
                c = starts[k].clone()
                if spec.dt > 0:
                    info = P.nn_step(system, starts[k], c, opts)
                else:
                    info = P.nn_qp_solve(system, c, opts)
                assert info["status"] == 0
                out[k] = c.cpu().numpy()
        except Exception as e:          # (reported by the main thread)
            errors.append(e)

    torch.cuda.synchronize()
    if parallel:
        threads = [threading.Thread(target=one, args=(k,)) for k in range(len(starts))]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
    else:
        for k in range(len(starts)):
            one(k)
    assert not errors, errors
    return out


@pytest.mark.parametrize("case", sorted(CASES))
def test_first_solves_on_one_system_from_threads(case):
    make, opts = CASES[case]
    spec = make()
    rng = np.random.default_rng(7)
    base = spec.c0 if spec.c0 is not None else np.zeros(spec.n_nodes)
    free = np.asarray(spec.dmask) == 0
    starts = []
    for _ in range(THREADS):
        c = np.array(base)
        c[free] = np.clip(c[free] + rng.uniform(0.0, 0.3, free.sum()), spec.lo, spec.hi)
        starts.append(torch.tensor(c, device=DEV))
    o = P.solve_opts(**opts)
    fresh = P.nn_assemble(P.Problem(spec, device=torch.device(DEV)))
    got = _run(fresh, spec, o, starts, parallel=True)
    ref = _run(P.nn_assemble(P.Problem(spec, device=torch.device(DEV))), spec, o, starts, parallel=False)
    for a, b in zip(got, ref):
        assert np.array_equal(a, b)
