"""The FP32 wide-stencil path (one marching pass over the interior, frame kernels near the faces) and the FP32
RK4 stages, against the FP64 oracle at the edges of their tiles: 120 columns of a wide tile and 128 of a narrow one,
full and one node more or less, bands of rows, blocks with a single interior node.  Bars as in test_gpu_parity: 2e-5
relative max-norm of one application on a random field, 1e-4 relative L2 of stepped smooth fields."""
import math

import numpy as np
import pytest

import workloads as W
from oracle.scheme import Oracle

pytestmark = pytest.mark.gpu

KINDS = ("robin", "displacement", "displacement", "robin")


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("order,n", [(2, (5, 5)), (2, (124, 6)), (4, (18, 18)), (4, (130, 29)), (4, (131, 40)),
                                     (6, (27, 27)), (6, (28, 90)), (6, (129, 43)), (6, (130, 27)), (6, (137, 61)),
                                     (6, (138, 44)), (6, (300, 45))])
@pytest.mark.parametrize("stencil", ["wide", "narrow"])
def test_apply(order, n, stencil):
    from paper_2003_12811_gb300 import Solver
    P = W.random_problem(kinds=KINDS, n=n, order=order)
    P.stencil = stencil
    O = Oracle(P)
    u = W.random_state(P)
    ref = O.unpack(O.A @ O.pack(u))
    S = Solver(P, "fp32")
    S.set_state(u, u, 0.0)
    got = S.apply()
    S.close()
    assert max(np.abs(a - b).max() for a, b in zip(got, ref)) <= 2e-5 * max(np.abs(b).max() for b in ref)


@pytest.mark.parametrize("stencil", ["wide", "narrow"])
@pytest.mark.parametrize("integrator", ["leapfrog", "rk4"])
@pytest.mark.parametrize("n", [(137, 61), (150, 70)])
def test_steps_with_sources(stencil, integrator, n):
    """Sources inside, near a face and across an interface; steps of smooth fields."""
    from paper_2003_12811_gb300 import Solver
    P = W.random_problem(kinds=KINDS, n=n, order=6, two_blocks=True)
    P.stencil = stencil
    P.sources = [W.PointSource(0, (0.5, 0.5), (0.6, -0.8), 1.0, 3.0, 0.1), W.PointSource(1, (0.4, 0.97), (0.0, 1.0), 1.0, 3.0, 0.1)]
    O = Oracle(P)
    dt = O.suggest_dt(0.25)
    u, v = W.smooth_state(P), [3.0 * x for x in W.smooth_state(P, seed=5)]
    S = Solver(P, "fp32")
    if integrator == "rk4":
        S.sbp_set_state_rk4(u, v, 0.05)
        S.sbp_step_rk4(6, dt)
        _, got = S.state()
        ref, _, _ = O.rk4(O.pack(u), O.pack(v), 0.05, dt, 6)
    else:
        prev = [a - dt * b for a, b in zip(u, v)]
        S.set_state(prev, u, 0.05)
        S.step(20, dt)
        _, got = S.state()
        _, ref, _ = O.leapfrog(O.pack(prev), O.pack(u), 0.05, dt, 20)
    S.close()
    ref = O.unpack(ref)
    err = math.sqrt(sum(np.sum((a - b) ** 2) for a, b in zip(got, ref)) / sum(np.sum(b ** 2) for b in ref))
    assert err <= 1e-4, err
