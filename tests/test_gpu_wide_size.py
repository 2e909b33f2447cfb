"""The FP32 wide stencil on both sides of the line between two passes over every node (small grids: fewer launches) and
the march over the interior, with the launches counted; the march at the edges of its tiles (120 columns, full and a
node more or less, bands of rows) against the FP64 operator, which the oracle pins in test_gpu_wide.  Bars as in
test_gpu_wide_march: 2e-5 relative max-norm of one application on a random field, 1e-4 relative L2 of steps."""
import math

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

KINDS = ("robin", "displacement", "displacement", "robin")


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _problem(order, n, two=False):
    P = W.random_problem(kinds=KINDS, n=n, order=order, two_blocks=two)
    P.stencil = "wide"
    P.sources = [W.PointSource(0, (0.5, 0.5), (0.6, -0.8), 1.0, 3.0, 0.1)]
    return P


# grids on which a step is bound by its launches: none of them pays for the march and the streams beside it
@pytest.mark.parametrize("order,n,two", [(6, (151, 140), False), (6, (201, 177), True), (4, (301, 252), True), (2, (401, 327), True)])
def test_small_grids_take_two_passes(order, n, two):
    from paper_2003_12811_gb300 import Solver
    P = _problem(order, n, two)
    S = Solver(P, "fp32")
    z = [np.zeros((2, b.N2, b.N1)) for b in P.blocks]
    S.set_state(z, z, 0.0)
    S.sbp_profile(True)
    S.sbp_profile(False)                                     # counters only
    S.step(3, S.suggest_dt(0.25))
    launches = list(S.sbp_profile_read()[1])
    S.close()
    # a pass of fluxes and one of divergences per block, the face terms, the traces and the sources
    assert launches[0] == 3 * 2 * len(P.blocks) and launches[1] == 3 and launches[3] == 3


@pytest.mark.parametrize("order,n,two", [(6, (129, 2800), False), (6, (130, 2700), False), (6, (137, 2600), False), (6, (138, 2610), False),
                                         (6, (257, 1401), False), (6, (12600, 28), False), (6, (150, 1300), True), (4, (131, 2800), False),
                                         (2, (124, 2900), False)])
def test_march(order, n, two):
    from paper_2003_12811_gb300 import Solver
    P = _problem(order, n, two)
    u, noise = W.smooth_state(P), W.random_state(P)
    v = [3.0 * x for x in W.smooth_state(P, seed=5)]
    out = []
    for prec in ("fp64", "fp32"):
        S = Solver(P, prec)
        dt = S.suggest_dt(0.25)
        S.set_state(noise, noise, 0.0)
        r = S.apply()
        S.set_state([a - dt * b for a, b in zip(u, v)], u, 0.05)
        S.step(10, dt)
        leap = S.state()[1]
        S.sbp_set_state_rk4(u, v, 0.05)
        S.sbp_step_rk4(3, dt)
        out.append((r, leap, S.state()[1]))
        S.close()
    ref, got = out
    assert max(np.abs(a - b).max() for a, b in zip(got[0], ref[0])) <= 2e-5 * max(np.abs(b).max() for b in ref[0])
    for x, y in zip(got[1:], ref[1:]):
        err = math.sqrt(sum(np.sum((a - b) ** 2) for a, b in zip(x, y)) / sum(np.sum(b ** 2) for b in y))
        assert err <= 1e-4, err
