"""FP32 steps in one launch with strip tiles of 32 nodes (grids whose strips make too many short ones), with more
off-strip source nodes than the launch takes itself, and over several blocks that share no face: against the FP64 oracle,
with the launches counted.  The misfit gradient on such a grid against the FP64 one.  Bars as in test_gpu_parity (1e-4
relative L2 of stepped smooth fields) and test_gpu_adjoint (2e-3 of the largest entry in FP32)."""
import math

import numpy as np
import pytest

import workloads as W
from oracle.scheme import Oracle

pytestmark = pytest.mark.gpu

KINDS = ("robin", "displacement", "displacement", "robin")
STEPS = 12


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _against_oracle(P):
    from paper_2003_12811_gb300 import Solver
    O = Oracle(P)
    dt = O.suggest_dt(0.25)
    u, v = W.smooth_state(P), W.smooth_state(P, seed=5)
    prev = [a - dt * b for a, b in zip(u, v)]
    _, ref, _ = O.leapfrog(O.pack(prev), O.pack(u), 0.05, dt, STEPS)
    ref = O.unpack(ref)
    S = Solver(P, "fp32")
    S.set_state(prev, u, 0.05)
    S.sbp_profile(True)
    S.sbp_profile(False)                                     # counters only
    S.step(STEPS, dt)
    _, got = S.state()
    launches = S.sbp_profile_read()[1]
    S.close()
    err = math.sqrt(sum(np.sum((a - b) ** 2) for a, b in zip(got, ref)) / sum(np.sum(b ** 2) for b in ref))
    return err, list(launches)


@pytest.mark.parametrize("order,n", [(6, (27, 1300)), (6, (1301, 40)), (4, (18, 1400)), (2, (5, 1400))])
def test_long_tiles(order, n):
    P = W.random_problem(kinds=KINDS, n=n, order=order)
    # inside, at the face and beside the strip's edge
    P.sources = [W.PointSource(0, x, (0.6, -0.8), 1.0, 3.0, 0.1) for x in ((0.5, 0.5), (0.0, 0.3), (0.36, 0.98))]
    err, launches = _against_oracle(P)
    assert launches[0] == STEPS and launches[1] == 0 and launches[3] == 0
    assert err <= 1e-4, err


@pytest.mark.parametrize("n", [(27, 1300), (150, 141)])
def test_more_sources_than_the_launch_takes(n):
    P = W.random_problem(kinds=KINDS, n=n, order=6)
    P.sources = [W.PointSource(0, (0.5, 0.1 + 0.05 * k), (0.6, -0.8), 1.0, 3.0, 0.1) for k in range(16)]   # 16 x 36 nodes
    err, launches = _against_oracle(P)
    assert launches[0] == STEPS and launches[1] == 0 and launches[3] == STEPS
    assert err <= 1e-4, err


def test_blocks_that_share_no_face():
    P = W.random_problem(kinds=KINDS, n=(150, 60), order=6)
    P.blocks += W.random_problem(kinds=KINDS[::-1], n=(61, 300), order=6, seed=7).blocks
    P.blocks += W.random_problem(kinds=KINDS, n=(27, 27), order=6, seed=8).blocks
    P.sources = [W.PointSource(b, (0.5, 0.5), (0.6, -0.8), 1.0, 3.0, 0.1) for b in (0, 1)]
    err, launches = _against_oracle(P)
    assert launches[0] == STEPS and launches[1] == 0
    assert err <= 1e-4, err


def test_gradient_with_long_tiles():
    from paper_2003_12811_gb300 import Solver
    P = W.random_problem(kinds=KINDS, n=(27, 1300), order=6)
    P.sources = [W.PointSource(0, (0.45, 0.55), (0.3, -1.0), 1.0, 3.0, 0.3)]
    u = W.smooth_state(P, seed=1, amplitude=0.1)
    rec = [(0, i1, i2) for i1 in (3, 13, 25) for i2 in range(0, 1300, 90)]
    dt = Oracle(P).suggest_dt(0.5)
    rng = np.random.default_rng(3)
    obs = 0.05 * rng.standard_normal((STEPS, len(rec), 2))
    res = []
    for prec in ("fp64", "fp32"):
        S = Solver(P, prec)
        S.set_state(u, u, 0.0)
        S.sbp_set_receivers(rec)
        res.append(S.sbp_misfit_gradient(STEPS, dt, obs))
        S.close()
    (p64, r64, c64), (p32, r32, c32) = res
    assert p32 == pytest.approx(p64, rel=1e-4)
    assert np.max(np.abs(r32[0] - r64[0])) <= 2e-3 * np.max(np.abs(r64[0]))
    assert np.max(np.abs(c32[0] - c64[0])) <= 2e-3 * np.max(np.abs(c64[0]))
