"""Misfit gradient with respect to the stiffness near the faces (k_grad_lines: narrow rows of the line ends;
k_grad_strip: the other terms) against the oracle's explicit-transpose adjoint: the smallest grids, a number of lines
beside a multiple of the launch's block, one level and a remainder of levels per segment.  Bar as in test_gpu_adjoint
(FP64, 1e-12 of the largest entry)."""
import numpy as np
import pytest

import workloads as W
from oracle import adjoint as AD
from oracle.scheme import Oracle

pytestmark = pytest.mark.gpu

NSTEPS = 15


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("order,n,every", [(2, (9, 7), 1), (4, (19, 21), 4), (6, (27, 70), 15), (6, (64, 29), 7)])
def test_gradient_near_faces(order, n, every):
    kinds = ("robin", "displacement", "displacement", "robin")
    P, Q = (W.random_problem(kinds=kinds, n=n, order=order, seed=s) for s in (3, 4))
    for X in (P, Q):
        X.sources = [W.PointSource(0, (0.45, 0.55), (0.3, -1.0), 1.0, 3.0, 0.3)]
    dt = Oracle(P).suggest_dt(0.5)
    u0 = W.smooth_state(P, seed=1, amplitude=0.1)
    rec = [(0, i1, i2) for i1 in range(0, n[0], 4) for i2 in range(0, n[1], 5)]
    oq = Oracle(Q)
    obs = AD.traces(oq, AD.forward(oq, u0, u0, 0.0, dt, NSTEPS)[0], rec)
    # every depth of the line ends, at lines inside and in the corners
    params = []
    for d in range(min(14, min(n) // 2)):
        for pl in ((0, 4, 7)[d % 3], 9):
            params += [(0, pl, d, n[1] // 2), (0, pl, n[0] - 1 - d, 2), (0, pl, n[0] // 2, d), (0, pl, n[0] - 3, n[1] - 1 - d)]
    ref = AD.gradient(P, u0, u0, 0.0, dt, NSTEPS, rec, obs, params)
    from paper_2003_12811_gb300 import Solver
    S = Solver(P, "fp64")
    S.set_state(u0, u0, 0.0)
    S.sbp_set_receivers(rec)
    phi, gr, gc = S.sbp_misfit_gradient(NSTEPS, dt, obs, checkpoint_every=every)
    S.close()
    assert phi == pytest.approx(ref["misfit"], rel=1e-12)
    assert np.max(np.abs(gr[0] - ref["grad_rho"][0])) <= 1e-12 * np.max(np.abs(ref["grad_rho"][0]))
    got = np.array([gc[b][pl, i2, i1] for (b, pl, i1, i2) in params])
    err = np.abs(got - ref["grad_C"])
    assert np.all(err <= 1e-12 * np.max(np.abs(ref["grad_C"]))), [(params[k], got[k], ref["grad_C"][k]) for k in np.argsort(-err)[:5]]
