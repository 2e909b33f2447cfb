"""sbp_batch_set_rows takes any positive height: one that no shot reaches means one band per column of tiles, and the
results are those of the default."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _run(rows):
    from paper_2003_12811_gb300 import Batch, Solver
    B = Batch(6, 2)
    B.sbp_batch_set_rows(rows)
    solvers = []
    for k, side in enumerate((61, 131)):
        S = Solver(W.shot_problem(side, 40 + k), "fp32")
        u = W.smooth_state(S.problem)
        S.set_state(u, u, 0.0)
        solvers.append((S, B.sbp_batch_add(S, 6, S.suggest_dt(0.3))))
    B.sbp_batch_step(6, None)
    B.sbp_batch_poll(None)
    out = []
    for S, slot in solvers:
        B.sbp_batch_remove(slot, None)
        out += S.state()[1]
        S.close()
    B.close()
    return out


@pytest.mark.parametrize("rows", [1, 4096, 2 ** 31 - 40, 2 ** 31 - 1])
def test_any_height(rows):
    assert all(np.array_equal(a, b) for a, b in zip(_run(rows), _run(0)))
