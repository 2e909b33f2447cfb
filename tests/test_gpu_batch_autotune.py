"""sbp_batch_autotune keeps the rule that divides the admitted shots' work evenly (rows = 0) unless a fixed height is
clearly faster on the shot it is timed with; the shot's state is left as it was."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def test_the_default_rule_is_a_candidate():
    from paper_2003_12811_gb300 import Batch, Solver
    P = W.shot_problem(301, 5)
    S = Solver(P, "fp32")
    u = W.smooth_state(P)
    S.set_state(u, u, 0.0)
    before = S.state()
    B = Batch(6, 2)
    chosen = [B.sbp_batch_autotune(S) for _ in range(5)]
    assert set(chosen) <= {0, 32, 64, 128, 256}
    assert 0 in chosen, chosen
    after = S.state()
    assert all(np.array_equal(a, b) for x, y in zip(before, after) for a, b in zip(x, y))
    B.close()
    S.close()
