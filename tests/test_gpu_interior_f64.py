"""The FP64 interior kernel with edge weights kept in memory and the FP64 boundary strips, against the
FP64 oracle: grids at which each tile shape and each strip-tile length is chosen, with full and ragged tiles, more blocks than one launch takes, and a handle
that had to give the edge weights back.  Bar as in test_gpu_parity: 1e-12 relative max-norm of one
operator application on a random field."""
import numpy as np
import pytest

import workloads as W
from oracle.scheme import Oracle

pytestmark = pytest.mark.gpu

FP64_TOL = 1e-12


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _deviation(S, O, u):
    ref = O.unpack(O.A @ O.pack(u))
    got = S.apply()
    return max(np.abs(a - b).max() for a, b in zip(got, ref)) / max(np.abs(b).max() for b in ref)


# (order, n1, n2): one interior row or column, one tile exactly and one node more, 16 x 4 / 32 x 4 /
# 32 x 8 / 32 x 16 tiles, long thin blocks
@pytest.mark.parametrize("order,n", [(2, (5, 5)), (2, (36, 9)), (2, (181, 133)), (4, (18, 18)), (4, (45, 29)),
                                     (4, (131, 127)), (6, (27, 27)), (6, (34, 22 + 5)), (6, (51, 35)),
                                     (6, (201, 201)), (6, (261, 262)), (6, (700, 28)), (6, (28, 413)),
                                     (6, (1301, 28)), (6, (28, 1315))])
def test_apply_matches_oracle(order, n):
    from paper_2003_12811_gb300 import Solver
    P = W.random_problem(kinds=("robin", "displacement", "displacement", "robin"), n=n, order=order)
    u = W.random_state(P)
    S = Solver(P, "fp64")
    S.set_state(u, u, 0.0)
    assert _deviation(S, Oracle(P), u) <= FP64_TOL
    S.close()


@pytest.mark.parametrize("n", [(61, 57), (413, 29), (1301, 28)])
def test_point_sources_on_strip_tiles_of_each_length(n):
    """Sources at a corner, along the bottom band and on the right side: their nodes are found by the
    strip tile (8, 16, 32 nodes long on these grids) that owns them."""
    from paper_2003_12811_gb300 import Solver
    P = W.random_problem(kinds=("robin", "displacement", "displacement", "robin"), n=n, order=6)
    P.sources = [W.PointSource(0, x, (0.6, -0.8), 1.0, 3.0, 0.1) for x in ((0.0, 0.0), (0.51, 0.07), (1.0, 0.46))]
    O = Oracle(P)
    u = W.random_state(P)
    ref = O.unpack(O.apply(O.pack(u), 0.12))
    S = Solver(P, "fp64")
    S.set_state(u, u, 0.0)
    got = S.apply(True, 0.12)
    assert max(np.abs(a - b).max() for a, b in zip(got, ref)) <= FP64_TOL * max(np.abs(b).max() for b in ref)
    S.close()


def test_more_blocks_than_a_launch_takes():
    from paper_2003_12811_gb300 import Solver
    P = W.config2(n=28, nbx=6, nby=6)
    u = W.random_state(P)
    S = Solver(P, "fp64")
    S.set_state(u, u, 0.0)
    assert _deviation(S, Oracle(P), u) <= FP64_TOL
    S.close()


def test_without_room_for_the_edge_weights():
    """A workspace that cannot fit is refused as before; the handle has given its edge weights back by
    then and goes on with the kernel that forms them."""
    from paper_2003_12811_gb300 import Solver, SbpError
    P = W.random_problem(kinds=("robin", "displacement", "displacement", "robin"), n=(60, 45), order=6)
    u = W.random_state(P)
    O = Oracle(P)
    S = Solver(P, "fp64")
    S.sbp_set_receivers([(0, 3, 3)])
    S.set_state(u, u, 0.0)
    with pytest.raises(SbpError) as e:
        S.sbp_misfit_gradient(20_000_000, 1e-4, np.zeros(2), checkpoint_every=20_000_000)
    assert "SBP_E_OOM" in str(e.value)
    assert _deviation(S, O, u) <= FP64_TOL
    S.sbp_set_material(0, P.blocks[0].rho, __import__("paper_2003_12811_gb300").binding.pair10(P.blocks[0].C))
    assert _deviation(S, O, u) <= FP64_TOL
    S.close()
