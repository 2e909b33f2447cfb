"""The 3-D line-end kernels and the divergence that completes their partial sums, against the FP64 3-D
oracle where they meet: even and odd x1 sizes (the column that the vector alignment leaves to the line
kernel, the half-filled last pair), the smallest blocks of every order, every face kind at each corner.
Bars as in test_gpu_3d: 1e-12 (FP64) and 1e-5 (FP32) of the size of one term of the sums."""
import numpy as np
import pytest

from workloads import box3d as B
from oracle.scheme3d import Oracle3D

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("order,N", [(2, (5, 5, 5)), (2, (6, 5, 7)), (4, (18, 18, 18)), (4, (19, 20, 18)),
                                     (6, (27, 27, 27)), (6, (28, 27, 29)), (6, (66, 27, 28))])
@pytest.mark.parametrize("faces", [("traction", "displacement") * 3, ("displacement", "traction") * 3])
@pytest.mark.parametrize("prec,bar", [("fp64", 1e-12), ("fp32", 1e-5)])
def test_apply(order, N, faces, prec, bar):
    from paper_2003_12811_gb300 import Solver3D
    b = B.random_block3(N=N, order=order, faces=faces)
    O = Oracle3D(b)
    u = B.random_state3(b, seed=5)
    ref = O.accel(u)
    S = Solver3D.from_block(b, prec)
    got = S.apply(u)
    S.close()
    scale = O.w.max() * np.abs(O.c).max() * max(1.0 / op.h for op in O.op) ** 2 * np.abs(u).max()
    assert np.abs(got - ref).max() < bar * scale
