"""sbp3_footprint is an upper bound of the device memory that a 3-D handle takes, also where the line-end sums and the
face fields are more than the reserve it counts (order 2; blocks long in x1)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("order,N", [(2, (300, 200, 90)), (2, (5, 700, 600)), (4, (2000, 40, 38)), (6, (3000, 27, 28)), (6, (120, 118, 125))])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_handle_fits_its_footprint(order, N, prec):
    import torch
    from paper_2003_12811_gb300 import Solver3D
    from paper_2003_12811_gb300.binding import footprint3_bytes
    x = [np.linspace(0.0, 1.0, n) for n in N]
    X = np.stack(np.meshgrid(x[2], x[1], x[0], indexing="ij")[::-1])
    warm = Solver3D(X, ["displacement"] * 6, order=order, precision=prec)    # modules are loaded now
    warm.close()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    S = Solver3D(X, ["displacement"] * 6, order=order, precision=prec)
    held = before - torch.cuda.mem_get_info()[0]
    S.close()
    # the allocator hands out 2 MiB pages: at most one more for each of the 11 buffers
    assert held <= footprint3_bytes(N, prec, order) + 11 * (2 << 20)
