"""The FP64 interior edge weights are memory that a handle can do without: reported and given back on request, taken by
no served solve (admitted by footprint), given up by an idle handle when another's allocation finds no room, and kept by a
handle whose steps a caller has captured.  Bars: results with and without them differ by rounding
(1e-12 of the largest value after a few steps, as test_gpu_parity has for one application)."""
import threading

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

TOL = 1e-12


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _problem(order=6, n=(90, 71), two=False):
    return W.random_problem(kinds=("robin", "displacement", "displacement", "robin"), n=n, order=order, two_blocks=two)


def _planes(P):
    return sum(6 * (P.order // 2) * b.N2 * ((b.N1 + 31) // 32 * 32) * 8 for b in P.blocks)


def _start(P, **kw):
    from paper_2003_12811_gb300 import Solver
    S = Solver(P, "fp64", **kw)
    u, v = W.smooth_state(P), W.smooth_state(P, seed=5)
    dt = S.suggest_dt(0.25)
    S.set_state([a - dt * b for a, b in zip(u, v)], u, 0.0)
    return S, dt


def _stepped(P, n, **kw):
    S, dt = _start(P, **kw)
    S.step(n, dt)
    out = S.state()[1]
    S.close()
    return out


def _close(got, ref):
    return max(np.abs(a - b).max() for a, b in zip(got, ref)) <= TOL * max(np.abs(b).max() for b in ref)


def _run_out_of_memory(S):
    """A workspace that cannot fit on any device."""
    from paper_2003_12811_gb300 import SbpError
    S.sbp_set_receivers([(0, 3, 3)])
    with pytest.raises(SbpError) as e:
        S.sbp_misfit_gradient(20_000_000, 1e-4, np.zeros(2), checkpoint_every=20_000_000)
    assert "SBP_E_OOM" in str(e.value)


@pytest.mark.parametrize("order,n,two", [(2, (9, 7), False), (4, (40, 33), True), (6, (90, 71), False), (6, (700, 410), False)])
def test_given_back_and_taken_again(order, n, two):
    import torch
    P = _problem(order, n, two)
    ref = _stepped(P, 6, edge_weights=False)
    S, dt = _start(P)
    assert S.sbp_edge_weights() == _planes(P)
    free = torch.cuda.mem_get_info()[0]
    S.step(2, dt)
    assert S.sbp_edge_weights(0) == 0
    if _planes(P) >= 8 << 20:
        assert torch.cuda.mem_get_info()[0] - free >= _planes(P) - (4 << 20)
    S.step(2, dt)
    S.sbp_set_material(0, P.blocks[0].rho, __import__("paper_2003_12811_gb300").binding.pair10(P.blocks[0].C))
    assert S.sbp_edge_weights() == 0
    assert S.sbp_edge_weights(1) == _planes(P)
    S.step(2, dt)
    assert _close(S.state()[1], ref)
    S.close()


def test_fp32_wide_and_served_handles_hold_none():
    from paper_2003_12811_gb300 import Solver
    from paper_2003_12811_gb300.serve import GpuBackend
    P = _problem()
    S = Solver(P, "fp32")
    assert S.sbp_edge_weights(1) == 0
    S.close()
    P.stencil = "wide"
    S = Solver(P, "fp64")
    assert S.sbp_edge_weights(1) == 0
    S.close()
    shot = GpuBackend("fp64").create(W.shot_problem(61, 5), 0.3)
    assert shot.S.sbp_edge_weights() == 0
    shot.close()


def test_another_handle_takes_the_memory():
    from paper_2003_12811_gb300 import Solver
    P = _problem()
    ref = _stepped(P, 8)
    S, dt = _start(P)
    S.step(4, dt)
    assert S.sbp_edge_weights() > 0
    other = Solver(_problem(n=(31, 29)), "fp32")
    z = [np.zeros((2, b.N2, b.N1)) for b in other.problem.blocks]
    other.set_state(z, z, 0.0)
    _run_out_of_memory(other)
    other.close()
    assert S.sbp_edge_weights() == 0
    S.step(4, dt)
    assert _close(S.state()[1], ref)
    S.close()


@pytest.mark.parametrize("n", [(61, 57), (700, 410)])
def test_a_handle_with_captured_steps_keeps_them(n):
    """The kernels that a caller captured read the planes whenever the graph is replayed."""
    import torch
    from paper_2003_12811_gb300 import SbpError, Solver
    P = _problem(6, n)
    ref = _stepped(P, 6)
    S, dt = _start(P)
    st = torch.cuda.Stream()
    S.step(2, dt, st.cuda_stream)                             # (first launches are not captured)
    st.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        S.step(2, dt, st.cuda_stream)
    g.replay()
    torch.cuda.synchronize()
    with pytest.raises(SbpError) as e:
        S.sbp_edge_weights(0)
    assert "SBP_E_STATE" in str(e.value)
    other = Solver(_problem(n=(31, 29)), "fp32")
    z = [np.zeros((2, b.N2, b.N1)) for b in other.problem.blocks]
    other.set_state(z, z, 0.0)
    _run_out_of_memory(other)
    other.close()
    assert S.sbp_edge_weights() == _planes(P)
    g.replay()
    torch.cuda.synchronize()
    assert all(np.array_equal(a, b) for a, b in zip(S.state()[1], ref))
    S.close()


def test_threads():
    """One thread steps while another keeps running out of memory on a handle of its own."""
    P = _problem(n=(201, 203))
    ref = _stepped(P, 400)
    S, dt = _start(P)
    from paper_2003_12811_gb300 import Solver
    other = Solver(_problem(n=(31, 29)), "fp32")
    z = [np.zeros((2, b.N2, b.N1)) for b in other.problem.blocks]
    other.set_state(z, z, 0.0)
    failed = []

    def starve():
        try:
            for _ in range(20):
                _run_out_of_memory(other)
        except BaseException as e:                           # noqa: BLE001 (reported below)
            failed.append(e)

    t = threading.Thread(target=starve)
    t.start()
    for _ in range(200):
        S.step(2, dt)
        S.sbp_edge_weights(1)
    t.join()
    assert not failed, failed
    assert _close(S.state()[1], ref)
    S.close()
    other.close()
