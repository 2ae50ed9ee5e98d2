"""Launching a step costs the host the same whatever the length of the march axis, and the
number of chunks that axis is cut into does not show in the result."""
import time

import numpy as np
import pytest

from paper_1901_02716_gb300 import inputs
from paper_1901_02716_gb300 import maclab as M

pytestmark = pytest.mark.gpu
D3 = inputs.D3Q19


@pytest.mark.parametrize("dims,kernel", [((16, 16, 65536), M.KERNEL_ROWS2), ((160, 8, 65536), M.KERNEL_FOLDED)])
def test_host_time_of_a_launch(dims, kernel):
    """A launch of some ten microseconds; a search over 65,536 chunk lengths takes 270 more.  Best
    of ten runs of twenty queued steps (the queue holds them without waiting for the device)."""
    torch = pytest.importorskip("torch")
    with M.Solver(D3, dims, 1.0, 1.0 / 6.0, M.F32, 0b111) as s:
        assert s.kernel_info()["kernel"] == kernel
        s.set_graph(0)
        s.step(2)
        best = 1e9
        for _ in range(10):
            torch.cuda.synchronize()
            t = time.perf_counter()
            s.step(20)
            best = min(best, (time.perf_counter() - t) / 20 * 1e6)
        torch.cuda.synchronize()
    assert best < 60.0, best


@pytest.mark.parametrize("dims", [(32, 16, 41), (64, 24, 17), (160, 8, 29), (100, 20, 33)])
def test_chunks_do_not_show(dims):
    case = inputs.random_case(D3, dims, 0b101, seed=211, u_amp=0.08, rho_amp=0.02, walls="box")
    out = []
    for tz in (0, 1, 3, 7, dims[2]):
        with M.Solver.from_case(case, M.F32) as s:
            s.set_tile(0, tz)
            s.step(5)
            out.append(s.get_lattice_state())
    for o in out[1:]:
        assert np.array_equal(o, out[0])
