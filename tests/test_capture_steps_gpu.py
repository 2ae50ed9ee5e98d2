"""The first steps of a handle captured in the caller's graph: a default grid whose steps need
no memory of their own takes none then (the block kernel, small and large), and the graph's
replays give the bits of the same steps without it."""
import numpy as np
import pytest

from paper_1901_02716_gb300 import inputs
from paper_1901_02716_gb300 import maclab as M

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(256, 60), (600, 520), (517, 600), (1000, 700)], ids=str)
@pytest.mark.parametrize("steps", [1, 5])
def test_first_steps_in_a_captured_graph(dims, steps):
    torch = pytest.importorskip("torch")
    case = inputs.random_case(inputs.D2Q9, dims, 0, seed=241, u_amp=0.05, rho_amp=0.01, walls="box")
    with M.Solver.from_case(case, M.F32) as s:
        for n in (2 * steps, 2 * steps, 3):  # two replays for every step call: an even count of steps each
            s.step(n)
        want = s.get_lattice_state()
    st = torch.cuda.Stream()
    with M.Solver.from_case(case, M.F32, stream=st.cuda_stream) as s:
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=st):
            s.step(steps)
            s.step(steps)
        graph.replay()
        graph.replay()
        torch.cuda.synchronize()
        s.step(3)
        assert np.array_equal(s.get_lattice_state(), want)
