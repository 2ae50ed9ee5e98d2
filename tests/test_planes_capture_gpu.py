"""maclab_get_planes and maclab_set_planes between device buffers are queued work only: on
padded rows too they allocate nothing, so a ghost exchange with its steps can be captured
in a graph, from the first call on."""
import numpy as np
import pytest

from paper_1901_02716_gb300 import inputs
from paper_1901_02716_gb300 import maclab as M

pytestmark = pytest.mark.gpu
D2, D3 = inputs.D2Q9, inputs.D3Q19


@pytest.mark.parametrize("lat,dims,periodic,walls,padded", [
    (D3, (64, 12, 9), 0b111, "none", False), (D3, (63, 40, 30), 0b000, "box", True),
    (D3, (95, 42, 40), 0b111, "none", True), (D2, (37, 21), 0b00, "box", True)])
def test_planes_in_a_captured_graph(lat, dims, periodic, walls, padded):
    torch = pytest.importorskip("torch")
    case = inputs.random_case(lat, dims, periodic, seed=231, u_amp=0.08, rho_amp=0.02, walls=walls)
    n = dims[-1]
    st = torch.cuda.Stream()
    with M.Solver(lat, dims, 1.0, 1.0 / 6.0, M.F32, periodic, case.node_type, case.wall_rho, case.wall_u,
                  stream=st.cuda_stream) as s:
        with torch.cuda.stream(st):
            s.set_state(torch.tensor(case.rho, device="cuda"), torch.tensor(case.u, device="cuda"))
            out = torch.empty(2 * s.state_bytes() // n, dtype=torch.uint8, device="cuda")
            back = torch.empty_like(out)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=st):  # the handle's first transfers
            M.maclab_get_planes(s.handle, 2, 2, out)
            M.maclab_set_planes(s.handle, 5, 2, out)
            M.maclab_get_planes(s.handle, 5, 2, back)
        graph.replay()
        torch.cuda.synchronize()
        raw = s.get_lattice_state()
        planes = raw.reshape(len(dims) + 1, n, -1)
        want = np.ascontiguousarray(planes[:, 2:4]).reshape(-1)
        assert np.array_equal(out.cpu().numpy(), want) and np.array_equal(back.cpu().numpy(), want)
        assert np.array_equal(planes[:, 5:7], planes[:, 2:4])
        # a buffer at an offset of one byte, and host memory
        odd = torch.empty(out.numel() + 1, dtype=torch.uint8, device="cuda")[1:]
        host = np.empty(out.numel(), dtype=np.uint8)
        M.maclab_get_planes(s.handle, 5, 2, odd)
        M.maclab_get_planes(s.handle, 5, 2, host)
        torch.cuda.synchronize()
        assert np.array_equal(odd.cpu().numpy(), want) and np.array_equal(host, want)
        M.maclab_set_planes(s.handle, 0, 2, odd)
        planes[:, 0:2] = planes[:, 5:7].copy()
        s.sync()
        assert np.array_equal(s.get_lattice_state(), raw)
