"""The periodic images of padded rows cost a small launch a step, not a second wave of the
step's blocks.  A closed domain of the same size has no images; best of five, bar 4.7 us more (the
launch takes 2 to 4; a step whose blocks leave the images' kernel no place 5 to 10)."""
import numpy as np
import pytest

from paper_1901_02716_gb300 import maclab as M

pytestmark = pytest.mark.gpu


def _us(torch, dims, periodic):
    kw = {}
    if not periodic:
        nt = np.zeros(tuple(reversed(dims)), np.uint8)
        for axis in range(3):
            edge = [slice(None)] * 3
            for i in (0, nt.shape[axis] - 1):
                edge[axis] = i
                nt[tuple(edge)] = 1
        kw = dict(node_type=nt, wall_u=np.zeros((1, 3)))
    with M.Solver(M.D3Q19, dims, 1.0, 1.0 / 6.0, M.F32, 0b111 if periodic else 0, **kw) as s:
        best = 1e9
        for _ in range(5):
            s.step(20)
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            a.record()
            s.step(200)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) / 200 * 1e3)
    return best


@pytest.mark.parametrize("dims", [(65, 65, 65), (81, 81, 81), (130, 40, 60)])
def test_images_cost_a_launch(dims):
    torch = pytest.importorskip("torch")
    periodic, closed = _us(torch, dims, True), _us(torch, dims, False)
    assert periodic <= closed + 4.7, (periodic, closed)
