"""maclab_set_lattice_state puts the wall nodes' values into both state buffers (the step
kernels never write a wall node): with the raw state's own walls whatever the width, and
without a pass of its own over the node types on padded rows."""
import numpy as np
import pytest

from paper_1901_02716_gb300 import maclab as M

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def solver(dims, precision=M.F32):
    rng = np.random.default_rng(5)
    nt = (rng.random(tuple(reversed(dims))) < 0.3).astype(np.uint8)
    for axis in range(nt.ndim):  # closed
        edge = [slice(None)] * nt.ndim
        for i in (0, -1):
            edge[axis] = i
            nt[tuple(edge)] = 1
    d = len(dims)
    return M.Solver(M.D2Q9 if d == 2 else M.D3Q19, dims, 1.0, 1 / 6, precision, 0, node_type=nt,
                    wall_u=np.zeros((1, d))), nt


@pytest.mark.parametrize("precision", [M.F64, M.F32, M.BF16_STORE], ids=["f64", "f32", "bf16"])
@pytest.mark.parametrize("dims", [(8, 3), (13, 3), (16, 12), (17, 4), (31, 33), (64, 17), (256, 5), (257, 4),
                                  (13, 3, 5), (40, 9, 9), (16, 4, 4), (33, 5, 4), (64, 8, 9)], ids=str)
def test_walls_of_a_raw_state_reach_both_buffers(dims, precision):
    s, nt = solver(dims, precision)
    with s:
        raw = torch.empty(s.state_bytes(), dtype=torch.uint8, device="cuda")
        g = tuple(reversed(dims))
        rest = np.ones(g), np.zeros((len(dims),) + g)
        s.set_state(*rest)
        s.get_lattice_state(raw)
        value = {M.F64: torch.float64, M.F32: torch.float32, M.BF16_STORE: torch.bfloat16}[precision]
        first = raw.clone()
        fields = first.view(value).reshape(len(dims) + 1, -1)
        # rows of whole quads are stored as pairs (x, x + nx / 2)
        stored = nt
        if dims[0] % 4 == 0:
            stored = np.stack(np.split(nt, 2, axis=-1), axis=-1)
        wall = torch.from_numpy(stored.reshape(-1) != 0).cuda()
        step = torch.arange(fields.numel(), device="cuda").reshape(fields.shape) % 13 + 1
        fields[:, wall] += (step / 256.0).to(value)[:, wall]
        s.set_state(*rest)  # the table's values in both buffers
        s.set_lattice_state(first)
        for _ in range(3):  # either buffer is the current one
            s.get_lattice_state(raw)
            assert torch.equal(raw.view(value).reshape(fields.shape)[:, wall], fields[:, wall])
            s.step(1)


def microseconds(call):
    best = np.inf
    for _ in range(7):
        for _ in range(5):
            call()
        a, b = (torch.cuda.Event(enable_timing=True) for _ in "ab")
        torch.cuda.synchronize()
        a.record()
        for _ in range(100):
            call()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) * 10)
    return best


def set_raw(dims, precision=M.F32):
    nt = np.ones(tuple(reversed(dims)), np.uint8)
    nt[(slice(1, -1),) * len(dims)] = 0
    s = M.Solver(M.D2Q9 if len(dims) == 2 else M.D3Q19, dims, 1.0, 1 / 6, precision, 0, node_type=nt,
                 wall_u=np.zeros((1, len(dims))))
    with s:
        raw = torch.empty(s.state_bytes(), dtype=torch.uint8, device="cuda")
        s.get_lattice_state(raw)
        other = torch.empty_like(raw)
        return microseconds(lambda: s.set_lattice_state(raw)), microseconds(lambda: other.copy_(raw))


@pytest.mark.parametrize("n", [17, 61])
def test_padded_rows_take_one_launch(n):
    # one launch against a copy and a launch (4.1 us against 8.2); both as two launches 1.0
    padded, whole = set_raw((n, n))[0], set_raw((n + 3, n + 3))[0]
    assert padded <= 0.8 * whole, (padded, whole)


def test_walls_of_a_large_state_cost_less_than_its_copy():
    # 128^3 of 16 bits: copy and walls 12.3 us, the copy alone 6.2; looked at node by node 16.1
    both, copy = set_raw((128, 128, 128), M.BF16_STORE)
    assert both <= 2.3 * copy, (both, copy)
