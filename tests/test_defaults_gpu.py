"""Which kernel the library takes by itself, where the choice shows in the result."""
import numpy as np
import pytest

from paper_1901_02716_gb300 import inputs
from paper_1901_02716_gb300 import maclab as M

pytestmark = pytest.mark.gpu
D2, D3 = inputs.D2Q9, inputs.D3Q19


@pytest.mark.parametrize("dims,walls", [((128, 16, 9), "box"), ((96, 8, 7), "mixed"), ((160, 12, 5), "none")])
@pytest.mark.parametrize("precision", [M.BF16_STORE, M.F16_STORE])
def test_16_bit_storage_keeps_the_folded_order(dims, walls, precision):
    """With 16-bit storage every step's rounding shows the order of the sums: where the folded
    kernel's tiles are whole, a run and its checkpoint have that kernel's bits."""
    case = inputs.random_case(D3, dims, 0b111 if walls == "none" else 0, seed=141, u_amp=0.08, rho_amp=0.02, walls=walls)
    out = []
    for kernel in (M.KERNEL_AUTO, M.KERNEL_FOLDED):
        with M.Solver.from_case(case, precision) as s:
            s.set_kernel(kernel)
            assert s.kernel_info()["kernel"] == M.KERNEL_FOLDED
            s.step(20)
            out.append(s.get_lattice_state())
    assert np.array_equal(*out)


def _box(dims, periodic):
    nt = np.zeros(tuple(reversed(dims)), np.uint8)
    for i in range(len(dims)):
        if not (periodic >> i) & 1:
            edge = [slice(None)] * len(dims)
            for k in (0, dims[i] - 1):
                edge[len(dims) - 1 - i] = k
                nt[tuple(edge)] = 1
    return dict(node_type=nt, wall_u=np.zeros((1, len(dims)))) if nt.any() else {}


@pytest.mark.parametrize("lat,dims,periodic,precision,name,launches", [
    # rows that no fast kernel takes, padded or not: natural rows, one launch a step
    (D3, (513, 40, 40), 0b111, M.F32, "step_naive", 1), (D3, (601, 20, 24), 0b001, M.BF16_STORE, "step_naive", 1),
    (D3, (55, 55, 55), 0b111, M.BF16_STORE, "step_naive", 1), (D3, (131, 3, 150), 0, M.F32, "step_naive", 1),
    (D2, (17, 16000), 0, M.F64, "step_naive", 1), (D2, (65, 4153), 0, M.F64, "step_naive", 1),
    (D2, (25, 6000), 0, M.F64, "step_naive", 1), (D2, (161, 1863), 0, M.F64, "step_naive", 1),
    (D2, (17, 20000), 0, M.F16_STORE, "step_naive", 1), (D2, (18, 66000), 0, M.F32, "step_naive", 1),
    # and the widths that padding brings to one
    (D3, (509, 40, 40), 0b111, M.F32, "step_fold", 2), (D3, (55, 55, 55), 0b111, M.F32, "step_rows2", 2),
    (D3, (51, 51, 51), 0, M.F32, "step_rows2", 1), (D3, (63, 7, 400), 0, M.F32, "step_tiled", 1),
    (D2, (17, 900), 0, M.F64, "step_block", 1), (D2, (257, 1167), 0, M.F64, "segment", 1),
    (D2, (401, 401), 0, M.F32, "step_block", 1), (D2, (25, 24000), 0, M.BF16_STORE, "segment", 1)])
def test_rows_are_padded_where_a_faster_kernel_takes_them(lat, dims, periodic, precision, name, launches):
    with M.Solver(lat, dims, 1.0, 1.0 / 6.0, precision, periodic, **_box(dims, periodic)) as s:
        info = s.kernel_info()
        assert info["name"].startswith(name) and info["launches_per_group"] == launches
        s.step(3)
        assert s.diagnostics()["nonfinite"] == 0
