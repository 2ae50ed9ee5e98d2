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
