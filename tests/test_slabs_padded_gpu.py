"""Slabs of domains whose width is not a multiple of 4: whether rows are stored padded (and so
which kernel sums a node's terms, in which order) depends on the domain's size, and the slabs
follow the undivided domain, not their own: interiors bit for bit equal to its run."""
import numpy as np
import pytest

from paper_1901_02716_gb300 import inputs, slabs
from paper_1901_02716_gb300 import maclab as M

pytestmark = pytest.mark.gpu
D2, D3 = inputs.D2Q9, inputs.D3Q19


# the undivided domain on padded rows and its slabs by themselves on natural ones, or the other way round
@pytest.mark.parametrize("lat,dims,periodic,walls,k,kernel", [
    (D3, (63, 63, 63), 0b000, "box", 8, "step_rows2"), (D3, (63, 40, 50), 0b110, "mixed", 5, "step_rows2"),
    (D3, (95, 42, 64), 0b111, "none", 7, "step_rows2"), (D3, (251, 30, 33), 0b101, "box", 4, "step_fold"),
    (D2, (17, 1600), 0b10, "box", 8, "step_naive"), (D2, (401, 300), 0b00, "mixed", 3, "step_block")])
@pytest.mark.parametrize("precision", [M.F32, M.F64, M.BF16_STORE])
def test_slabs_equal_undivided_run(lat, dims, periodic, walls, k, kernel, precision):
    case = inputs.random_case(lat, dims, periodic, seed=221, u_amp=0.08, rho_amp=0.02, walls=walls)
    s = M.Solver.from_case(case, precision)
    if precision == (M.F64 if kernel == "step_naive" else M.F32):
        assert s.kernel_tag().startswith(kernel)
    s.step(8)
    r1, u1 = s.get_state()
    s.close()
    for depth in (1, 4):
        dom = slabs.SlabDomain(case, k, precision, depth=depth)
        dom.step(8)
        r2, u2 = dom.get_state()
        dom.close()
        assert np.array_equal(r1, r2) and np.array_equal(u1, u2)


def test_create_slab_checks_its_planes():
    cfg, keep = M.make_config(D3, (8, 8, 8), 1.0, 1.0 / 6.0, M.F32, 0b111, None, None, None, None, 1.0, None)
    for planes in (0, -1, (1 << 30) + 1):
        with pytest.raises(M.MacLABError) as e:
            M.maclab_create_slab(cfg, planes)
        assert e.value.status == M.ERR_INVALID
