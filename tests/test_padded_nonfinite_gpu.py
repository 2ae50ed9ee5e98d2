"""A density that is not a number, in the first and last columns of padded rows and away
from them: it reaches the nodes that the oracle's does, no other, and the rest of the state
stays by the oracle's: the padding, its periodic images and the seams between columns carry
none of it further.  Bounds: FP64 and FP32 a few tens of roundings of values below 1 and
0.2; 16 bits the four roundings of a state below 0.2, 4 * 0.2 * 2^-9 = 1.6e-3."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_1901_02716_gb300 import inputs
from paper_1901_02716_gb300 import maclab as M

pytestmark = pytest.mark.gpu
D2, D3 = inputs.D2Q9, inputs.D3Q19


@pytest.mark.parametrize("lat,dims,periodic,walls", [
    (D2, (17, 13), 0b00, "box"), (D2, (23, 40), 0b00, "mixed"), (D2, (401, 37), 0b00, "box"), (D2, (61, 61), 0b11, "none"),
    (D3, (63, 16, 50), 0b100, "box"), (D3, (126, 20, 20), 0b010, "mixed"), (D3, (251, 17, 12), 0b000, "box"),
    (D3, (33, 69, 66), 0b111, "none"), (D3, (95, 42, 38), 0b111, "none"), (D3, (127, 33, 36), 0b011, "box"),
    (D3, (251, 25, 24), 0b111, "none")], ids=str)
@pytest.mark.parametrize("precision", [M.F64, M.F32, M.BF16_STORE])
@pytest.mark.parametrize("steps", [1, 2, 3])
def test_reaches_the_nodes_it_should(lat, dims, periodic, walls, precision, steps):
    case = inputs.random_case(lat, dims, periodic, seed=111, u_amp=0.05, rho_amp=0.01, walls=walls)
    fluid = np.ones(case.rho.shape, bool) if case.node_type is None else case.node_type == 0
    middle = tuple(n // 2 for n in reversed(dims))[:-1]
    for column in (0, 1, dims[0] // 2, dims[0] - 2, dims[0] - 1):
        node = middle + (column,)
        if not fluid[node]:
            continue
        rho = case.rho.copy()
        rho[node] = np.nan
        want_rho, want_u = orc.step(lat, rho, case.u, periodic, wall=case.wall_mask, nsteps=steps)
        with M.Solver.from_case(case, precision) as s:
            s.set_state(rho, case.u)
            s.step(steps)
            got_rho, got_u = s.get_state()
        lost = np.isnan(want_rho)
        assert lost.any() and not lost[fluid].all()
        np.testing.assert_array_equal(np.isnan(got_rho), lost)
        np.testing.assert_array_equal(np.isnan(got_u), np.broadcast_to(lost, got_u.shape))
        tol = {M.F64: 1e-12, M.F32: 2e-6, M.BF16_STORE: 2e-3}[precision]
        assert np.abs(got_rho - want_rho)[~lost].max() <= tol
        assert np.abs(got_u - want_u)[:, ~lost].max() <= tol
