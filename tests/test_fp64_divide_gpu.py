"""Eq. (5)'s division in FP64 storage, for every kernel that serves a domain: correctly
rounded, and with the IEEE results at the ends of the range."""
import numpy as np
import pytest

from paper_1901_02716_gb300 import inputs
from paper_1901_02716_gb300 import maclab as M

pytestmark = pytest.mark.gpu
D2, D3 = inputs.D2Q9, inputs.D3Q19


def kernels(s):
    for k in (M.KERNEL_AUTO, M.KERNEL_REFERENCE, M.KERNEL_TILED, M.KERNEL_SEGMENT, M.KERNEL_BLOCK):
        try:
            s.set_kernel(k)
        except M.MacLABError:
            continue
        yield k


@pytest.mark.parametrize("lat,dims", [(D2, (64, 12)), (D2, (37, 12)), (D3, (16, 8, 6))])
def test_infinite_density_divides_to_zero(lat, dims):
    """A resting state so dense that 36 drho' overflows: with integer weights m' = 0 exactly, so
    u' = 0 / inf = 0 (the reference kernel's rounded weights leave both finite)."""
    d = len(dims)
    with M.Solver(lat, dims, 1.0, 1.0 / 6.0, M.F64, (1 << d) - 1) as s:
        n = int(np.prod(dims))
        state = np.zeros((d + 1, n))
        state[0] = 6e306
        for k in kernels(s):
            if k == M.KERNEL_REFERENCE:
                continue
            s.set_lattice_state(state.view(np.uint8).reshape(-1))
            s.step(1)
            out = s.get_lattice_state().view(np.float64).reshape(d + 1, n)
            assert (out[1:] == 0.0).all(), k
            assert np.isinf(out[0]).all(), k


@pytest.mark.parametrize("lat,dims", [(D2, (64, 12)), (D2, (37, 12)), (D3, (16, 8, 6))])
def test_uniform_flow_keeps_its_velocity(lat, dims):
    """A uniform flow is a fixed point of the update, which then divides u (36 + R) by 36 + R: at
    most the roundings of the nineteen weighted sums and one each of the product and the quotient."""
    d = len(dims)
    with M.Solver(lat, dims, 1.0, 1.0 / 6.0, M.F64, (1 << d) - 1) as s:
        n = int(np.prod(dims))
        g = inputs.rng(171)
        for _ in range(20):
            drho, u = g.uniform(-0.5, 0.5), g.uniform(-0.1, 0.1, d)
            state = np.empty((d + 1, n))
            state[0] = drho
            state[1:] = u[:, None]
            for k in kernels(s):
                s.set_lattice_state(state.view(np.uint8).reshape(-1))
                s.step(1)
                out = s.get_lattice_state().view(np.float64).reshape(d + 1, n)
                assert np.abs(out[1:] - u[:, None]).max() <= 24 * 2.0 ** -53 * 1.0, k
