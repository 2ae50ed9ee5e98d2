"""The force gradient of the reverse step: the sum of lam_u over the fluid nodes, kept to
what FP64 sums of the same values give, whatever kernel the row width takes.

A thread's sum of up to 32 FP32 values keeps the error of every addition in a second
word, whose own additions round: 32 * 2^-24 of at most 32 * 2^-25, below 2^-39 of the sum
of magnitudes; sums between threads are in FP64."""
import numpy as np
import pytest

from paper_1901_02716_gb300 import inputs
from paper_1901_02716_gb300 import maclab as M

pytestmark = pytest.mark.gpu
D2, D3 = inputs.D2Q9, inputs.D3Q19


@pytest.mark.parametrize("lat,dims,periodic,walls", [
    (D2, (129, 33), 0b00, "box"), (D2, (130, 40), 0b11, "none"), (D2, (256, 20), 0b10, "mixed"),
    (D3, (27, 13, 25), 0b111, "none"), (D3, (97, 11, 26), 0b010, "mixed"), (D3, (64, 21, 17), 0b111, "none"),
    (D3, (32, 16, 24), 0b000, "box")])
def test_force_gradient_is_the_sum_of_lam(lat, dims, periodic, walls):
    torch = pytest.importorskip("torch")
    case = inputs.random_case(lat, dims, periodic, seed=161, u_amp=0.08, rho_amp=0.02, walls=walls,
                              force=(1e-4,) * len(dims))
    d, nx = len(dims), dims[0]
    with M.Solver.from_case(case, M.F32) as s:
        s0, s1 = (torch.empty(s.state_bytes(), dtype=torch.uint8, device="cuda") for _ in range(2))
        s.get_lattice_state(s0)
        s.step(1)
        s.get_lattice_state(s1)
        lam = inputs.rng(162).standard_normal((d + 1,) + case.rho.shape).astype(np.float32)
        l1 = torch.tensor(lam, device="cuda")
        l0 = torch.empty_like(l1)
        gf = torch.zeros(3, dtype=torch.float64, device="cuda")
        M.maclab_adjoint_step(s.handle, s0, s1, l1, l0, gf)
    fluid = np.ones(case.rho.shape, bool) if case.node_type is None else np.asarray(case.node_type) == 0
    if nx % 4 == 0:  # the stored order of a row: its two halves interleaved
        fluid = fluid.reshape(fluid.shape[:-1] + (2, nx // 2)).swapaxes(-1, -2).reshape(fluid.shape)
    for i in range(d):
        v = lam[1 + i][fluid].astype(np.float64)
        assert abs(float(gf[i]) - v.sum()) <= 2.0 ** -39 * np.abs(v).sum()
