"""The tiled reverse step on rows of any width (natural rows, odd and even, with
the image of node 0 in the last pair's second lane; ragged tiles), against the reference two-kernel reverse step on the same
states: gradients, wall sums and the force gradient.  Both sum the same terms in
another order: bounds as for the interleaved rows (FP64 1e-12, FP32 2e-6 of the
largest value)."""
import numpy as np
import pytest

from paper_1901_02716_gb300 import inputs
from paper_1901_02716_gb300 import maclab as M

pytestmark = pytest.mark.gpu
D2, D3 = inputs.D2Q9, inputs.D3Q19


@pytest.mark.parametrize("lat,dims,periodic,walls", [
    (D2, (5, 9), 0b11, "none"), (D2, (6, 7), 0b01, "mixed"), (D2, (129, 33), 0b00, "box"), (D2, (511, 12), 0b11, "none"),
    (D2, (130, 16), 0b10, "mixed"), (D2, (3, 5), 0b11, "none"),
    (D3, (3, 3, 3), 0b111, "none"), (D3, (5, 6, 4), 0b111, "none"), (D3, (7, 13, 5), 0b000, "box"),
    (D3, (63, 9, 8), 0b101, "mixed"), (D3, (65, 10, 9), 0b111, "none"), (D3, (97, 11, 6), 0b011, "box"),
    (D3, (127, 5, 7), 0b110, "mixed"), (D3, (128, 7, 5), 0b111, "none"), (D3, (24, 21, 9), 0b110, "box"),
    (D3, (96, 18, 40), 0b111, "none"), (D3, (129, 6, 5), 0b111, "none"), (D3, (300, 5, 6), 0b111, "none")])
@pytest.mark.parametrize("precision", [M.F64, M.F32])
def test_reverse_step_on_any_rows(lat, dims, periodic, walls, precision):
    torch = pytest.importorskip("torch")
    case = inputs.random_case(lat, dims, periodic, seed=78, u_amp=0.08, rho_amp=0.02, walls=walls,
                              force=tuple([2e-4] * len(dims)))
    out = []
    for kern in (M.KERNEL_REFERENCE, M.KERNEL_AUTO):
        with M.Solver.from_case(case, precision) as s:
            s.set_kernel(kern)
            s0, s1 = (torch.empty(s.state_bytes(), dtype=torch.uint8, device="cuda") for _ in range(2))
            s.get_lattice_state(s0)
            s.step(1)
            s.get_lattice_state(s1)
            g = inputs.rng(79)
            lam1 = torch.empty(s.adjoint_bytes(), dtype=torch.uint8, device="cuda")
            lam0 = torch.full_like(lam1, 0x7b)
            M.maclab_adjoint_seed(s.handle, torch.tensor(g.standard_normal(case.rho.shape), device="cuda"),
                                  torch.tensor(g.standard_normal(case.u.shape), device="cuda"), s1, lam1)
            gf = torch.zeros(3, dtype=torch.float64, device="cuda")
            M.maclab_adjoint_step(s.handle, s0, s1, lam1, lam0, gf)
            gr = torch.empty(case.rho.shape, dtype=torch.float64, device="cuda")
            gu = torch.empty(case.u.shape, dtype=torch.float64, device="cuda")
            nw = 0 if case.wall_u is None else len(case.wall_u)
            res = M.maclab_adjoint_finish(s.handle, lam0, s0, gr, gu, 0.0, gf.cpu().tolist(), nw)
            out.append((gr.cpu().numpy(), gu.cpu().numpy(), res["wall"], gf.cpu().numpy()))
    (r1, u1, w1, f1), (r2, u2, w2, f2) = out
    tol = 1e-12 if precision == M.F64 else 2e-6
    assert np.abs(r1 - r2).max() <= tol * np.abs(r1).max()
    assert np.abs(u1 - u2).max() <= tol * np.abs(u1).max()
    assert np.allclose(w1, w2, rtol=tol * 10, atol=tol * max(np.abs(r1).max(), np.abs(u1).max()))
    assert np.allclose(f1, f2, rtol=1e-6 if precision == M.F32 else 1e-12, atol=tol * np.abs(u1).max())


@pytest.mark.parametrize("dims,periodic,walls", [
    ((3, 3, 3), 0b111, "none"), ((5, 6, 4), 0b111, "none"), ((7, 13, 5), 0b000, "box"), ((63, 9, 8), 0b101, "mixed"),
    ((65, 10, 9), 0b111, "none"), ((97, 11, 6), 0b011, "box"), ((127, 5, 7), 0b110, "mixed"), ((30, 7, 33), 0b100, "box")])
def test_viscosity_term_on_natural_rows(dims, periodic, walls):
    """The pass over natural rows (the state after the step given) against the
    per-node kernel.  A node's term is a sum of about 40 products of lam with
    values below 0.1 (second order in u = 0.08, first in drho = 0.02), so both
    differ by at most 40 * 0.1 * 2^-24 < 2^-21 of the sum of |lam|."""
    torch = pytest.importorskip("torch")
    case = inputs.random_case(D3, dims, periodic, seed=80, u_amp=0.08, rho_amp=0.02, walls=walls, force=(3e-4,) * 3)
    with M.Solver.from_case(case, M.F32) as s:
        s0, s1 = (torch.empty(s.state_bytes(), dtype=torch.uint8, device="cuda") for _ in range(2))
        s.get_lattice_state(s0)
        s.step(1)
        s.get_lattice_state(s1)
        g = inputs.rng(81)
        lam = torch.tensor(g.standard_normal(s.adjoint_bytes() // 4), dtype=torch.float32, device="cuda")
        node, rows = (torch.zeros(1, dtype=torch.float64, device="cuda") for _ in range(2))
        M.maclab_adjoint_nu_term(s.handle, s0, lam, node)
        M.maclab_adjoint_nu_term(s.handle, s0, lam, rows, s1)
    assert abs(float(node) - float(rows)) <= 2.0 ** -21 * float(lam.abs().double().sum())
    assert float(node) != 0.0
