"""The reverse step at the widths where its kernel changes.  FP64 interleaved rows, each
built block of the rows kernel and ragged y, against the reference two-kernel reverse step
on the same states (the same terms in another order: 1e-12 of the largest value).  Widths
that no tiled reverse step serves run the reference kernels whatever is asked, so these
are compared with the oracle's reverse step instead (FP64 1e-11; FP32 2e-5, states and
lam rounded to 32 bits)."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_1901_02716_gb300 import inputs
from paper_1901_02716_gb300 import maclab as M

pytestmark = pytest.mark.gpu
D2, D3 = inputs.D2Q9, inputs.D3Q19


@pytest.fixture(scope="module")
def torch():
    from paper_1901_02716_gb300 import _build
    _build.build()
    return pytest.importorskip("torch")


def reverse(torch, case, precision, kernel, lr, lu):
    """(lam_rho, lam_u, force gradient) one step back from (lr, lu)."""
    with M.Solver.from_case(case, precision) as s:  # e = 1, rho0 = 1
        s.set_kernel(kernel)
        s0, s1 = (torch.empty(s.state_bytes(), dtype=torch.uint8, device="cuda") for _ in range(2))
        s.get_lattice_state(s0)
        s.step(1)
        s.get_lattice_state(s1)
        lam1 = torch.empty(s.adjoint_bytes(), dtype=torch.uint8, device="cuda")
        lam0 = torch.full_like(lam1, 0x7b)
        M.maclab_adjoint_seed(s.handle, torch.tensor(lr, device="cuda"), torch.tensor(lu, device="cuda"), s1, lam1)
        gf = torch.zeros(3, dtype=torch.float64, device="cuda")
        M.maclab_adjoint_step(s.handle, s0, s1, lam1, lam0, gf)
        gr = torch.empty(case.rho.shape, dtype=torch.float64, device="cuda")
        gu = torch.empty(case.u.shape, dtype=torch.float64, device="cuda")
        nw = 0 if case.wall_u is None else len(case.wall_u)
        M.maclab_adjoint_finish(s.handle, lam0, s0, gr, gu, 0.0, gf.cpu().tolist(), nw)
        return gr.cpu().numpy(), gu.cpu().numpy(), gf.cpu().numpy()[:len(case.dims)]


def problem(lat, dims, periodic, walls):
    case = inputs.random_case(lat, dims, periodic, seed=101, u_amp=0.08, rho_amp=0.02, walls=walls,
                              force=(2e-4,) * len(dims))
    g = inputs.rng(102)
    return case, g.standard_normal(case.rho.shape), g.standard_normal(case.u.shape)


@pytest.mark.parametrize("lat,dims", [
    (D2, (4, 3)), (D2, (8, 5)), (D2, (64, 9)), (D2, (128, 13)), (D2, (132, 4)), (D2, (256, 7)), (D2, (512, 5)),
    (D3, (4, 5, 3)), (D3, (64, 7, 5)), (D3, (68, 6, 4)), (D3, (96, 5, 6)), (D3, (100, 9, 5)), (D3, (128, 11, 4))],
    ids=str)
@pytest.mark.parametrize("edges", ["periodic", "box", "mixed"])
def test_fp64_rows(torch, lat, dims, edges):
    d = len(dims)
    periodic = {"periodic": (1 << d) - 1, "box": 0, "mixed": 1}[edges]
    case, lr, lu = problem(lat, dims, periodic, "none" if edges == "periodic" else edges)
    want = reverse(torch, case, M.F64, M.KERNEL_REFERENCE, lr, lu)
    got = reverse(torch, case, M.F64, M.KERNEL_AUTO, lr, lu)
    for w, a in zip(want[:2], got[:2]):
        assert np.abs(w - a).max() <= 1e-12 * np.abs(w).max()
    assert np.allclose(want[2], got[2], rtol=1e-12, atol=1e-12 * np.abs(want[1]).max())


@pytest.mark.parametrize("lat,dims,precision", [
    (D2, (516, 5), M.F64), (D2, (17, 9), M.F64), (D2, (513, 4), M.F32), (D2, (1028, 4), M.F32),
    (D3, (5, 6, 4), M.F64), (D3, (97, 5, 4), M.F64), (D3, (132, 6, 5), M.F64), (D3, (256, 5, 3), M.F64),
    (D3, (129, 6, 5), M.F32), (D3, (300, 5, 6), M.F32), (D3, (516, 4, 3), M.F32)], ids=str)
@pytest.mark.parametrize("edges", ["periodic", "box"])
def test_widths_of_the_reference_kernels(torch, lat, dims, precision, edges):
    d = len(dims)
    case, lr, lu = problem(lat, dims, (1 << d) - 1 if edges == "periodic" else 0, "none" if edges == "periodic" else edges)
    wr, wu, wf = orc.adjoint_step(lat, case.rho, case.u, case.periodic, lr, lu, wall=case.wall_mask, force=case.force)
    gr, gu, gf = reverse(torch, case, precision, M.KERNEL_AUTO, lr, lu)
    tol = 1e-11 if precision == M.F64 else 2e-5
    fluid = np.ones(case.rho.shape, bool) if case.node_type is None else case.node_type == 0
    assert np.abs(gr - wr)[fluid].max() <= tol * np.abs(wr).max()
    assert np.abs(gu - wu)[:, fluid].max() <= tol * np.abs(wu).max()
    assert np.abs(gf - wf).max() <= (1e-12 if precision == M.F64 else 1e-6) * np.abs(wf).max() * np.sqrt(lu.size)
