"""Choosing kernels by hand, by tuning and by tile: what each call leaves in place."""
import pytest

from paper_1901_02716_gb300 import inputs
from paper_1901_02716_gb300 import maclab as M

pytestmark = pytest.mark.gpu
D2, D3 = inputs.D2Q9, inputs.D3Q19


def _reverse(torch, s):
    """One reverse step and viscosity term on fixed arrays."""
    g = torch.Generator(device="cuda").manual_seed(7)
    s0, s1, lam = (0.02 * torch.randn(s.state_bytes() // 4, generator=g, device="cuda") for _ in range(3))
    out = torch.empty_like(lam)
    acc = torch.zeros(1, dtype=torch.float64, device="cuda")
    M.maclab_adjoint_step(s.handle, s0, s1, lam, out, None)
    M.maclab_adjoint_nu_term(s.handle, s0, lam, acc, s1)
    return out, acc


@pytest.mark.parametrize("lat,dims", [(D3, (64, 16, 12)), (D2, (128, 40))])
def test_reverse_step_follows_a_kernel_that_tuning_replaced(lat, dims, monkeypatch):
    torch = pytest.importorskip("torch")
    monkeypatch.delenv("MACLAB_TUNE_CACHE", raising=False)
    d = len(dims)
    got = {}
    for how in ("library", "reference", "reference, then tuned"):
        with M.Solver(lat, dims, 1.0, 1.0 / 6.0, M.F32, (1 << d) - 1) as s:
            if how != "library":
                s.set_kernel(M.KERNEL_REFERENCE)
            if how.endswith("tuned"):
                s.tune()
                assert s.kernel_info()["kernel"] != M.KERNEL_REFERENCE
            got[how] = _reverse(torch, s)
    assert torch.equal(got["library"][0], got["reference, then tuned"][0])
    assert not torch.equal(got["library"][0], got["reference"][0])
    scale = float(got["library"][1].abs())
    assert float((got["library"][1] - got["reference, then tuned"][1]).abs()) <= 1e-12 * scale


@pytest.mark.parametrize("tile", [(3, 0), (0, 16), (2, 8), (1, 4)])
def test_segment_tiles_of_a_grid_the_block_kernel_serves(tile):
    """A tile that only the segment kernel has (rows per item, the persistent form) selects it on
    the larger grids of the block kernel's default; the bits are those of the default."""
    case = inputs.random_case(D2, (600, 520), 0, seed=191, u_amp=0.08, rho_amp=0.02, walls="box")
    out = []
    for t in (None, tile):
        with M.Solver.from_case(case, M.F32) as s:
            if t:
                s.set_tile(*t)
                assert s.kernel_info()["kernel"] == M.KERNEL_SEGMENT
            s.step(11)
            out.append(s.get_lattice_state())
    assert (out[0] == out[1]).all()


def test_tiles_that_stay_refused():
    case = inputs.random_case(D2, (64, 40), 0, seed=192, walls="box")
    with M.Solver.from_case(case, M.F32) as s:  # the block kernel's own range
        with pytest.raises(M.MacLABError):
            s.set_tile(3, 0)
    case = inputs.random_case(D2, (600, 520), 0, seed=193, walls="box")
    with M.Solver.from_case(case, M.F32) as s:
        s.set_kernel(M.KERNEL_BLOCK)
        with pytest.raises(M.MacLABError):
            s.set_tile(3, 0)
