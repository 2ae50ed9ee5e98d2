"""maclab_adjoint_step on raw states and adjoints that are aligned to one value only
(a view into a larger buffer): interleaved rows are read a quad or a pair at a time
only where every array allows it.  Against the same call on aligned arrays: the same
terms summed in another order (FP64 1e-12, FP32 2e-6 of the largest value)."""
import pytest

from paper_1901_02716_gb300 import inputs
from paper_1901_02716_gb300 import maclab as M

pytestmark = pytest.mark.gpu
D2, D3 = inputs.D2Q9, inputs.D3Q19


@pytest.mark.parametrize("lat,dims,periodic", [
    (D3, (64, 9, 7), 0b111), (D3, (24, 21, 9), 0b111), (D3, (520, 4, 3), 0b111), (D3, (65, 9, 7), 0b111),
    (D2, (64, 33), 0b11), (D2, (61, 9), 0b11)])
@pytest.mark.parametrize("precision", [M.F64, M.F32])
def test_arrays_aligned_to_one_value(lat, dims, periodic, precision):
    torch = pytest.importorskip("torch")
    kind, size, tol = (torch.float64, 8, 1e-12) if precision == M.F64 else (torch.float32, 4, 2e-6)
    case = inputs.random_case(lat, dims, periodic, seed=151, u_amp=0.08, rho_amp=0.02)
    with M.Solver.from_case(case, precision) as s:
        nb = s.state_bytes()
        buf = [torch.zeros(nb + 64, dtype=torch.uint8, device="cuda") for _ in range(4)]
        s0, s1, l1, l0 = (b[:nb] for b in buf)
        s.get_lattice_state(s0)
        s.step(1)
        s.get_lattice_state(s1)
        g = inputs.rng(152)
        l1.view(kind).copy_(torch.tensor(g.standard_normal(nb // size), dtype=kind))
        M.maclab_adjoint_step(s.handle, s0, s1, l1, l0, None)
        want = l0.view(kind).double()
        for moved in range(4):  # each array by itself off the boundary
            args = []
            for i, a in enumerate((s0, s1, l1, l0)):
                if i == moved:
                    b = torch.zeros(nb + 64, dtype=torch.uint8, device="cuda")[size:size + nb]
                    b.copy_(a)
                    a = b
                args.append(a)
            if moved != 3:
                args[3] = torch.zeros(nb + 64, dtype=torch.uint8, device="cuda")[:nb]
            M.maclab_adjoint_step(s.handle, *args, None)
            got = args[3].view(kind).double()
            assert (got - want).abs().max() <= tol * want.abs().max()
