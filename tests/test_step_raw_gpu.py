"""maclab_step_raw (steps between raw states, without copies) against
maclab_step between copies: the same bits, for every kernel that serves it, with
walls and a body force; the handle's own state is untouched where it must be."""
import numpy as np
import pytest

from paper_1901_02716_gb300 import inputs
from paper_1901_02716_gb300 import maclab as M

pytestmark = pytest.mark.gpu
D2, D3 = inputs.D2Q9, inputs.D3Q19


@pytest.mark.parametrize("lat,dims,periodic,walls,served", [
    (D2, (5, 4), 0b11, "none", True), (D2, (64, 40), 0b00, "mixed", True), (D2, (1024, 560), 0b10, "box", True),
    (D2, (37, 9), 0b00, "box", False), (D3, (7, 5, 6), 0b111, "none", True), (D3, (32, 24, 9), 0b101, "mixed", True),
    (D3, (160, 16, 6), 0b000, "box", True), (D3, (45, 40, 41), 0b000, "box", False)])
@pytest.mark.parametrize("precision", [M.F32, M.F64, M.BF16_STORE])
def test_steps_between_raw_states(lat, dims, periodic, walls, served, precision):
    torch = pytest.importorskip("torch")
    case = inputs.random_case(lat, dims, periodic, seed=33, u_amp=0.05, rho_amp=0.01, walls=walls,
                              force=tuple([1e-4] * len(dims)))
    a, b = M.Solver.from_case(case, precision), M.Solver.from_case(case, precision)

    def raw(s):
        t = torch.empty(s.state_bytes(), dtype=torch.uint8, device="cuda")
        s.get_lattice_state(t)
        return t

    want = [raw(a)]
    for _ in range(4):
        a.step(1)
        want.append(raw(a))
    got = [torch.full_like(want[0], 0x7b) for _ in range(4)]
    if not M.maclab_step_raw(b.handle, want[0], got[0]):
        assert not served or precision == M.F64  # FP64 has other padding rules
        return
    assert served or precision != M.F32
    assert torch.equal(got[0], want[1])
    assert M.maclab_step_raw(b.handle, got[0], got[1]) and torch.equal(got[1], want[2])
    assert torch.equal(raw(b), want[0])                      # own state as it was
    assert M.maclab_step_raw(b.handle, got[1]) and torch.equal(raw(b), want[3])
    b.step(1)
    assert torch.equal(raw(b), want[4])
    b.set_lattice_state(want[1])
    assert M.maclab_step_raw(b.handle, None, got[2]) and torch.equal(got[2], want[2])
    assert torch.equal(raw(b), want[1])
    assert M.maclab_step_raw(b.handle) and torch.equal(raw(b), want[2])
    assert not M.maclab_step_raw(b.handle, got[0].data_ptr() + 4, got[1])
    with pytest.raises(M.MacLABError):
        M.maclab_step_raw(b.handle, got[0], got[0])
    a.close(), b.close()


@pytest.mark.parametrize("lat,dims,periodic,walls", [
    (D2, (64, 33), 0b00, "mixed"), (D2, (37, 21), 0b00, "box"), (D3, (24, 16, 9), 0b111, "none")])
@pytest.mark.parametrize("steps,seg", [(1, 0), (2, 1), (7, 3), (9, 9)])
def test_rollout_states_do_not_depend_on_the_segments(lat, dims, periodic, walls, steps, seg):
    """The final state of a rollout is that of as many plain steps."""
    torch = pytest.importorskip("torch")
    from paper_1901_02716_gb300 import adjoint

    case = inputs.random_case(lat, dims, periodic, seed=34, u_amp=0.05, rho_amp=0.01, walls=walls)
    spec = adjoint.RolloutSpec(lat, dims, case.dx if hasattr(case, "dx") else 1.0, steps, periodic, case.node_type,
                               case.wall_rho, M.F32, checkpoint_every=seg)
    wu = None if case.wall_u is None else torch.tensor(np.asarray(case.wall_u), device="cuda")
    rho = torch.tensor(case.rho, device="cuda")
    u = torch.tensor(case.u, device="cuda")
    r1, u1 = adjoint.rollout(rho, u, wu, 1 / 6, spec)
    with M.Solver(lat, dims, spec.dx, 1 / 6, M.F32, periodic, case.node_type, case.wall_rho, case.wall_u) as s:
        s.set_state(rho, u)
        s.step(steps)
        r2, u2 = torch.empty_like(rho), torch.empty_like(u)
        s.get_state_into(r2, u2)
    assert torch.equal(r1, r2) and torch.equal(u1, u2)
