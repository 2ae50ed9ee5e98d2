"""X axes whose width is not a multiple of 4 (stored in padded rows) and row
counts that no tile divides (a last tile moved up), against the oracle, and the
calls that show the raw state: its layout has no padding.

The bars are those of test_parity_gpu (the same arithmetic on other rows).
"""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_1901_02716_gb300 import inputs
from paper_1901_02716_gb300 import maclab as M
from test_parity_gpu import assert_parity, run_both

pytestmark = pytest.mark.gpu

D2, D3 = inputs.D2Q9, inputs.D3Q19


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1901_02716_gb300 import _build
    _build.build()


# widths with one, two and three padding positions, the narrowest padded one,
# box and mask walls, every kernel the library picks for the widths and types (3D:
# from the node counts on where rows are padded)
PADDED = [
    (D2, (17, 13), 0b00, "box"), (D2, (18, 9), 0b10, "box"), (D2, (23, 40), 0b00, "mixed"),
    (D2, (401, 37), 0b00, "box"), (D2, (1026, 1030), 0b10, "box"),
    (D3, (17, 49, 61), 0b110, "box"), (D3, (30, 40, 42), 0b000, "mixed"), (D3, (63, 16, 50), 0b100, "box"),
    (D3, (65, 29, 27), 0b000, "box"), (D3, (126, 20, 20), 0b010, "box"), (D3, (127, 21, 19), 0b000, "mixed"),
    (D3, (133, 18, 21), 0b010, "box"), (D3, (251, 17, 12), 0b000, "box"), (D3, (257, 14, 14), 0b100, "mixed"),
    (D3, (511, 10, 10), 0b000, "box"),
]
# periodic x: two to five padding positions, which hold the periodic images
WRAPPED = [
    (D3, (17, 96, 92), 0b111, "none"), (D3, (18, 92, 91), 0b001, "box"), (D3, (19, 88, 90), 0b101, "mixed"),
    (D3, (33, 69, 66), 0b111, "none"), (D3, (62, 48, 51), 0b011, "box"), (D3, (95, 42, 38), 0b111, "mixed"),
    (D3, (126, 40, 30), 0b111, "none"), (D3, (127, 33, 36), 0b011, "box"), (D3, (251, 25, 24), 0b111, "none"),
    (D3, (258, 24, 25), 0b001, "mixed"), (D3, (511, 18, 17), 0b111, "none"),
]
RAGGED = [
    (D3, (32, 13, 6), 0b111, "none"), (D3, (64, 11, 5), 0b000, "box"), (D3, (128, 10, 7), 0b010, "box"),
    (D3, (96, 5, 6), 0b101, "mixed"), (D3, (256, 9, 5), 0b111, "none"), (D3, (200, 6, 5), 0b000, "box"),
    (D3, (500, 7, 5), 0b010, "mixed"),
]


@pytest.mark.parametrize("lat,dims,periodic,walls", PADDED + WRAPPED + RAGGED)
@pytest.mark.parametrize("precision", [M.F64, M.F32, M.BF16_STORE])
def test_matches_oracle(lat, dims, periodic, walls, precision):
    case = inputs.random_case(lat, dims, periodic, seed=131, u_amp=0.08, rho_amp=0.02, walls=walls,
                              force=tuple([1e-4] * len(dims)))
    assert_parity(*run_both(case, precision, 3 if dims[0] > 1000 else 11), precision)


@pytest.mark.parametrize("lat,dims,periodic,walls", [PADDED[2], PADDED[3], PADDED[6], PADDED[12], WRAPPED[1], WRAPPED[5], WRAPPED[8]])
@pytest.mark.parametrize("precision", [M.F64, M.F32, M.F16_STORE])
def test_raw_state_has_no_padding(lat, dims, periodic, walls, precision):
    """The raw state is (d + 1) * N values in natural order; a run resumed from it, on the host or the
    device, repeats the bits; planes are parts of it; wall nodes keep their values."""
    torch = pytest.importorskip("torch")
    case = inputs.random_case(lat, dims, periodic, seed=132, u_amp=0.06, rho_amp=0.02, walls=walls)
    d = len(dims)
    s = M.Solver.from_case(case, precision)
    np_t = M.STORAGE_NP[precision]
    assert s.state_bytes() == (d + 1) * case.n_nodes * np.dtype(np_t).itemsize
    s.step(5)
    snap = s.get_lattice_state().copy()
    fields = snap.view(np_t).reshape((d + 1,) + case.grid)
    r, u = s.get_state()
    assert np.array_equal(fields[0].astype(np.float64) + 1.0, r)
    assert np.array_equal(fields[1:].astype(np.float64), u)
    wall = case.wall_mask
    if wall is not None:
        assert np.array_equal(fields[1:, wall], case.u[:, wall].astype(np_t))
    dev = torch.empty(s.state_bytes() + 1, dtype=torch.uint8, device="cuda")
    for t in (dev[:-1], dev[1:]):  # aligned, and a byte off
        s.get_lattice_state(t)
        assert np.array_equal(t.cpu().numpy(), snap)
    planes = dims[-1]
    part = np.empty((d + 1, 2) + case.grid[1:], dtype=np_t)
    M.maclab_get_planes(s.handle, planes - 3, 2, part)
    assert np.array_equal(part, fields[:, planes - 3:planes - 1])
    s.step(6)
    want = s.get_lattice_state().copy()
    for state in (snap, dev[1:]):
        s.set_lattice_state(state)
        s.step(6)
        assert np.array_equal(s.get_lattice_state(), want)
    part_dev = torch.from_numpy(part.view(np.uint8)).cuda()
    for state in (part, part_dev):
        M.maclab_set_planes(s.handle, planes - 3, 2, state)
        got = s.get_lattice_state().view(np_t).reshape(fields.shape)
        assert np.array_equal(got[:, planes - 3:planes - 1], part)
        assert np.array_equal(got[:, :planes - 3], want.view(np_t).reshape(fields.shape)[:, :planes - 3])
    s.close()


@pytest.mark.parametrize("lat,dims,periodic,walls", [PADDED[1], PADDED[2], PADDED[12], RAGGED[3], WRAPPED[2], WRAPPED[4]])
def test_diagnostics_and_wall_values(lat, dims, periodic, walls):
    """Diagnostics skip the padding; per-node wall values reach every wall node."""
    case = inputs.random_case(lat, dims, periodic, seed=133, u_amp=0.06, rho_amp=0.02, walls=walls)
    g = inputs.rng(134)
    wall = case.wall_mask
    rho_w = np.where(wall, 1 + 0.01 * g.uniform(-1, 1, size=case.grid), 5.0)
    u_w = np.where(wall, 0.05 * g.uniform(-1, 1, size=case.u.shape), 5.0)
    rho, u = np.where(wall, rho_w, case.rho), np.where(wall, u_w, case.u)
    s = M.Solver.from_case(case, M.F64)
    s.set_wall_state(rho_w, u_w)
    s.step(7)
    r_g, u_g = s.get_state()
    r_o, u_o = orc.step(lat, rho, u, periodic, wall=wall, nsteps=7)
    assert_parity(r_g, u_g, r_o, u_o, M.F64)
    diag = s.diagnostics()
    assert diag["mass"] == pytest.approx(r_o[~wall].sum(), rel=1e-12)
    assert diag["kinetic"] == pytest.approx(0.5 * (r_o * (u_o ** 2).sum(0))[~wall].sum(), rel=1e-11)
    assert diag["max_u_lattice"] == pytest.approx(np.sqrt((u_o ** 2).sum(0)[~wall].max()), rel=1e-11)
    assert diag["nonfinite"] == 0
    s.close()


@pytest.mark.parametrize("depth", [1, 2, 3])
@pytest.mark.parametrize("precision", [M.F32, M.F64])
def test_batch_of_odd_widths(depth, precision):
    """Closed members of any width share one launch and give the bits of standalone runs."""
    cases = [inputs.cavity2d(65, lid=0.08), inputs.cavity2d(50, lid=0.05, nx=39), inputs.cavity2d(96, lid=0.1),
             inputs.random_case(D2, (130, 41), 0b10, seed=135, u_amp=0.05, walls="mixed")]
    b = M.Batch.from_cases(cases, precision)
    b.set_depth(depth)
    assert b.info()["launches_per_step"] == 1 and b.info()["nodes"] == sum(c.n_nodes for c in cases)
    b.step(13)
    b.sync()
    for m, case in zip(b.members, cases):
        s = M.Solver.from_case(case, precision)
        s.step(13)
        assert np.array_equal(m.get_lattice_state(), s.get_lattice_state())
        s.close()
    b.close()


def test_tuned_padded_domain_keeps_the_result():
    case = inputs.random_case(D3, (70, 27, 29), 0b000, seed=136, u_amp=0.06, rho_amp=0.02, walls="box")
    s = M.Solver.from_case(case, M.F32)
    s.tune()
    s.step(9)
    r_g, u_g = s.get_state()
    s.close()
    r_o, u_o = orc.step(D3, case.rho, case.u, case.periodic, wall=case.wall_mask, nsteps=9)
    assert_parity(r_g, u_g, r_o, u_o, M.F32)


def test_refused_choices_stay_refused():
    """By hand, kernels take the widths and row counts they always took."""
    for case, kernels in ((inputs.cavity2d(65, lid=0.05), (M.KERNEL_TILED, M.KERNEL_SEGMENT, M.KERNEL_BLOCK)),
                          (inputs.random_case(D3, (32, 13, 6), 0b111, seed=137), (M.KERNEL_ROWS2, M.KERNEL_FOLDED))):
        s = M.Solver.from_case(case, M.F32)
        for kernel in kernels:
            with pytest.raises(M.MacLABError) as ei:
                s.set_kernel(kernel)
            assert ei.value.status == M.ERR_UNSUPPORTED
        s.close()


@pytest.mark.parametrize("dims,periodic,walls", [((32, 13, 6), 0b111, "none"), ((96, 9, 7), 0b101, "box")])
def test_viscosity_term_of_ragged_rows(dims, periodic, walls):
    """Row counts that no tile divides: the tiled viscosity-term pass against the per-node one (each
    fluid row counted once; both sum FP32 terms, so they agree to the rounding of the terms)."""
    torch = pytest.importorskip("torch")
    case = inputs.random_case(D3, dims, periodic, seed=138, u_amp=0.06, rho_amp=0.02, walls=walls)
    s = M.Solver.from_case(case, M.F32)
    states = []
    for _ in range(2):
        buf = torch.empty(s.state_bytes(), dtype=torch.uint8, device="cuda")
        s.get_lattice_state(buf)
        states.append(buf)
        s.step(1)
    lam = torch.randn(4 * case.n_nodes, device="cuda", generator=torch.Generator("cuda").manual_seed(139))
    sums = []
    for after in (states[1], None):  # None: the per-node pass
        acc = torch.zeros(1, dtype=torch.float64, device="cuda")
        M.maclab_adjoint_nu_term(s.handle, states[0], lam, acc, after)
        sums.append(float(acc.item()))
    s.close()
    terms = 4 * case.n_nodes * 0.1  # no term's magnitude exceeds |lam| * 0.1 here
    assert abs(sums[0] - sums[1]) <= 16 * 2.0 ** -24 * terms
