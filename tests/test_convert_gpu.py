"""The unit maps of maclab_set_state / maclab_get_state on 32-bit arrays against
their definition in FP64: stored = rho / rho0 - 1 and u / e, physical = rho0 (1 +
stored) and e * stored, rounded once.

The FP32 forms differ from that by at most one unit in the last place of the
rounded result (a value within 2^-23 ulp of a rounding boundary may go to the
other side); where FP64 is used (rho0 not a power of two) the same bound holds.
Sizes: interleaved and natural rows, one quad a row, ragged counts; user tensors
at an offset of one value take the unaligned path.
"""
import numpy as np
import pytest

from paper_1901_02716_gb300 import inputs
from paper_1901_02716_gb300 import maclab as M

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1901_02716_gb300 import _build
    _build.build()


def _ulps(got, want):
    """Largest difference in units of the last place of float32."""
    return float(np.max(np.abs(got.astype(np.float64) - want) / np.spacing(np.abs(want).astype(np.float32))))


@pytest.mark.parametrize("lat,dims", [(M.D2Q9, (4, 3)), (M.D2Q9, (37, 11)), (M.D2Q9, (260, 9)),
                                      (M.D3Q19, (12, 5, 7)), (M.D3Q19, (31, 6, 5))])
@pytest.mark.parametrize("rho0,dx,nu", [(1.0, 1.0, 1 / 6), (2.0, 0.0025, 0.0004), (1.3, 0.157, 0.0314)])
@pytest.mark.parametrize("offset", [0, 1])
def test_unit_maps_round_once(lat, dims, rho0, dx, nu, offset):
    torch = pytest.importorskip("torch")
    d = len(dims)
    grid = tuple(reversed(dims))
    g = inputs.rng(91)
    rho = (rho0 * (1 + 0.01 * g.uniform(-1, 1, size=grid))).astype(np.float32)
    s = M.Solver(lat, dims, dx, nu, M.F32, (1 << d) - 1, rho0=rho0)
    e = s.params["e"]
    u = (e * 0.05 * g.uniform(-1, 1, size=(d,) + grid)).astype(np.float32)

    def device(a):
        t = torch.zeros(a.size + offset, dtype=torch.float32, device="cuda")[offset:].view(a.shape)
        t.copy_(torch.from_numpy(a))
        return t

    s.set_state(device(rho), device(u))
    raw = s.get_lattice_state().view(np.float32).reshape((d + 1,) + grid).copy()
    if dims[0] % 4 == 0:  # back to logical order
        h = dims[0] // 2
        raw = raw.reshape(raw.shape[:-1] + (h, 2)).swapaxes(-1, -2).reshape(raw.shape)
    want_r, want_u = rho.astype(np.float64) * (1 / rho0) - 1.0, u.astype(np.float64) * (1 / e)
    assert _ulps(raw[0], want_r) <= 1.0 and _ulps(raw[1:], want_u) <= 1.0
    rho_t, u_t = device(np.zeros_like(rho)), device(np.zeros_like(u))
    s.get_state_into(rho_t, u_t)
    assert _ulps(rho_t.cpu().numpy(), rho0 * (1.0 + raw[0].astype(np.float64))) <= 1.0
    assert _ulps(u_t.cpu().numpy(), e * raw[1:].astype(np.float64)) <= 1.0
    s.close()


def test_infinities_and_nan_pass_through():
    """Non-finite inputs stay what they were (the residual of the split product is NaN there)."""
    rho = np.ones((3, 8), dtype=np.float32)
    u = np.zeros((2, 3, 8), dtype=np.float32)
    u[0, 1, 2], u[1, 1, 3], rho[0, 0] = np.inf, -np.inf, np.nan
    s = M.Solver(M.D2Q9, (8, 3), 0.1, 0.01, M.F32, 0b11)
    s.set_state(rho, u)
    r, v = s.get_state(np.float32)
    assert np.isnan(r[0, 0]) and v[0, 1, 2] == np.inf and v[1, 1, 3] == -np.inf
    assert np.isfinite(np.delete(r.reshape(-1), 0)).all() and np.isfinite(v).sum() == v.size - 2
    s.close()
