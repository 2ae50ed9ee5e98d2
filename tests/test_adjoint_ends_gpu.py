"""The ends of the reverse pass (maclab_adjoint_seed, maclab_adjoint_finish):
their unit maps and the sum lam_ut . ut against FP64 on the same arrays, over
row layouts, storage types, array types and the forms of the unit map
(rho0 a power of two or not), and with arrays that are not aligned to quads.

Bounds: a 32-bit result is the FP64 value rounded once, up to 2^-23 ulp about a
rounding boundary: |error| <= 2^-24 (1 + 2^-20) |value|.  The sum keeps the
rounding errors of at most 12 products and additions a unit: 2^-44 of the sum
of magnitudes."""
import numpy as np
import pytest

from paper_1901_02716_gb300 import inputs
from paper_1901_02716_gb300 import maclab as M

pytestmark = pytest.mark.gpu
D2, D3 = inputs.D2Q9, inputs.D3Q19


def _to_storage(a, nx):
    """Logical rows -> the order of the stored rows (interleaved halves where nx % 4 == 0)."""
    if nx % 4:
        return a
    out = np.empty_like(a)
    out[..., 0::2] = a[..., :nx // 2]
    out[..., 1::2] = a[..., nx // 2:]
    return out


@pytest.mark.parametrize("scale", [1.0, 1e-30])
@pytest.mark.parametrize("offset", [0, 4])
@pytest.mark.parametrize("dtype,precision,rho0", [
    ("float32", M.F32, 1.0), ("float32", M.F32, 0.25), ("float32", M.F32, 1.3), ("float64", M.F32, 1.0),
    ("float32", M.BF16_STORE, 1.0), ("float32", M.F64, 1.0), ("float64", M.F64, 1.0)])
@pytest.mark.parametrize("lat,dims,walls", [
    (D2, (4, 3), "none"), (D2, (37, 5), "box"), (D2, (68, 9), "box"), (D3, (8, 5, 3), "none"),
    (D3, (7, 5, 3), "none"), (D3, (24, 6, 7), "box"), (D3, (96, 40, 33), "none")])
def test_ends_of_the_reverse_pass(lat, dims, walls, dtype, precision, rho0, offset, scale):
    torch = pytest.importorskip("torch")
    d, nx = len(dims), dims[0]
    case = inputs.random_case(lat, dims, 0 if walls == "box" else (1 << d) - 1, seed=91, u_amp=0.08, rho_amp=0.02,
                              walls=walls)
    if offset and precision == M.F64:
        offset = 8
    with M.Solver(case.lattice, case.dims, 1.0, 1 / 6, precision, case.periodic, case.node_type, case.wall_rho,
                  case.wall_u, rho0=rho0) as s:
        e = s.params["e"]
        s.set_state(case.rho * rho0, case.u)
        raw = torch.empty(s.state_bytes(), dtype=torch.uint8, device="cuda")
        s.get_lattice_state(raw)
        kind = {M.F64: torch.float64, M.F32: torch.float32, M.BF16_STORE: torch.bfloat16}[precision]
        state = raw.view(kind).double().cpu().numpy().reshape((d + 1,) + case.rho.shape)
        g = inputs.rng(92)
        td = getattr(torch, dtype)
        g_rho = torch.tensor(g.standard_normal(case.rho.shape) * scale, dtype=td, device="cuda")
        g_u = torch.tensor(g.standard_normal(case.u.shape) * scale, dtype=td, device="cuda")
        lam_kind = torch.float64 if precision == M.F64 else torch.float32
        block = torch.zeros(s.adjoint_bytes() + 16, dtype=torch.uint8, device="cuda")
        lam = block[offset:offset + s.adjoint_bytes()]
        dot = M.maclab_adjoint_seed(s.handle, g_rho, g_u, raw, lam)
        got = lam.clone().view(lam_kind).double().cpu().numpy().reshape((d + 1,) + case.rho.shape)
        want = np.concatenate([rho0 * g_rho.double().cpu().numpy()[None], e * g_u.double().cpu().numpy()])
        ulp = 2.0 ** -24 * (1 + 2.0 ** -20) if lam_kind == torch.float32 else 2.0 ** -52
        sw = _to_storage(want, nx)
        assert (np.abs(got - sw) <= ulp * np.abs(sw) + 1e-45).all()
        terms = sw[1:] * state[1:]
        assert abs(dot - terms.sum()) <= 2.0 ** -44 * np.abs(terms).sum()

        gr = torch.empty_like(g_rho)
        gu = torch.empty_like(g_u)
        nw = 0 if case.wall_u is None else len(case.wall_u)
        res = M.maclab_adjoint_finish(s.handle, lam, raw, gr, gu, 0.0, [0.0] * 3, nw)
        out_ulp = 2.0 ** -24 * (1 + 2.0 ** -20) if dtype == "float32" else 2.0 ** -51
        fluid = np.ones(case.rho.shape, bool) if case.node_type is None else np.asarray(case.node_type) == 0
        exact = np.concatenate([got[:1] / rho0, got[1:] / e])
        back = np.concatenate([_to_storage(gr.double().cpu().numpy()[None], nx),
                               _to_storage(gu.double().cpu().numpy(), nx)])
        ref = np.where(_to_storage(fluid[None], nx), exact, 0.0)
        assert (np.abs(back - ref) <= out_ulp * np.abs(ref) + 1e-45).all()
        terms = got[1:] * state[1:]
        assert abs(-res["e"] * e - terms.sum()) <= 2.0 ** -44 * np.abs(terms).sum() + 2.0 ** -50 * abs(terms.sum())
        for k in range(nw):
            at = _to_storage((np.asarray(case.node_type) == k + 1)[None], nx)[0]
            for f in range(d + 1):
                t = exact[f][at]
                assert abs(res["wall"][k][f] - t.sum()) <= 2.0 ** -44 * np.abs(t).sum() + 1e-300
