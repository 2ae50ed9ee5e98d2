"""Diagnostics of widths that are not a multiple of 4 cost what those of the next multiple do, or
less (device time, best of seven), and padded FP64 rows give FP64 sums of their fluid nodes."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_1901_02716_gb300 import inputs
from paper_1901_02716_gb300 import maclab as M

pytestmark = pytest.mark.gpu
D2 = inputs.D2Q9


def _us(torch, s):
    out = torch.zeros(9, dtype=torch.float64, device="cuda")
    best = 1e9
    for _ in range(7):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        for _ in range(50):
            M.maclab_diagnostics_device(s.handle, out)
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) * 20)
    return best


@pytest.mark.parametrize("n", [61, 401])
def test_padded_fp64_rows_cost_no_more(n):
    """Node by node: 0.8 (61^2) and 0.7 (401^2) of the row form that the next width takes; bar 0.9."""
    torch = pytest.importorskip("torch")
    us = []
    for m in (n, n + 3):
        with M.Solver.from_case(inputs.cavity2d(m), M.F64) as s:
            s.step(3)
            us.append(_us(torch, s))
    assert us[0] <= 0.9 * us[1], us


@pytest.mark.parametrize("dims,walls", [((61, 40), "box"), ((37, 23), "mixed"), ((402, 30), "box"), ((19, 33), "box")])
def test_padded_fp64_sums(dims, walls):
    case = inputs.random_case(D2, dims, 0, seed=241, u_amp=0.08, rho_amp=0.02, walls=walls)
    with M.Solver.from_case(case, M.F64) as s:
        s.step(4)
        d = s.diagnostics()
        r, u = s.get_state()
    ref = orc.diagnostics(r, u, fluid=case.node_type == 0)
    assert d["mass"] == pytest.approx(ref["mass"], rel=1e-13)
    assert d["kinetic"] == pytest.approx(ref["kinetic"], rel=1e-12)
    largest = np.sqrt((u ** 2).sum(axis=0)[case.node_type == 0].max())
    assert d["max_u_lattice"] == pytest.approx(largest, rel=1e-14)
