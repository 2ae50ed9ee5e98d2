"""The sums lam_u . u of maclab_adjoint_seed and maclab_adjoint_finish on 32-bit arrays:
as exact as FP64 additions of the same products.  One storage quad (or node) at a time, so that
nothing averages out: the sum of its 2 to 12 products is rounded once to FP64, the FP64
steps that follow add zeros (2^-52 of the magnitudes), e = 6 nu / dx = 1."""
from fractions import Fraction

import numpy as np
import pytest

from paper_1901_02716_gb300 import inputs
from paper_1901_02716_gb300 import maclab as M

pytestmark = pytest.mark.gpu
D2, D3 = inputs.D2Q9, inputs.D3Q19


@pytest.mark.parametrize("lat,dims", [(D2, (4, 1)), (D3, (4, 1, 1)), (D2, (1, 1)), (D3, (1, 1, 1))])
def test_sums_of_one_unit(lat, dims):
    torch = pytest.importorskip("torch")
    d, n = len(dims), int(np.prod(dims))
    g = inputs.rng(181)
    f32 = lambda shape, scale: (scale * g.standard_normal(shape)).astype(np.float32)
    with M.Solver(lat, dims, 1.0, 1.0 / 6.0, M.F32, (1 << d) - 1) as s:
        assert s.params["e"] == 1.0
        lam = torch.empty(s.adjoint_bytes(), dtype=torch.uint8, device="cuda")
        grid = tuple(reversed(dims))
        for _ in range(150):
            state, gu = f32((d + 1, n), 0.1), f32((d, n), 1.0)
            raw = torch.tensor(state, device="cuda")
            if n == 4:  # user arrays are in logical order, the raw state interleaved
                gu_l = gu[:, [0, 2, 1, 3]]
            else:
                gu_l = gu
            tu = torch.tensor(np.ascontiguousarray(gu_l), device="cuda").view((d,) + grid)
            dot = M.maclab_adjoint_seed(s.handle, None, tu, raw, lam)
            terms = [Fraction(float(a)) * Fraction(float(b)) for a, b in zip(gu.ravel(), state[1:].ravel())]
            exact, size = sum(terms), float(sum(abs(t) for t in terms))
            assert abs(float(Fraction(dot) - exact)) <= 2.0 ** -52 * size
            res = M.maclab_adjoint_finish(s.handle, lam, raw, torch.empty(grid, device="cuda"), torch.empty_like(tu), 0.0,
                                          [0.0] * 3, 0)
            assert abs(float(Fraction(-res["e"]) - exact)) <= 2.0 ** -52 * size
