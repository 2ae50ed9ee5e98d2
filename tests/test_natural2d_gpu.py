"""The D2Q9 block kernel on a periodic x axis whose width is not a multiple of 4
(natural rows), and the FP64 tiles' row counts, against the oracle and, bit for
bit, runs of single steps (a run of n steps takes several per launch).

Bars as in test_parity_gpu.
"""
import numpy as np
import pytest

from paper_1901_02716_gb300 import inputs
from paper_1901_02716_gb300 import maclab as M
from test_parity_gpu import assert_parity, run_both

pytestmark = pytest.mark.gpu

D2 = inputs.D2Q9


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1901_02716_gb300 import _build
    _build.build()


# odd widths and widths of 4 k + 2 around the tile's 32 pairs, the narrowest
# served, fewer rows than the halo; and interleaved rows of at most and of more
# than 32 pairs for the FP64 tiles
CASES = [((33, 40), 0b11, "none"), ((63, 17), 0b01, "box"), ((65, 64), 0b11, "none"), ((66, 3), 0b11, "none"),
         ((127, 70), 0b01, "mixed"), ((401, 33), 0b11, "mixed"), ((530, 401), 0b01, "box"),
         ((64, 64), 0b11, "none"), ((60, 31), 0b00, "box"), ((68, 19), 0b01, "mixed"), ((8, 130), 0b10, "box")]


@pytest.mark.parametrize("dims,periodic,walls", CASES)
@pytest.mark.parametrize("precision", [M.F64, M.F32])
@pytest.mark.parametrize("steps", [1, 19])
def test_matches_oracle_and_single_steps(dims, periodic, walls, precision, steps):
    case = inputs.random_case(D2, dims, periodic, seed=141, u_amp=0.08, rho_amp=0.02, walls=walls,
                              force=(1e-4, -2e-4))
    s = M.Solver.from_case(case, precision)
    assert s.kernel_info()["kernel"] == M.KERNEL_BLOCK
    s.close()
    assert_parity(*run_both(case, precision, steps), precision)
    runs = []
    for calls in ([steps], [1] * steps):
        s = M.Solver.from_case(case, precision)
        for n in calls:
            s.step(n)
        runs.append((s.get_lattice_state().copy(), s.diagnostics()["residual"]))
        s.close()
    assert np.array_equal(runs[0][0], runs[1][0]) and runs[0][1] == runs[1][1]


def test_batch_member_of_natural_rows():
    """A batch that cannot run in one launch steps such a member with the same kernel, one step at a time."""
    cases = [inputs.random_case(D2, (65, 40), 0b11, seed=142, u_amp=0.05), inputs.cavity2d(64, lid=0.05)]
    b = M.Batch.from_cases(cases, M.F32)
    b.step(11)
    for m, case in zip(b.members, cases):
        s = M.Solver.from_case(case, M.F32)
        s.step(11)
        assert np.array_equal(m.get_lattice_state(), s.get_lattice_state())
        s.close()
    b.close()


def test_choices_by_hand_stay_refused():
    s = M.Solver.from_case(inputs.random_case(D2, (65, 40), 0b11, seed=143), M.F32)
    for call in (lambda: s.set_kernel(M.KERNEL_BLOCK), lambda: s.set_tile(8, 0)):
        with pytest.raises(M.MacLABError) as ei:
            call()
        assert ei.value.status == M.ERR_UNSUPPORTED
    s.close()
