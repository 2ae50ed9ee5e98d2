"""Runs of a few steps, advanced one call at a time (a monitor, a coupled solver): the bits of
a long run, and no more time than the one-step launches that the segment kernel has."""
import numpy as np
import pytest

from paper_1901_02716_gb300 import inputs
from paper_1901_02716_gb300 import maclab as M

pytestmark = pytest.mark.gpu
D2 = inputs.D2Q9


@pytest.mark.parametrize("dims,walls", [((600, 520), "box"), ((1024, 530), "mixed"), ((517, 600), "box"),
                                        ((1080, 1000), "none")])
@pytest.mark.parametrize("precision", [M.F32, M.F64])
def test_single_steps_give_the_bits_of_a_run(dims, walls, precision):
    case = inputs.random_case(D2, dims, 0b11 if walls == "none" else 0, seed=201, u_amp=0.08, rho_amp=0.02, walls=walls)
    out = []
    for parts in ([9], [1] * 9, [2, 3, 4], [5, 1, 3]):
        with M.Solver.from_case(case, precision) as s:
            for n in parts:
                s.step(n)
            out.append(s.get_lattice_state())
    for o in out[1:]:
        assert np.array_equal(o, out[0])


def test_single_steps_of_a_batch_give_the_bits_of_a_run():
    cases = [inputs.random_case(D2, (n, n + 8), 0, seed=202 + n, u_amp=0.08, rho_amp=0.02, walls="box")
             for n in (64, 37, 256, 130)]
    out = []
    for parts in ([9], [1] * 9, [2, 7]):
        b = M.Batch.from_cases(cases, M.F32)
        b.set_depth(2)
        for n in parts:
            b.step(n)
        out.append([m.get_lattice_state() for m in b.members])
        b.close()
    for o in out[1:]:
        assert all(np.array_equal(x, y) for x, y in zip(o, out[0]))


@pytest.mark.parametrize("n", [1000, 1024])
def test_a_single_step_costs_one_step(n):
    """The default's single steps against one-step launches of the segment kernel in four-row items,
    which these grids had for them (the block kernel's one-step launch and the two-step work
    list take 1.55 and 1.28 of that): best of five, bar 1.15."""
    torch = pytest.importorskip("torch")
    us = {}
    for name in ("default", "one step"):
        with M.Solver.from_case(inputs.cavity2d(n), M.F32) as s:
            if name == "one step":
                s.set_kernel(M.KERNEL_SEGMENT)
                s.set_tile(1, 4)
            best = 1e9
            for _ in range(5):
                for _ in range(20):
                    s.step(1)
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                torch.cuda.synchronize()
                a.record()
                for _ in range(200):
                    s.step(1)
                b.record()
                torch.cuda.synchronize()
                best = min(best, a.elapsed_time(b) / 200 * 1e3)
            us[name] = best
    assert us["default"] <= 1.15 * us["one step"], us


@pytest.mark.parametrize("dims", [(33, 1000), (128, 128), (97, 340)])
def test_short_fp64_runs_cost_what_long_ones_do(dims):
    """Runs of ten steps mix launches of four, two and one; best of five, bar 1.3 of the time a
    step takes in runs of fifty (1.4 to 1.8 where every change of instance drains the device)."""
    torch = pytest.importorskip("torch")
    us = {}
    case = inputs.random_case(D2, dims, 0, seed=203, u_amp=0.05, rho_amp=0.01, walls="box")
    with M.Solver.from_case(case, M.F64) as s:
        for n in (10, 50):
            best = 1e9
            for _ in range(5):
                s.step(n)
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                torch.cuda.synchronize()
                a.record()
                for _ in range(20):
                    s.step(n)
                b.record()
                torch.cuda.synchronize()
                best = min(best, a.elapsed_time(b) / (20 * n) * 1e3)
            us[n] = best
    assert us[10] <= 1.3 * us[50], us
