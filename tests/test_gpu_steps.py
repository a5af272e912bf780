"""Small boxes on the work list take several steps in one launch (one block keeps its tiles, counters order the
jobs): equal bit for bit to the two-pass step for every share of tiles per block, however the steps are cut into
calls and checks, and a launch whose counters are not its own says so."""

import numpy as np
import pytest

from gpu_helpers import coexistence, lattice, physics

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1805_08643_gb300 import _build

    _build.build()


def _box(grid, op, mode, eos="cs", stream=None):
    if eos == "exp":
        phys, (rl, rv) = physics(eos="exp", G=-10.0 / 3.0), (2.78, 0.37)
    else:
        phys, (rl, rv) = physics(sigma=0.105), coexistence(0.8)
    lat = lattice(grid, op, "f32", phys, stream=stream)
    lat.set_tuning(mode)
    lat.init_droplet(tuple(0.4 * n for n in grid), 0.3 * min(grid), 3.0, rl, rv)
    return lat


def _equal(a, b):
    return all(np.array_equal(x, y) for x, y in zip(a, b))


# tiles: 1, 2, 5, 27; 1024 and 1088 (one and two per block of a full GB300 grid); 3906, 4292; and 9 x 5 x 4 past 512
@pytest.mark.parametrize("grid", [(4, 3, 3), (6, 5, 7), (16, 9, 5), (32, 24, 9), (64, 64, 64), (64, 64, 68),
                                  (100, 100, 100), (102, 104, 104), (500, 9, 5), (514, 9, 5)])
@pytest.mark.parametrize("op", ["nonorth", "orth", "nonorth_d3q15"])
def test_steps_equal_two_pass_bit_for_bit(grid, op):
    a, b = _box(grid, op, False), _box(grid, op, "queue")
    a.step(21)
    b.step(21)
    assert a.check() == 0 and b.check() == 0 and b.steps == 21
    ra, rb = a.moments(), b.moments()
    fa, fb = a.populations(), b.populations()
    a.close()
    b.close()
    assert _equal(ra, rb) and np.array_equal(fa, fb)


@pytest.mark.parametrize("eos, arith", [("cs", "f32x2"), ("exp", "f64"), ("exp", "f32x2")])
def test_steps_of_the_other_equations_of_state(eos, arith):
    out = []
    for mode in (False, "queue"):
        lat = _box((40, 24, 20), "nonorth", mode, eos)
        lat.set_eos_arith(arith)
        lat.step(30)
        assert lat.check() == 0
        out.append(lat.moments())
        lat.close()
    assert _equal(*out)


def test_any_cut_into_calls_checks_and_modes():
    """600 steps (three launches) against calls of 1, 2, 3, ... with reads between them, a check interval that cuts
    launches short, per-launch timing, and other step kinds in between."""
    grid = (48, 20, 12)
    a = _box(grid, "nonorth", "queue")
    a.step(600)
    ref = a.moments()
    a.close()
    b = _box(grid, "nonorth", "queue")
    b.set_check_interval(7)
    done = 0
    for k, n in enumerate([1, 2, 3, 255, 14]):
        b.step(n)
        done += n
        b.diag() if k % 2 else b.moments()
    b.set_check_interval(0)
    b.set_tuning(False)
    b.step(5)
    b.set_tuning("lagged")
    b.step(3)
    b.set_tuning("queue")
    b.set_profiling(True)
    b.step(4)
    times = b.kernel_times()
    assert times["fused_launches"] == 4
    b.set_profiling(False)
    b.step(600 - done - 12)
    assert b.steps == 600 and b.check() == 0
    got = b.moments()
    b.close()
    assert _equal(ref, got)


def test_a_replayed_launch_reports_its_counters():
    import torch

    from paper_1805_08643_gb300.lbm import ERR_TIMEOUT

    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        lat = _box((32, 16, 12), "nonorth", "queue", stream=s)
        lat.step(2)
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        g.capture_begin()
        lat.step(2)
        g.capture_end()
        g.replay()  # the launch the capture stands for
        s.synchronize()
        assert lat.check() == 0
        g.replay()  # its counters have moved on
        s.synchronize()
        assert lat.check() == ERR_TIMEOUT
        lat.close()
