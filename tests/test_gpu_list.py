"""The work list proper (queue_kernel): boxes that the several-steps kernel leaves to it, being past five tiles per
resident block, wider than its tiles of consecutive pairs (Nx > 512), or stored in FP16.  Equal bit for bit to the two
passes for every operator and equation of state; the claims stay in step across mode switches and new states; waits
are bounded; a launch replayed on counters that have moved on says so."""

import numpy as np
import pytest

from gpu_helpers import coexistence, lattice, physics

pytestmark = pytest.mark.gpu

LARGE, WIDE, HALF = (128, 120, 112), (514, 9, 5), (32, 16, 12)


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1805_08643_gb300 import _build

    _build.build()
    # LARGE is past the several-steps kernel's limit: 128 pairs a tile, 7 blocks an SM, 5 tiles a block
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert LARGE[2] * -(-LARGE[0] // 2 * LARGE[1] // 128) > 5 * 7 * sms


def _box(grid, op, prec, mode, eos="cs", stream=None):
    if eos == "exp":
        phys, (rl, rv) = physics(eos="exp", G=-10.0 / 3.0), (2.78, 0.37)
    else:
        phys, (rl, rv) = physics(sigma=0.105), coexistence(0.8)
    lat = lattice(grid, op, prec, phys, stream=stream)
    lat.set_tuning(mode)
    lat.init_droplet(tuple(0.4 * n for n in grid), 0.3 * min(grid), 3.0, rl, rv)
    return lat


def _equal(a, b):
    return np.array_equal(a.populations(), b.populations()) and all(
        np.array_equal(x, y) for x, y in zip(a.moments(), b.moments()))


@pytest.mark.parametrize("eos, arith", [("cs", "f64"), ("cs", "f32x2"), ("exp", "f64")])
@pytest.mark.parametrize("op", ["nonorth", "orth", "nonorth_d3q15"])
@pytest.mark.parametrize("grid, prec", [(LARGE, "f32"), (WIDE, "f32"), (HALF, "f16")])
def test_equals_two_pass_bit_for_bit(grid, prec, op, eos, arith):
    a, b = _box(grid, op, prec, False, eos), _box(grid, op, prec, "queue", eos)
    for lat in (a, b):
        lat.set_eos_arith(arith)
        lat.step(9)
        assert lat.check() == 0
    assert _equal(a, b)
    a.close()
    b.close()


BOXES = [(LARGE, "f32"), (WIDE, "f32"), (HALF, "f16")]


@pytest.mark.parametrize("grid, prec", BOXES)
def test_claims_stay_in_step_across_modes_and_states(grid, prec):
    a, b = _box(grid, "nonorth", prec, False), _box(grid, "nonorth", prec, "queue")
    a.step(15)
    for n in (1, 2, 5):
        b.step(n)
    b.set_tuning(False)
    b.step(3)
    b.set_tuning("queue")
    b.step(4)
    assert a.check() == 0 and b.check() == 0 and _equal(a, b)
    f = b.populations()
    b.set_populations(f)  # a new state on the same counters
    for lat in (a, b):
        lat.set_populations(f)
        lat.step(4)
        assert lat.check() == 0
    assert _equal(a, b)
    a.close()
    b.close()


@pytest.mark.parametrize("grid, prec", BOXES[1:])
def test_bounded_waits(grid, prec):
    from paper_1805_08643_gb300.lbm import ERR_TIMEOUT

    a, b = _box(grid, "nonorth", prec, False), _box(grid, "nonorth", prec, "queue")
    f = b.populations()
    b.set_wait_budget(64, inject_unreachable=True)
    b.step(2)
    assert b.check() == ERR_TIMEOUT
    b.set_wait_budget(0, inject_unreachable=False)
    for lat in (a, b):
        lat.set_populations(f)
        lat.step(6)
        assert lat.check() == 0
    assert _equal(a, b)
    a.close()
    b.close()


@pytest.mark.parametrize("grid, prec", BOXES[1:])
def test_a_replayed_launch_reports_its_counters(grid, prec):
    import torch

    from paper_1805_08643_gb300.lbm import ERR_TIMEOUT

    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        lat = _box(grid, "nonorth", prec, "queue", stream=s)
        lat.step(2)
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        g.capture_begin()
        lat.step(2)
        g.capture_end()
        g.replay()  # the launches the capture stands for
        s.synchronize()
        assert lat.check() == 0
        g.replay()  # their counters have moved on
        s.synchronize()
        assert lat.check() == ERR_TIMEOUT
        lat.close()
