"""The two-pass step's launches overlap their predecessors' ends (programmatic stream serialization): the same
results from many short calls as from one long one, behind unrelated work on the stream, and when a captured graph
of steps is replayed."""

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


def _start(grid, prec, stream=None):
    rl, rv = coexistence(0.8)
    lat = lattice(grid, "nonorth", prec, physics(sigma=0.105), stream=stream)
    lat.set_tuning(False)
    lat.init_droplet(tuple(n / 2 for n in grid), min(grid) / 4, 2.0, rl, rv)
    return lat


@pytest.mark.parametrize("prec", ["f64", "f32", "f16"])
@pytest.mark.parametrize("grid", [(6, 5, 7), (33, 20, 18), (96, 64, 40)])
def test_step_by_step_and_behind_other_work_equals_one_call(grid, prec):
    import torch

    a = _start(grid, prec)
    a.step(12)
    ref = a.moments()
    a.close()
    b = _start(grid, prec)
    x = torch.zeros(1 << 20, device="cuda")
    for k in range(12):
        x.add_(float(k))
        b.step(1)
        if k % 5 == 0:
            b.diag()
    got = b.moments()
    assert b.check() == 0
    b.close()
    assert np.array_equal(ref[0], got[0]) and np.array_equal(ref[1], got[1])
    assert float(x[0]) == sum(range(12))


@pytest.mark.parametrize("prec", ["f64", "f16"])
def test_captured_steps_replay(prec):
    import torch

    grid = (32, 24, 20)
    a = _start(grid, prec)
    a.step(8)
    ref = a.moments()
    a.close()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        b = _start(grid, prec, stream=s)
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        g.capture_begin()
        b.step(2)  # two steps: the state is back in the buffer the capture read
        g.capture_end()
        for _ in range(4):
            g.replay()
        s.synchronize()
        got = b.moments()
        assert b.check() == 0
        b.close()
    assert np.array_equal(ref[0], got[0]) and np.array_equal(ref[1], got[1])
