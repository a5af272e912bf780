"""The orthogonal FP16 fused pass takes blocks of four rows where Nx is a multiple of 64 and Ny of 4: equal bit for bit
to the work list, which visits nodes in another order, on both sides of that rule."""

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


@pytest.mark.parametrize("sigma", [0.0, 0.105])
@pytest.mark.parametrize("grid", [(64, 4, 3), (128, 12, 5), (64, 6, 4), (192, 8, 3), (96, 8, 3)])
def test_two_passes_equal_the_work_list(grid, sigma):
    rl, rv = coexistence(0.8)
    out = []
    for mode in (False, "queue"):
        lat = lattice(grid, "orth", "f16", physics(sigma=sigma))
        lat.set_tuning(mode)
        lat.init_droplet(tuple(0.37 * n for n in grid), 0.3 * min(grid), 2.0, rl, rv)
        lat.step(7)
        assert lat.check() == 0
        out.append(lat.moments())
        lat.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
