"""The momentum of a node whose rest population is far larger than the moving ones keeps FP64's accuracy relative to
those: the observables' sums are exact in the FP32-arithmetic forms, at the scale of what they sum."""

import numpy as np
import pytest

from gpu_helpers import lattice, physics
from oracle import d3q15 as D
from oracle import lbm_oracle as L

pytestmark = pytest.mark.gpu

GRID = (18, 9, 7)


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1805_08643_gb300 import _build

    _build.build()


@pytest.mark.parametrize("op", ["nonorth", "nonorth_d3q15"])
@pytest.mark.parametrize("down", [0, 20, 33, 48])
def test_momentum_beside_a_large_rest_population(op, down):
    M = D if op == "nonorth_d3q15" else L
    rng = np.random.default_rng(3)
    f = rng.standard_normal((M.Q, *GRID[::-1])).astype(np.float32).astype(float) * 2.0**-down
    f[0] = (1 + rng.random(GRID[::-1])).astype(np.float32)
    lat = lattice(GRID, op, "f32", physics(eos="none", G=0.0))
    lat.init_field(np.ones(GRID[::-1]), 0.0)
    lat.set_populations(f)
    rho, u = lat.moments()
    lat.close()
    fl = f.astype(np.longdouble)
    # twenty roundings of sums of that size, and two of the quotient
    assert np.all(np.abs(rho - fl.sum(0)) <= 20 * 2.0**-53 * np.abs(f).sum(0))
    for k in range(3):
        j = sum(int(e[k]) * fl[a] for a, e in enumerate(M.E))
        size = sum(np.abs(f[a]) for a, e in enumerate(M.E) if e[k])
        assert np.all(np.abs(u[k] * rho.astype(np.longdouble) - j) <= 24 * 2.0**-53 * size)
