"""psi = psi0 exp(-rho0 / rho) of the FP32-arithmetic forms is the FP64 value rounded once, whatever rho_ref: populations
whose only deviation is that of the rest population give densities without a rounding, and u at rest is F / (2 rho)."""

import numpy as np
import pytest

from oracle import d3q15 as D
from oracle import lbm_oracle as L

pytestmark = pytest.mark.gpu

GRID, G = (64, 40, 32), -10.0 / 3.0


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1805_08643_gb300 import _build

    _build.build()


@pytest.mark.parametrize("op", ["nonorth", "nonorth_d3q15"])
@pytest.mark.parametrize("arith", ["f64", "f32x2"])
@pytest.mark.parametrize("lo, hi", [(0.015, 0.05), (0.05, 6.0)])
@pytest.mark.parametrize("rho_ref", [0.0, 0.37, 2.78])
def test_psi_is_the_fp64_value_rounded_once(rho_ref, lo, hi, arith, op):
    from paper_1805_08643_gb300.lbm import Lattice, Rates

    M = D if op == "nonorth_d3q15" else L
    rng = np.random.default_rng(5)
    d = (np.exp(rng.uniform(np.log(lo), np.log(hi), GRID[::-1])) - rho_ref).astype(np.float32).astype(float)
    rho = rho_ref + d
    f = M.W_LATTICE[:, None, None, None] * np.full((1, *GRID[::-1]), rho_ref)
    f[0] += d
    lat = Lattice(GRID, operator=op, precision="f32", eos="exp", psi0=1.0, rho0=1.0, G=G, rates=Rates())
    lat.set_eos_arith(arith)
    lat.init_field(rho, rho_ref)
    lat.set_populations(f)
    got_rho, u = lat.moments()
    assert lat.check() == 0
    lat.close()
    assert np.abs(got_rho - rho).max() <= 2.0**-50  # w_a rho_ref as two roundings here and a contracted one there
    psi = np.exp(-1.0 / rho).astype(np.float32).astype(float)
    S, size = np.zeros((3, *rho.shape)), np.zeros_like(rho)
    for w, e in zip(M.W_FORCE, M.E):
        if w:
            nb = w * L.shifted(psi, e)
            size += nb
            for k in range(3):
                S[k] += int(e[k]) * nb
    # some twenty FP64 roundings of sums of that size; one FP32 place in one psi is 2^-24 / 24 of it or more
    assert np.all(np.abs(u - -0.5 * G * psi * S / got_rho) <= 64 * 2.0**-53 * abs(G) * psi * size / rho)
