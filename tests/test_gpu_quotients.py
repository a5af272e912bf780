"""Velocities are FP64 quotients with the one rounding of a division: states whose sums are exact."""

import numpy as np
import pytest

from gpu_helpers import lattice, physics
from oracle import d3q15 as D
from oracle import lbm_oracle as L

pytestmark = pytest.mark.gpu

GRID = (22, 11, 9)


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1805_08643_gb300 import _build

    _build.build()


def _state(op, scale):
    """Populations that are whole multiples of 2^-16 times the scale: every sum is exact in FP64."""
    M = D if op == "nonorth_d3q15" else L
    rng = np.random.default_rng(9)
    f = rng.integers(1, 1 << 12, (M.Q, *GRID[::-1])).astype(float) * 2.0**-16 * scale
    j = np.stack([sum(int(e[k]) * f[a] for a, e in enumerate(M.E)) for k in range(3)])
    return f, f.sum(0), j


def _half_ulps(got, num, den):
    q = num.astype(np.longdouble) / den
    return np.abs(got - q) / np.spacing(np.abs(q).astype(float))


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("op", ["nonorth", "nonorth_d3q15"])
@pytest.mark.parametrize("scale", [1.0, 2.0**-60, 2.0**90])
def test_velocities_and_largest_speed(op, prec, scale):
    if prec == "f32" and scale > 1e20:
        scale = 2.0**60
    f, rho, j = _state(op, scale)
    lat = lattice(GRID, op, prec, physics(eos="none", G=0.0))
    lat.init_field(np.full(GRID[::-1], 1.0), 0.0)
    lat.set_populations(f)
    got_rho, u = lat.moments()
    d = lat.diag()
    lat.close()
    assert np.array_equal(got_rho, rho)
    assert _half_ulps(u, j, rho).max() <= 0.5001
    speed = np.sqrt((j.astype(np.longdouble) ** 2).sum(0)) / rho
    # |j|^2 of three roundings, a root and a quotient; before the maximum is taken, nodes within a few of those tie
    assert abs(d["max_u"] / speed.max() - 1) <= 4 * 2.0**-53


@pytest.mark.parametrize("bad, want", [(0.0, np.inf), (np.inf, np.nan)])
def test_densities_that_are_no_divisor(bad, want):
    """rho = 0 gives infinite velocities, an infinite population undefined ones, as a division does."""
    lat = lattice(GRID, "nonorth", "f64", physics(eos="none", G=0.0))
    f, rho, j = _state("nonorth", 1.0)
    f[:, 4, 5, 6] = 0.0
    f[1, 4, 5, 6] = 1.0 if bad == 0.0 else bad  # (pulled: the node's own population)
    f[0, 4, 5, 6] = -1.0 if bad == 0.0 else 1.0
    lat.init_field(np.full(GRID[::-1], 1.0), 0.0)
    lat.set_populations(f)
    got_rho, u = lat.moments()
    lat.close()
    assert got_rho[4, 5, 6] == bad
    assert np.isnan(u[0, 4, 5, 6]) if np.isnan(want) else u[0, 4, 5, 6] == want
