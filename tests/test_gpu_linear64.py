"""The FP64 collisions form their sums in 64-bit fixed point at the scale of a node's largest value.  States at the
edges of that: scales far from one, values of very different size in a node, nothing but zeros, values the sums are
left to FP64 for (very small, infinite)."""

import numpy as np
import pytest

from gpu_helpers import lattice, oracle_params, physics
from oracle import d3q15 as D
from oracle import lbm_oracle as L

pytestmark = pytest.mark.gpu

GRID = (7, 5, 6)
OPS = ["nonorth", "orth", "nonorth_d3q15"]
SIX_RATES = dict(s_e=1.25, s_nu=0.75, s_q=1.5, s_pi=0.875, s_eps=1.125, s_m=1.375)


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1805_08643_gb300 import _build

    _build.build()


def _lattice(op, rho_ref=0.0):
    lat = lattice(GRID, op, "f64", physics(eos="none", G=0.0, rates=SIX_RATES))
    lat.init_field(np.ones(GRID[::-1]), rho_ref)
    return lat


def _populations(op, seed):
    M = D if op == "nonorth_d3q15" else L
    rng = np.random.default_rng(seed)
    return M.W_LATTICE[:, None, None, None] * (1 + 0.2 * rng.standard_normal((M.Q,) + GRID[::-1]))


def _step(lat, f):
    lat.set_populations(f)
    lat.step(1)
    return lat.populations()


@pytest.mark.parametrize("op", OPS)
def test_results_scale_with_the_state(op):
    lat = _lattice(op)
    f = _populations(op, 1)
    ref = _step(lat, f)
    for k in (-300, -40, 200):  # every operation is exact under a power of two
        assert np.array_equal(_step(lat, f * 2.0**k), ref * 2.0**k), k
    # sums in FP64: 64 roundings of partial sums up to three times the largest population
    small = _step(lat, f * 2.0**-1000)
    assert np.abs(small * 2.0**1000 - ref).max() <= 64 * 2.0**-53 * 3 * np.abs(f).max()
    lat.close()


@pytest.mark.parametrize("op", OPS)
def test_values_of_very_different_size_match_the_oracle(op):
    M = D if op == "nonorth_d3q15" else L
    rng = np.random.default_rng(2)
    f = _populations(op, 2)
    f[1:] *= 2.0 ** -rng.integers(0, 70, f[1:].shape).astype(float)
    f[1:][rng.random(f[1:].shape) < 0.1] = 0.0
    lat = _lattice(op)
    got = _step(lat, f)
    lat.close()
    p = oracle_params(GRID, "orth" if op == "orth" else "nonorth", physics(eos="none", G=0.0, rates=SIX_RATES))
    rho = f.sum(0)
    F = np.zeros((3,) + rho.shape)
    star = M.collide(p, f, rho, M.velocity(f, rho, F), F, np.zeros_like(rho))
    bound = 1e-13 * np.abs(f).sum(0)  # the oracle's dense matrices: some 20 x 30 x 2^-53 of it
    for a in range(M.Q):
        ex, ey, ez = (int(c) for c in M.E[a])
        assert (np.abs(np.roll(got[a], (-ez, -ey, -ex), (0, 1, 2)) - star[a]) <= bound).all(), a


@pytest.mark.parametrize("op", OPS)
def test_a_state_of_zero_deviations_stays(op):
    lat = _lattice(op, rho_ref=1.0)
    f = lat.populations()
    lat.step(3)
    assert np.array_equal(lat.populations(), f)
    lat.close()


@pytest.mark.parametrize("op", OPS)
@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_a_node_that_is_not_finite_reaches_its_neighbours_only(op, bad):
    M = D if op == "nonorth_d3q15" else L
    lat = _lattice(op)
    f = _populations(op, 3)
    ref = _step(lat, f)
    f[8, 2, 3, 4] = bad
    got = _step(lat, f)
    lat.close()
    hit = np.zeros(got.shape, bool)
    for a in range(M.Q):
        ex, ey, ez = M.E[a]
        hit[a, (2 + ez) % GRID[2], (3 + ey) % GRID[1], (4 + ex) % GRID[0]] = True
    assert not np.isfinite(got[hit]).any() and np.array_equal(got[~hit], ref[~hit])


@pytest.mark.parametrize("op", OPS)
def test_densities_of_such_states_give_the_oracles_psi(op):
    M = D if op == "nonorth_d3q15" else L
    rng = np.random.default_rng(4)
    f = _populations(op, 4)
    f[1:] *= 2.0 ** -rng.integers(0, 70, f[1:].shape).astype(float)
    f[1:][rng.random(f[1:].shape) < 0.1] = 0.0
    f *= 0.1 + 0.3 * rng.random(f.shape[1:])
    phys = physics(T_over_Tc=0.8, sigma=0.105, rates=SIX_RATES)
    lat = lattice(GRID, op, "f64", phys)
    lat.init_field(np.full(GRID[::-1], 0.1), 0.0)
    got = _step(lat, f)
    assert lat.check() == 0
    p = oracle_params(GRID, "orth" if op == "orth" else "nonorth", phys)
    rho, u, psi, F = M.macroscopic(p, f)
    # a few hundred roundings of quantities up to ten times the density, which is at least 0.05
    assert np.abs(got - M.stream(M.collide(p, f, rho, u, F, psi))).max() <= 1e-12
    f[5, 1, 2, 3] = np.nan
    _step(lat, f)
    assert lat.check() != 0
    lat.close()
