"""rho and u of lbm_moments, lbm_diag and lbm_batch_max_du against sums over the populations in numpy.

The FP32-arithmetic forms sum on the FP32 units through an exact split of every value; the split's constants follow
the largest population of a node, so the nodes here range over many orders of magnitude, and include all-zero
deviations, values below and above the range the split takes, and infinities.
"""

import numpy as np
import pytest

from gpu_helpers import coexistence, lattice, max_abs, physics
from oracle import d3q15, lbm_oracle as L

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1805_08643_gb300 import _build

    _build.build()


def _velocities(op):
    return (d3q15.E if op == "nonorth_d3q15" else L.E).astype(np.longdouble)


def _by_hand(op, f):
    """rho, u and the sums of |f| (extended precision) of populations f (Q, nz, ny, nx) without a force."""
    f = f.astype(np.longdouble)
    rho = f.sum(0)
    j = np.tensordot(_velocities(op).T, f, axes=(1, 0))
    return rho, j / rho, np.abs(f).sum(0)


@pytest.mark.parametrize("prec", ["f64", "f32", "f16"])
@pytest.mark.parametrize("op", ["nonorth", "nonorth_d3q15"])
@pytest.mark.parametrize("grid", [(5, 4, 3), (34, 6, 5), (33, 9, 4)])
def test_moments_are_the_sums_of_the_populations(grid, op, prec):
    rng = np.random.default_rng(7)
    phys = physics(eos="none", G=0.0)
    lat = lattice(grid, op, prec, phys)
    nz, ny, nx = grid[::-1]
    lat.init_field(np.ones(nx * ny * nz), rho_ref=0.0 if prec != "f16" else 1.0)
    q = lat.q
    w = (d3q15.W_LATTICE if op == "nonorth_d3q15" else L.W_LATTICE).reshape(q, 1, 1, 1)
    f = w * (1.0 + 0.3 * rng.standard_normal((q, nz, ny, nx)))
    if prec != "f16":
        f = np.abs(f) * 10.0 ** rng.uniform(-9, 9, (1, nz, ny, nx)) * 10.0 ** rng.uniform(-6, 0, (q, nz, ny, nx))
        f[:, 0, 0, 0] = w[:, 0, 0, 0] * 1e-25  # below the split's range
        f[:, 0, 0, 1] = w[:, 0, 0, 0] * 1e25   # above it
    else:
        f[:, 0, 0, 0] = w[:, 0, 0, 0]          # no deviation from the uniform state
    lat.set_populations(f)
    rho, u = lat.moments()
    stored = lat.populations()
    lat.close()
    r, v, tot = _by_hand(op, stored)
    # populations() rounds every value once (its w rho_ref + deviation), moments at most once per addition of
    # a 19-term tree and a handful of times after it: 64 roundings of the sum of magnitudes cover both
    assert np.all(np.abs(rho - r) <= 64 * EPS * tot)
    assert np.all(np.abs(u - v) <= 64 * EPS * tot / np.abs(r) * (1 + np.abs(v)))


@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_moments_of_an_infinite_population(prec):
    grid = (6, 4, 3)
    lat = lattice(grid, "nonorth", prec, physics(eos="none", G=0.0))
    lat.init_field(np.ones(72), rho_ref=0.0)
    f = lat.populations()
    f[3, 1, 2, 4] = np.inf
    lat.set_populations(f)
    rho, u = lat.moments()
    d = lat.diag()
    lat.close()
    bad = np.zeros(rho.shape, bool)
    bad[1, 2, 4] = True
    assert np.isinf(rho[bad]).all() and np.isnan(u[1][bad]).all()
    assert np.isfinite(rho[~bad]).all() and np.isfinite(u[:, ~bad]).all()
    assert np.isinf(d["mass"]) and np.isnan(d["max_u"])


@pytest.mark.parametrize("prec", ["f32", "f16"])
@pytest.mark.parametrize("op", ["nonorth", "nonorth_d3q15"])
@pytest.mark.parametrize("grid", [(24, 20, 28), (25, 18, 16)])
def test_moments_and_diag_with_the_force_against_the_fp64_form(grid, op, prec):
    """The same populations in an FP64 box: rho and u differ only by psi's rounding to FP32."""
    rl, rv = coexistence(0.8)
    a = lattice(grid, op, prec, physics())
    centre = tuple(n / 2 for n in grid)
    a.init_droplet(centre, min(grid) / 4, 2.0, rl, rv)
    a.step(7)
    rho, u = a.moments()
    d = a.diag()
    f = a.populations()
    a.close()
    b = lattice(grid, op, "f64", physics())
    b.init_droplet(centre, min(grid) / 4, 2.0, rl, rv)
    b.set_populations(f)
    rho64, u64 = b.moments()
    d64 = b.diag()
    b.close()
    p = L.Params(grid=grid, T=0.8 * L.critical_temperature(1.0, 4.0, 1.0), G=-1.0)
    psi = L.pseudopotential(rho64, p).max()
    # psi carries FP32's rounding (and the FP32 sum of rho behind it, a few more of them): 16 roundings of
    # each of the two factors of F / 2, whose weights sum to 2
    tol = 2 * 16 * 2.0 ** -24 * psi * psi / rho64.min()
    assert max_abs(rho, rho64) <= 64 * EPS * rho64.max()
    assert max_abs(u, u64) <= tol
    assert abs(d["mass"] - d64["mass"]) <= 1e-13 * d64["mass"]
    assert abs(d["max_u"] - np.sqrt((u ** 2).sum(0)).max()) <= 16 * EPS
    assert abs(d["max_u"] - d64["max_u"]) <= 2 * tol
    assert max(abs(np.array(d["momentum"]) - (rho * u).reshape(3, -1).sum(1))) <= 1e-12 * np.abs(rho * u).sum()


def test_max_du_is_the_largest_change_of_u():
    from paper_1805_08643_gb300.lbm import Batch

    rl, rv = coexistence(0.8)
    Tc = L.critical_temperature(1.0, 4.0, 1.0)
    b = Batch("f32", "cs")
    ids = []
    for grid in ((24, 20, 16), (17, 12, 10)):
        ids.append(b.add(grid, "nonorth", T=0.8 * Tc))
        b.init_droplet(ids[-1], tuple(n / 2 for n in grid), min(grid) / 4, 2.0, rl, rv)
    before = [np.zeros((3, *g[::-1])) for g in ((24, 20, 16), (17, 12, 10))]
    for steps in (6, 5):
        b.step(steps)
        now = [b.moments(i)[1] for i in ids]
        du = b.max_du(ids)
        for d, u, v in zip(du, now, before):
            want = np.sqrt(((u - v.astype(np.float32)) ** 2).sum(0)).max()  # the earlier u is kept in FP32
            assert abs(d - want) <= 1e-13 * want + 1e-16
        before = now
    b.close()


@pytest.mark.parametrize("arith", ["f64", "f32x2"])
@pytest.mark.parametrize("psi0, rho0", [(1.0, 1.0), (4.0, 0.3)])
def test_exponential_psi_over_its_range(psi0, rho0, arith):
    """u at rest is F / (2 rho), so it shows psi = psi0 exp(-rho0 / rho): densities from where psi leaves FP32's
    normal range (the FP64 functions) through vapour and liquid to beyond."""
    from paper_1805_08643_gb300.lbm import Lattice, Rates

    grid, G = (36, 10, 9), -10.0 / 3.0
    rng = np.random.default_rng(11)
    field = rho0 * np.exp(rng.uniform(np.log(0.006), np.log(40.0), grid[::-1]))
    lat = Lattice(grid, operator="nonorth", precision="f32", eos="exp", psi0=psi0, rho0=rho0, G=G, rates=Rates())
    lat.set_eos_arith(arith)
    lat.init_field(field, rho_ref=0.0)
    rho, u = lat.moments()
    assert lat.check() == 0
    lat.close()
    p = L.Params(grid=grid, eos="exp", psi0=psi0, rho0=rho0, G=G)
    psi = L.pseudopotential(rho, p)
    want = L.interaction_force(psi, G) / (2 * rho)
    # psi sees rho after an FP32 sum (8 roundings) and is rounded itself: a relative error of 8 rho0 / rho + 1
    # roundings, at the node and at its neighbours; below FP32's normal range the spacing is absolute
    e = psi * (8 * rho0 / rho + 2) * 2.0 ** -24 + psi0 * 2.0 ** -140
    near = sum(wf * L.shifted(psi, d) for wf, d in zip(L.W_FORCE, L.E))
    tol = abs(G) * (e * near + psi * sum(wf * L.shifted(e, d) for wf, d in zip(L.W_FORCE, L.E))) / (2 * rho)
    assert np.all(np.abs(u - want) <= tol + 1e-14 * np.abs(want))
