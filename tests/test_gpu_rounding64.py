"""One FP64 step against the same step in extended precision: its populations are off by no more than one last place
(2^-52, as norms).  A moment-by-moment evaluation in FP64 is off by 1.1 to 1.4 of it on these states."""

from fractions import Fraction

import numpy as np
import pytest

from gpu_helpers import physics
from oracle import d3q15 as D
from oracle import lbm_oracle as L

pytestmark = pytest.mark.gpu

GRID, SIGMA, A, B, G = (14, 12, 13), 0.116, 0.25, 4.0, -1.0
LD = np.longdouble


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1805_08643_gb300 import _build

    _build.build()


def _inverse(rows):
    """Inverse of an integer matrix, exact, in extended precision."""
    n = len(rows)
    a = [[Fraction(int(v)) for v in r] + [Fraction(int(i == j)) for j in range(n)] for i, r in enumerate(rows)]
    for c in range(n):
        p = next(r for r in range(c, n) if a[r][c])
        a[c], a[p] = a[p], a[c]
        a[c] = [v / a[c][c] for v in a[c]]
        for r in range(n):
            if r != c and a[r][c]:
                a[r] = [x - a[r][c] * y for x, y in zip(a[r], a[c])]
    return np.array([[LD(v.numerator) / LD(v.denominator) for v in r[n:]] for r in a])


def _operator(op, r):
    """Velocities, M, its inverse, lattice and force weights, rates of an operator."""
    e = np.asarray((D if op == "nonorth_d3q15" else L).E).astype(int)
    x, y, z = e.T
    n = (e * e).sum(1)
    if op == "orth":
        rows = [n**0, 19 * n - 30, (21 * n * n - 53 * n + 24) // 2, x, (5 * n - 9) * x, y, (5 * n - 9) * y, z,
                (5 * n - 9) * z, 3 * x * x - n, (3 * n - 5) * (3 * x * x - n), y * y - z * z,
                (3 * n - 5) * (y * y - z * z), x * y, y * z, x * z, (y * y - z * z) * x, (z * z - x * x) * y,
                (x * x - y * y) * z]
        rate = [1, r["s_e"], r["s_eps"], 1, r["s_q"], 1, r["s_q"], 1, r["s_q"], r["s_nu"], r["s_pi"], r["s_nu"],
                r["s_pi"], r["s_nu"], r["s_nu"], r["s_nu"], r["s_m"], r["s_m"], r["s_m"]]
    else:
        rows = [n**0, x, y, z, n, 3 * x * x - n, y * y - z * z, x * y, x * z, y * z, x * x * y, x * y * y, x * x * z]
        if op == "nonorth":
            rows += [x * z * z, y * y * z, y * z * z, x * x * y * y, x * x * z * z, y * y * z * z]
            rate = [1] * 4 + [r["s_e"]] + [r["s_nu"]] * 5 + [r["s_q"]] * 6 + [r["s_pi"]] * 3
        else:
            rows += [x * y * z, x * x * y * y]
            rate = [1] * 4 + [r["s_e"]] + [r["s_nu"]] * 5 + [r["s_q"]] * 4 + [r["s_pi"]]
    rows = np.array(rows)
    axis, diag = ((9, 72), (3, 24)) if len(e) == 15 else ((18, 36), (6, 12))
    w = np.array([LD(2) / 9 if len(e) == 15 else LD(1) / 3] + [LD(1) / axis[0 if k == 1 else 1] for k in n[1:]])
    wf = [LD(1) / diag[0 if k == 1 else 1] for k in n[1:]]
    return e, rows.astype(LD), _inverse(rows), w, wf, np.array(rate, dtype=float).astype(LD)[:, None, None, None]


def _step(op, phys, f):
    e, M, Minv, w, wf, lam = _operator(op, phys)
    f = f.astype(LD)
    rho = f.sum(0)
    eta = LD(B) * rho / 4
    p = rho * LD(phys["R"]) * LD(phys["T"]) * (1 + eta + eta**2 - eta**3) / (1 - eta) ** 3 - LD(A) * rho**2
    psi = np.sqrt(2 * (p - rho / 3) / LD(G))
    S = np.zeros((3, *rho.shape), dtype=LD)
    for wk, ek in zip(wf, e[1:]):
        S += ek.astype(LD)[:, None, None, None] * (wk * L.shifted(psi, ek))
    F = -LD(G) * psi * S
    u = (np.tensordot(e.T.astype(LD), f, 1) + F / 2) / rho
    dS = 6 * LD(SIGMA) * LD(G) ** 2 / (1 / LD(phys["s_e"]) - LD(1) / 2) * (S * S).sum(0)
    uu, Fu, third = (u * u).sum(0), (u * F).sum(0), LD(1) / 3
    if op == "orth":
        eu, eF, wx = np.tensordot(e.astype(LD), u, 1), np.tensordot(e.astype(LD), F, 1), w[:, None, None, None]
        meq = np.tensordot(M, wx * rho * (1 + 3 * eu + LD(9) / 2 * eu * eu - LD(3) / 2 * uu), 1)
        src = np.tensordot(M, wx * (3 * (eF - Fu) + 9 * eu * eF), 1)
        src[1] += 19 * dS
        src[2] -= 16 * dS
    else:
        (x, y, z), (Fx, Fy, Fz), zero = u, F, np.zeros_like(rho)
        c, phi = rho * third, rho / 9 * (1 - LD(3) / 2 * uu)
        meq = [rho, rho * x, rho * y, rho * z, rho + rho * uu, rho * (2 * x * x - y * y - z * z), rho * (y * y - z * z),
               rho * x * y, rho * x * z, rho * y * z]
        src = [zero, Fx, Fy, Fz, 2 * Fu + dS, 2 * (2 * Fx * x - Fy * y - Fz * z), 2 * (Fy * y - Fz * z),
               Fx * y + Fy * x, Fx * z + Fz * x, Fy * z + Fz * y]
        if op == "nonorth":
            meq += [c * y, c * x, c * z, c * x, c * z, c * y]
            meq += [phi + c * (x * x + y * y), phi + c * (x * x + z * z), phi + c * (y * y + z * z)]
            src += [Fy / 3, Fx / 3, Fz / 3, Fx / 3, Fz / 3, Fy / 3]
            src += [2 * third * (x * Fx + y * Fy), 2 * third * (x * Fx + z * Fz), 2 * third * (y * Fy + z * Fz)]
        else:
            meq += [c * y, c * x, c * z, zero, phi + 2 * third * c * uu]
            src += [Fy / 3, Fx / 3, Fz / 3, zero, 4 * third * third * Fu]
        meq, src = np.stack(meq), np.stack(src)
    m = np.tensordot(M, f, 1)
    out = np.tensordot(Minv, m + lam * (meq - m) + (1 - lam / 2) * src, 1)
    return np.stack([np.roll(v, (int(k[2]), int(k[1]), int(k[0])), (0, 1, 2)) for v, k in zip(out, e)])


@pytest.mark.parametrize("op", ["nonorth", "orth", "nonorth_d3q15"])
@pytest.mark.parametrize("field", ["droplet", "slab"])
def test_one_step_is_within_a_last_place(op, field):
    from paper_1805_08643_gb300 import thermo
    from paper_1805_08643_gb300.lbm import Lattice, Rates

    rl, rv = thermo.coexistence_cs(0.7, A, B, 1.0)
    phys = physics(sigma=SIGMA)
    phys["T"] = 0.7 * thermo.critical_temperature(A, B, 1.0)
    rates = Rates(*(phys[k] for k in ("s_e", "s_nu", "s_q", "s_pi", "s_eps", "s_m")))
    lat = Lattice(GRID, operator=op, precision="f64", a=A, b=B, R=1.0, T=phys["T"], G=G, rates=rates, sigma=SIGMA)
    if field == "droplet":
        lat.init_droplet((7.2, 6.1, 6.4), 3.0, 3.0, rl, rv)
    else:
        lat.init_flat(2, 3.3, 9.6, 3.0, rl, rv)
    lat.step(20)
    f = lat.populations()
    f *= 1 + 1e-3 * np.random.default_rng(5).standard_normal(f.shape)
    lat.set_populations(f)
    lat.step(1)
    got = lat.populations()
    assert lat.check() == 0
    lat.close()
    want = _step(op, phys, f)
    off = float(np.sqrt(((got - want) ** 2).sum() / (want**2).sum()))
    print(op, field, off * 2.0**52)
    assert off <= 2.0**-52
