"""Boxes with an odd Nx in the FP32-arithmetic forms: stored rows get one element more, which repeats node 0, and
the two-node kernels step them.  The same box on every path (a batch's work list and tile kernels, in a mix with even
boxes) must agree bit for bit in FP32; the single box's two passes collide an odd box's nodes one by one, with other
roundings.  The padding must survive every way a state is set, read and handed from one kind of step to another."""

import numpy as np
import pytest

from gpu_helpers import coexistence, lattice, max_abs, physics

pytestmark = pytest.mark.gpu

GRIDS = [(3, 4, 5), (5, 3, 3), (25, 20, 28), (63, 6, 5), (65, 5, 4), (129, 4, 3)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1805_08643_gb300 import _build

    _build.build()


def _field(grid, seed):
    """A density field between vapour and liquid without symmetry, so that a wrong neighbour shows."""
    rl, rv = coexistence(0.8)
    rng = np.random.default_rng(seed)
    rho = rv + (rl - rv) * (0.3 + 0.02 * rng.random(grid[::-1]))
    return rho, rv


def _two_pass(grid, op, prec, steps, sigma=0.105):
    lat = lattice(grid, op, prec, physics(sigma=sigma))
    lat.set_tuning(False)
    rl, rv = coexistence(0.8)
    lat.init_droplet(tuple(0.37 * n for n in grid), 0.3 * min(grid), 2.0, rl, rv)
    lat.step(steps)
    assert lat.check() == 0
    out = lat.moments()
    lat.close()
    return out


@pytest.mark.parametrize("prec", ["f32", "f16"])
@pytest.mark.parametrize("op", ["nonorth", "orth"])
def test_batch_steps_odd_boxes_as_the_two_pass_single_box(op, prec):
    from paper_1805_08643_gb300.lbm import Batch, Rates

    phys = physics(sigma=0.105)
    rl, rv = coexistence(0.8)
    first = {}
    for tile in (3, 0, 1, 2) if prec == "f32" else (3,):  # the FP16 tile kernels may differ by half an ulp
        b = Batch(prec, "cs")
        boxes = []
        for grid in GRIDS + [(32, 8, 6)]:
            i = b.add(grid, op, T=phys["T"], sigma=0.105, rates=Rates(s_e=1.1, s_nu=1.0))
            b.init_droplet(i, tuple(0.37 * n for n in grid), 0.3 * min(grid), 2.0, rl, rv)
            boxes.append((i, grid))
        b.set_tuning(tile)
        b.step(4)
        b.step(3)
        assert b.check() == 0
        for i, grid in boxes:
            rho, u = b.moments(i)
            rho1, u1 = _two_pass(grid, op, prec, 7)
            if prec == "f32" and grid[0] % 2:
                assert max_abs(rho, rho1) <= 1e-6 and max_abs(u, u1) <= 1e-6, (tile, grid)
                rho1, u1 = first.setdefault(grid, (rho, u))
            assert np.array_equal(rho, rho1) and np.array_equal(u, u1), (tile, grid)
        b.close()


@pytest.mark.parametrize("grid", GRIDS)
@pytest.mark.parametrize("prec", ["f32", "f16"])
def test_padding_survives_mode_switches_and_state_transfers(grid, prec):
    rho0, rv = _field(grid, 3)
    tol = 2e-6 if prec == "f32" else 2e-3  # as between the single pass and the two passes elsewhere

    def run(plan):
        lat = lattice(grid, "nonorth", prec, physics())
        lat.init_field(rho0, rv)
        for what in plan:
            if what == "transfer":
                f = lat.populations()
                lat.set_populations(f)
                assert max_abs(lat.populations(), f) <= (1e-7 if prec == "f32" else 1e-3) * np.abs(f).max()
            else:
                lat.set_tuning(what == "single")
                lat.step(3)
        assert lat.check() == 0
        out = lat.moments()
        lat.close()
        return out

    ref = run(["two", "two", "two"])
    for plan in (["single", "two", "single"], ["two", "transfer", "two", "two"], ["single", "transfer", "two", "single"]):
        rho, u = run(plan)
        assert max_abs(rho, ref[0]) <= tol and max_abs(u, ref[1]) <= tol, plan


@pytest.mark.parametrize("prec", ["f32", "f16"])
def test_odd_boxes_keep_refusing_the_even_modes(prec):
    from paper_1805_08643_gb300.lbm import LBMError

    lat = lattice((25, 8, 6), "nonorth", prec, physics())
    for mode in ("tma", "onchip", "lagged", "queue"):
        with pytest.raises(LBMError, match="ERR_ARG"):
            lat.set_tuning(mode)
    assert lat.tuning()["single_pass"] is False
    lat.close()
