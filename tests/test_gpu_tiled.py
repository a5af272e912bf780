"""A periodic box filled with copies of a small one evolves as the small one does, whatever kernels the sizes choose.
So small boxes are the reference for what only large ones reach: odd-Nx boxes too large for padded rows, which the
one-node kernels step, and whose rounding every odd box has; and two-pass steps whose launches overlap."""

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


def _tile(grid, seed=7):
    """A density field between the phases without symmetry."""
    rl, rv = coexistence(0.8)
    rng = np.random.default_rng(seed)
    return rv + (rl - rv) * (0.3 + 0.02 * rng.random(grid[::-1])), rv


def _fields(grid, op, prec, tile, copies, steps, mode=False):
    """rho and u on the device after `steps` steps of copies (x, y, z) of the tile."""
    import torch

    rho0, rv = tile
    big = tuple(g * c for g, c in zip(grid, copies))
    lat = lattice(big, op, prec, physics(sigma=0.105))
    lat.set_tuning(mode)
    lat.init_field(torch.from_numpy(rho0).cuda().repeat(copies[::-1]).reshape(-1), rv)
    lat.step(steps)
    rho = torch.empty(lat.n, dtype=torch.float64, device="cuda")
    u = torch.empty(3 * lat.n, dtype=torch.float64, device="cuda")
    lat.moments_device(rho, u)
    assert lat.check() == 0
    lat.close()
    return torch.cat([rho, u]).reshape(4, big[2], big[1], big[0])


def _assert_tiled(big, small):
    _, nz, ny, nx = small.shape
    d, z, y, x = big.shape
    for k in range(d):
        parts = big[k].view(z // nz, nz, y // ny, ny, x // nx, nx)
        assert bool((parts == small[k].view(1, nz, 1, ny, 1, nx)).all()), k


# 6 x 6144 x 6300 padded nodes times 19 directions pass 2^32, 5 x 6144 x 6300 times 19 do not
ODD, ODD_COPIES = (5, 6, 7), (1, 1024, 900)


@pytest.mark.parametrize("prec", ["f32", "f16"])
@pytest.mark.parametrize("op", ["nonorth", "orth", "nonorth_d3q15"])
def test_odd_rows_round_as_the_one_node_kernels(op, prec):
    import torch

    tile = _tile(ODD)
    small = _fields(ODD, op, prec, tile, (1, 1, 1), 12)
    big = _fields(ODD, op, prec, tile, ODD_COPIES, 12)
    _assert_tiled(big, small)
    del big
    torch.cuda.empty_cache()


def _chained_pair(tile_grid, copies, op, prec):
    """A box above the sizes from which launches overlap, and its tile below them, on the two-pass step."""
    rho0, rv = _tile(tile_grid)
    small = lattice(tile_grid, op, prec, physics(sigma=0.105))
    big = lattice(tuple(g * c for g, c in zip(tile_grid, copies)), op, prec, physics(sigma=0.105))
    assert small.n < 1 << 15 and big.n >= (1 << 18 if prec == "f64" else 1 << 15)
    for lat, rho in ((small, rho0), (big, np.tile(rho0, copies[::-1]))):
        lat.set_tuning(False)
        lat.init_field(rho, rv)
    return small, big


def _assert_same_populations(small, big):
    import torch

    fs, fb = torch.from_numpy(small.populations()), torch.from_numpy(big.populations())
    assert small.check() == 0 and big.check() == 0
    _assert_tiled(fb, fs)


CHAINED = [((12, 10, 9), (6, 6, 8)), ((13, 10, 9), (5, 6, 8)), ((32, 8, 5), (4, 10, 14))]


@pytest.mark.parametrize("prec", ["f64", "f32", "f16"])
@pytest.mark.parametrize("op", ["nonorth", "orth", "nonorth_d3q15"])
@pytest.mark.parametrize("tile_grid, copies", CHAINED)
def test_overlapping_launches_step_as_separate_ones(tile_grid, copies, op, prec):
    small, big = _chained_pair(tile_grid, copies, op, prec)
    small.step(40)
    for n in (1, 1, 3, 35):
        big.step(n)
    _assert_same_populations(small, big)
    small.close()
    big.close()


@pytest.mark.parametrize("prec", ["f64", "f32", "f16"])
def test_overlapping_launches_replayed_from_a_graph(prec):
    import torch

    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        small, big = _chained_pair(*CHAINED[0], "nonorth", prec)
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        g.capture_begin()
        big.step(2)  # two steps: the state is back in the buffer the capture read
        g.capture_end()
        for _ in range(20):
            g.replay()
        small.step(40)
        s.synchronize()
        _assert_same_populations(small, big)
        small.close()
        big.close()


def _batch(prec, grid, others=()):
    """A slab along x in a box of a batch, other boxes beside it: rho and u on the device after 9 steps."""
    import ctypes

    import torch

    from paper_1805_08643_gb300.lbm import Batch, Rates, lib

    phys = physics(sigma=0.105)
    rl, rv = coexistence(0.8)
    b = Batch(prec, "cs")
    ids = []
    for g in (grid, *others):
        ids.append(b.add(g, "nonorth", T=phys["T"], sigma=0.105, rates=Rates(s_e=1.1, s_nu=1.0)))
        b.init_flat(ids[-1], 0, 0.3 * g[0], 0.7 * g[0], 1.5, rl, rv)
    b.step(4)
    b.step(5)
    assert b.check() == 0
    n = grid[0] * grid[1] * grid[2]
    out = torch.empty(4 * n, dtype=torch.float64, device="cuda")
    assert lib.lbm_batch_moments(b._h, ids[0], ctypes.c_void_p(out.data_ptr()),
                                 ctypes.c_void_p(out.data_ptr() + 8 * n), 1) == 0
    b.stream.synchronize()
    b.close()
    return out.reshape(4, *grid[::-1])


# rows that cannot be padded: past 2^32 elements; more tiles in a plane than a work list has numbers for
@pytest.mark.parametrize("grid", [(5, 6144, 6300), (511, 33000, 3)])
@pytest.mark.parametrize("prec", ["f32", "f16"])
def test_batches_step_odd_boxes_without_padding(grid, prec):
    import torch

    big = _batch(prec, grid, [(16, 12, 10), (15, 12, 10)])
    row = big[:, :1, :1].clone()
    assert bool((big == row).all())  # nothing varies along y and z
    small = _batch(prec, (grid[0], 8, 6))[:, :1, :1]
    assert float((row - small).abs().max()) <= (2e-6 if prec == "f32" else 2e-3)
    del big
    torch.cuda.empty_cache()
