"""Loads through the sort's records: cells, offsets, momenta and ids of the
species a call loads, of the ones it keeps (another layout) and of the ones it
keeps in place (same counts), for counts around the kernels' block and slot
sizes and positions on and outside the box's faces."""
import numpy as np
import pytest

from paper_1101_0809_gb300 import workloads as W
from pichelpers import tile_sort_perm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1101_0809_gb300 import build as B
    B.build()
    from paper_1101_0809_gb300 import pic
    return pic


def inputs(wl, count, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    x = np.zeros((3, count))
    for a in range(wl.dims):
        N = float(wl.n[a])
        x[a] = rng.uniform(-1.5 * N, 2.5 * N, count)
        edge = np.array([0.0, N, -N, 2 * N, np.nextafter(N, 0), -1e-17, 1e-17, np.nextafter(1.0, 0), N - 1e-9, 3.0])
        x[a][:min(count, 10)] = np.roll(edge, a)[:min(count, 10)]
    return x, rng.normal(0.0, 1.0, size=(3, count))


def stored(wl, x):
    """Cell and FP32 offsets of positions: wrapped into [0, N), an offset that
    rounds to 1 goes to the next cell."""
    ci, off = [], []
    for a in range(wl.dims):
        N = float(wl.n[a])
        inside = (x[a] >= 0) & (x[a] < N)
        y = np.where(inside, x[a], x[a] - N * np.floor(x[a] / N))
        y = np.where(y >= N, y - N, y)
        y = np.where(y < 0, 0.0, y)
        c = np.minimum(np.floor(y).astype(np.int64), wl.n[a] - 1)
        o = (y - c).astype(np.float32)
        up = o >= 1
        ci.append(np.where(up, (c + 1) % wl.n[a], c))
        off.append(np.where(up, np.float32(0), o))
    cell = ci[0] + wl.n[0] * (ci[1] + wl.n[1] * (ci[2] if wl.dims == 3 else 0))
    return cell.astype(np.int32), off


def check(wl, grid, species, x, w):
    cell, off, wg, ident = grid.particles(species)
    want, woff = stored(wl, x)
    np.testing.assert_array_equal(np.sort(ident), np.arange(x.shape[1]))
    np.testing.assert_array_equal(cell, want[ident])
    for a in range(wl.dims):
        np.testing.assert_array_equal(off[a], woff[a][ident])
    for a in range(3):
        np.testing.assert_array_equal(wg[a], w[a].astype(np.float32)[ident])
    return want, ident


@pytest.mark.parametrize("dims", [2, 3])
@pytest.mark.parametrize("count", [1, 7, 256, 1023, 1025, 5001])
def test_loaded_and_kept_species_hold_their_particles(P, dims, count):
    n, tile = ((37, 29, 1), (8, 8, 1)) if dims == 2 else ((19, 13, 17), (8, 4, 4))
    wl = W.thermal_plasma("load", dims, n, 1, 0.1, 1, W.SEED_BASE + 79, tile=tile)
    grid = P.Grid(P.make_desc(dims, wl.n, wl.d, wl.dt, wl.c, P.PIC_FP32, tile=tile))
    xe, we = inputs(wl, count, 1)
    grid.load(0, -1.0, 1.0, 1.0, xe, we)
    want, ident = check(wl, grid, 0, xe, we)
    perm = tile_sort_perm(wl, want, tile, 1, True, P.pic_tile_layout(grid.h)[2])
    np.testing.assert_array_equal(ident, perm)
    xi, wi = inputs(wl, count + 3, 2)
    grid.load(1, 1.0, 1836.0, 1.0, xi, wi)          # another layout: the electrons are kept
    check(wl, grid, 0, xe, we)
    check(wl, grid, 1, xi, wi)
    xe, we = inputs(wl, count, 3)
    grid.load(0, -1.0, 1.0, 1.0, xe, we)            # the same counts: the ions are kept in place
    check(wl, grid, 0, xe, we)
    check(wl, grid, 1, xi, wi)
    grid.close()
