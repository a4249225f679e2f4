"""Work items of small and uneven pools: a tile's particles are cut into equal
parts of whole warps when whole tiles would leave SMs idle.  Every particle must
be stepped and deposited once, whatever the counts: one particle, one item
exactly, one over, the last part a few particles, and a tile longer than
particles_per_block."""
import numpy as np
import pytest

import oracle as O
from paper_1101_0809_gb300 import workloads as W
from pichelpers import FP32_TOL, FP64_TOL, close, compare_particles, make_grid

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1101_0809_gb300 import build as B
    B.build()
    from paper_1101_0809_gb300 import pic
    return pic


def one_dense_tile(dims, count):
    """count particles in the first tile and a thin plasma elsewhere; positions
    and momenta are FP32 values, so that both precisions start alike."""
    n = (32, 24, 1) if dims == 2 else (16, 14, 12)
    tile = (8, 8, 1) if dims == 2 else (8, 4, 4)
    wl = W.thermal_plasma("dense tile", dims, n, 1, 0.1, 1, W.SEED_BASE + 77, tile=tile, dt_courant=0.45)
    rng = np.random.Generator(np.random.PCG64(count))
    sp = wl.species[0]
    far = sp.x[0] >= tile[0]
    x = np.zeros((3, count))
    for a in range(dims):
        x[a] = rng.integers(0, tile[a], count) + rng.random(count, dtype=np.float32).astype(np.float64)
    rest = np.floor(sp.x[:, far]) + (sp.x[:, far] % 1.0).astype(np.float32).clip(max=np.float32(1 - 2.0 ** -24))
    sp.x = np.ascontiguousarray(np.concatenate([x, rest], axis=1))
    sp.w = np.ascontiguousarray(rng.normal(0.0, 1.0, size=sp.x.shape).astype(np.float32).astype(np.float64))
    return wl


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("dims", [2, 3])
@pytest.mark.parametrize("count,ppb", [(1, 0), (64, 0), (65, 0), (257, 0), (2079, 0), (9001, 0), (130, 64)])
def test_every_particle_of_a_cut_tile_is_stepped_once(P, prec, dims, count, ppb):
    wl = one_dense_tile(dims, count)
    f64 = prec == "fp64"
    tol = FP64_TOL if f64 else FP32_TOL
    grid = make_grid(P, wl, P.PIC_FP64 if f64 else P.PIC_FP32, ppb=ppb)
    osp = [O.Species(s.q, s.m, s.weight, s.x.copy(), s.w.copy()) for s in wl.species]
    g = O.Grid(wl.dims, wl.n, wl.d, wl.dt, wl.c)
    E, B, J = g.zeros(), g.zeros(), g.zeros()
    P.pic_step(grid.h, 1)
    P.pic_sync(grid.h)
    O.step(g, E, B, J, osp)
    gE, gB, gJ = grid.get_fields()
    for a in range(3):
        close(gJ[a], J[a], tol, f"J[{a}]")
        close(gE[a], E[a], tol, f"E[{a}]")
    compare_particles(wl, 0, grid, osp, tol, x_prev=None if f64 else wl.species[0].x)
    grid.close()
