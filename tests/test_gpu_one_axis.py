"""The 3D deposit of particles that crossed one axis, queued apart from those
that crossed several: plasmas whose particles cross mostly one given axis, any
one, or several at once, in tiles whose deposit queues have room for both kinds
and in tiles whose queues have not, for the three interpolations."""
import numpy as np
import pytest

import oracle as O
from paper_1101_0809_gb300 import workloads as W
from pichelpers import FP32_TOL, close, compare_particles, fp64_field_tol, make_grid

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1101_0809_gb300 import build as B
    B.build()
    from paper_1101_0809_gb300 import pic
    return pic


def plasma(sigma, ppc):
    """Momenta with a standard deviation per axis (in c), on sizes ragged against
    the tiles; FP32 values throughout."""
    wl = W.thermal_plasma("crossings", 3, (21, 18, 19), ppc, 0.1, 1, W.SEED_BASE + 82, dt_courant=0.45)
    sp = wl.species[0]
    sp.x = np.floor(sp.x) + (sp.x % 1.0).astype(np.float32).clip(max=np.float32(1 - 2.0 ** -24))
    rng = np.random.Generator(np.random.PCG64(ppc))
    w = rng.normal(size=sp.w.shape) * np.array(sigma)[:, None] * wl.c
    sp.w = np.ascontiguousarray(w.astype(np.float32).astype(np.float64))
    return wl


@pytest.mark.parametrize("tile", [(8, 4, 4), (8, 4, 8), (8, 8, 8), (5, 3, 4)])
@pytest.mark.parametrize("order2", [3, 4, 5])
@pytest.mark.parametrize("sigma,ppc", [((2.0, 0.0, 0.0), 4), ((0.0, 0.0, 2.0), 1), ((0.1, 0.1, 0.1), 16),
                                       ((1.0, 2.0, 1.0), 6)])
def test_one_step_matches_the_oracle(P, tile, order2, sigma, ppc):
    wl = plasma(sigma, ppc)
    for prec in (P.PIC_FP32, P.PIC_FP64):
        f64 = prec == P.PIC_FP64
        halo = 0 if order2 == 5 and tile[2] == 8 else 1
        try:
            grid = make_grid(P, wl, prec, tile=tile, halo=halo, order2=order2)
        except P.PicError as e:      # tiles of FP64 values that no SM has the shared memory for
            assert f64 and e.code == P.PIC_ERR_INVALID_ARG and "shared memory" in str(e)
            continue
        osp = [O.Species(s.q, s.m, s.weight, s.x.copy(), s.w.copy()) for s in wl.species]
        g = O.Grid(wl.dims, wl.n, wl.d, wl.dt, wl.c, order2)
        E, B, J = g.zeros(), g.zeros(), g.zeros()
        P.pic_step(grid.h, 1)
        P.pic_sync(grid.h)
        O.step(g, E, B, J, osp)
        tol = fp64_field_tol(wl, osp) if f64 else FP32_TOL
        gE, gB, gJ = grid.get_fields()
        # a component without motion along its axis carries rounding only: on the scale of the vector
        scale = max(float(np.sqrt(np.mean(J[a] ** 2))) for a in range(3))
        for a in range(3):
            assert float(np.abs(gJ[a] - J[a]).max()) <= tol * max(scale, float(np.abs(J[a]).max())), f"J[{a}]"
        if all(v > 0 for v in sigma):
            for a in range(3):
                close(gE[a], E[a], tol, f"E[{a}]")
        compare_particles(wl, 0, grid, osp, tol, x_prev=None if f64 else [wl.species[0].x][0])
        grid.close()
