"""Grids of different tiles alive at once: the shared-memory limit of a kernel is
one per process, so a grid must still launch after another, with smaller or
slightly larger tiles, was created.  Steps, the persistent step, the split calls,
diagnostics and the adjoint of both grids are taken in turn, in both orders of
creation, and must give what each grid gives alone."""
import numpy as np
import pytest

from paper_1101_0809_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1101_0809_gb300 import build as B
    B.build()
    from paper_1101_0809_gb300 import pic
    return pic


def build(P, dims, prec, order2, tile):
    n = (60, 44, 1) if dims == 2 else (24, 20, 22)
    wl = W.thermal_plasma("two", dims, n, 2, 0.1, 1, W.SEED_BASE + 86, dt_courant=0.45)
    g = P.Grid(P.make_desc(dims, n, wl.d, wl.dt, wl.c, prec, tile=tile, rho_bg=wl.rho_bg, sort_interval=2, order2=order2))
    sp = wl.species[0]
    g.load(0, sp.q, sp.m, sp.weight, sp.x, sp.w)
    return g


def calls(P, g, order2):
    yield lambda: P.pic_step(g.h, 3)
    if order2 == 3:
        yield lambda: P.pic_step_persistent(g.h, 3)

    def parts():
        P.pic_yee_update(g.h, P.PIC_B_HALF)
        P.pic_gather_push(g.h)
        P.pic_deposit_current(g.h)
        P.pic_yee_update(g.h, P.PIC_B_HALF)
        P.pic_yee_update(g.h, P.PIC_E_FULL)

    yield parts
    yield lambda: P.pic_diagnostics(g.h)
    if order2 == 3:
        import torch
        dt = torch.float64 if g.precision == P.PIC_FP64 else torch.float32
        lam = [[torch.full(s, 0.5, dtype=dt, device="cuda") for _ in range(3)]
               for s in (g.shape, g.shape, (P.pic_num_particles(g.h, 0),), (P.pic_num_particles(g.h, 0),))]
        yield lambda: P.pic_adjoint_step(g.h, *lam)
    yield lambda: P.pic_step(g.h, 1)


# 3D FP64: 4x4x2 leaves room for two blocks per SM with the larger deposit queues
# (115264 bytes), 4x4x5 does not (100352 bytes, with the smaller ones)
TILES = [(2, 0, 3, (24, 24, 1), (8, 8, 1)), (2, 1, 3, (24, 20, 1), (16, 16, 1)), (2, 1, 5, (24, 24, 1), (8, 8, 1)),
         (3, 1, 3, (8, 8, 8), (8, 4, 4)), (3, 1, 3, (8, 4, 4), (4, 4, 4)), (3, 0, 3, (8, 8, 8), (4, 4, 4)),
         (3, 0, 3, (4, 4, 2), (4, 4, 5)), (3, 1, 5, (6, 6, 6), (4, 4, 4)),
         (3, 1, 4, (8, 8, 8), (4, 4, 4))]


@pytest.mark.parametrize("dims,prec,order2,one,two", TILES)
@pytest.mark.parametrize("swap", [False, True])
def test_grids_of_different_tiles_step_in_turn(P, dims, prec, order2, one, two, swap):
    tiles = (two, one) if swap else (one, two)
    grids = [build(P, dims, prec, order2, t) for t in tiles]
    for pair in zip(*[list(calls(P, g, order2)) for g in grids]):
        for call in pair:
            call()
    for g in grids:
        P.pic_sync(g.h)
    both = [g.get_fields() for g in grids]
    for g in grids:
        g.close()
    for t, f in zip(tiles, both):
        g = build(P, dims, prec, order2, t)
        for call in calls(P, g, order2):
            call()
        P.pic_sync(g.h)
        # the same kernels on the same numbers, but for the order of the sums of J:
        # a few roundings a step
        tol = 64 * (2.0 ** -52 if prec == 0 else 2.0 ** -23)
        alone = g.get_fields()
        for u, v in zip(f[0] + f[1], alone[0] + alone[1]):
            np.testing.assert_allclose(u, v, rtol=0, atol=tol * max(float(np.abs(v).max()), 1e-300))
        g.close()
