"""Streaming plasmas between sorts: a work item whose particles ran past its
staged tile stages the tile where they are.  Steps through the wrap of the box,
along and against every axis, with one stream and with two that leave the tile
on opposite sides, must equal the oracle's whatever the items staged."""
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


def stream(dims, beam, steps, two):
    """Electrons at v_th = 0.1c on sizes ragged against the tiles, with the
    momentum `beam` (in c) added to all of them, or taken from every second one."""
    n = (36, 28, 1) if dims == 2 else (21, 18, 15)
    wl = W.thermal_plasma("stream", dims, n, 4, 0.1, steps, W.SEED_BASE + 78, tile=(8, 8, 1) if dims == 2 else (8, 4, 4),
                          dt_courant=0.45)
    sp = wl.species[0]
    sp.x = np.floor(sp.x) + (sp.x % 1.0).astype(np.float32).clip(max=np.float32(1 - 2.0 ** -24))
    sign = np.ones(sp.n)
    if two:
        sign[::2] = -1.0
    for a in range(3):
        sp.w[a] += beam[a] * wl.c * sign
    sp.w = np.ascontiguousarray(sp.w.astype(np.float32).astype(np.float64))
    return wl


CASES = [(2, (3.0, 0.0, 0.0), False), (2, (-2.0, 2.0, 0.5), False), (2, (2.0, 1.0, 0.0), True),
         (3, (3.0, 0.0, 0.0), False), (3, (-1.5, 2.0, -1.5), False), (3, (0.0, 0.0, 3.0), True)]


def shifted(wl, grid, halo):
    """Particles more than `halo` cells past the tile they were sorted in."""
    cell, _, _, ident = grid.particles(0)
    c = [cell % wl.n[0], (cell // wl.n[0]) % wl.n[1], cell // (wl.n[0] * wl.n[1])]
    out = np.zeros(cell.size, dtype=bool)
    for a in range(wl.dims):
        d = (c[a] - (np.floor(wl.species[0].x[a][ident]).astype(np.int64) // wl.tile[a]) * wl.tile[a]) % wl.n[a]
        out |= (d >= wl.tile[a] + halo) & (d < wl.n[a] - halo)
    return int(out.sum())


@pytest.mark.parametrize("dims,beam,two", CASES)
@pytest.mark.parametrize("halo", [0, 2])
def test_streams_between_sorts_match_oracle(P, dims, beam, two, halo):
    steps = 7
    wl = stream(dims, beam, steps, two)
    for prec in (P.PIC_FP64, P.PIC_FP32):
        f64 = prec == P.PIC_FP64
        grid = make_grid(P, wl, prec, halo=halo, sort_interval=1000, ppb=512)
        osp = [O.Species(s.q, s.m, s.weight, s.x.copy(), s.w.copy()) for s in wl.species]
        g = O.Grid(wl.dims, wl.n, wl.d, wl.dt, wl.c)
        E, B, J = g.zeros(), g.zeros(), g.zeros()
        for _ in range(steps):
            O.step(g, E, B, J, osp)
        P.pic_step(grid.h, steps)
        P.pic_sync(grid.h)
        assert shifted(wl, grid, halo) > 0
        tol = fp64_field_tol(wl, osp) if f64 else steps * FP32_TOL
        gE, gB, gJ = grid.get_fields()
        for a in range(3):
            close(gE[a], E[a], tol, f"E[{a}]")
            close(gB[a], B[a], tol, f"B[{a}]")
            close(gJ[a], J[a], tol, f"J[{a}]")
        if f64:
            compare_particles(wl, 0, grid, osp, tol)
        grid.close()


@pytest.mark.parametrize("dims,beam,two", [CASES[1], CASES[5]])
def test_the_split_step_of_a_stream_equals_the_oracle(P, dims, beam, two):
    steps = 6
    wl = stream(dims, beam, steps, two)
    grid = make_grid(P, wl, P.PIC_FP64, halo=1, sort_interval=1000)
    osp = [O.Species(s.q, s.m, s.weight, s.x.copy(), s.w.copy()) for s in wl.species]
    g = O.Grid(wl.dims, wl.n, wl.d, wl.dt, wl.c)
    E, B, J = g.zeros(), g.zeros(), g.zeros()
    for _ in range(steps):
        P.pic_yee_update(grid.h, P.PIC_B_HALF)
        P.pic_gather_push(grid.h)
        P.pic_deposit_current(grid.h)
        P.pic_yee_update(grid.h, P.PIC_B_HALF)
        P.pic_yee_update(grid.h, P.PIC_E_FULL)
        O.step(g, E, B, J, osp)
    tol = fp64_field_tol(wl, osp)
    gE, gB, gJ = grid.get_fields()
    for a in range(3):
        close(gE[a], E[a], tol, f"E[{a}]")
        close(gJ[a], J[a], tol, f"J[{a}]")
    compare_particles(wl, 0, grid, osp, tol)
    grid.close()
