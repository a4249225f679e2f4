"""Every device allocation of a load and of a grid's creation, made to fail in
turn: each of them is reported, and a load that fails before its pools are complete
keeps the particles that were there."""
import numpy as np
import pytest

from paper_1101_0809_gb300 import workloads as W
from pichelpers import make_grid

pytestmark = pytest.mark.gpu

# of a 2D load that changes the layout: the two pools; then the group tables (2), the
# sort's keys and values (4), histogram, sums, counts (5), mover count and classes,
# the tile starts, their scan, the work items, the saved cells and offsets (3)
POOLS, LOAD = 2, 2 + 2 + 4 + 2 + 5 + 2 + 3 + 3
# fields, run tables (3), error word, item count, the diagnostics' four
CREATE = 1 + 3 + 2 + 4


@pytest.fixture(scope="module")
def P():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1101_0809_gb300 import build as B
    B.build()
    from paper_1101_0809_gb300 import pic
    return pic


@pytest.fixture(autouse=True)
def disarm(P):
    yield
    P.pic_inject_alloc_failure(-1)


@pytest.mark.parametrize("after", list(range(LOAD + 1)))
def test_every_allocation_of_a_load(P, after):
    wl = W.c0_small2d(steps=4)
    grid = make_grid(P, wl, P.PIC_FP32)
    P.pic_step(grid.h, 3)
    sp = wl.species[0]
    before = grid.particles(0)
    P.pic_inject_alloc_failure(after)
    if after < LOAD:
        with pytest.raises(P.PicError) as e:
            grid.load(0, sp.q, sp.m, sp.weight, sp.x[:, :4000], sp.w[:, :4000])
        assert e.value.code == P.PIC_ERR_OOM
    else:
        grid.load(0, sp.q, sp.m, sp.weight, sp.x[:, :4000], sp.w[:, :4000])
    P.pic_inject_alloc_failure(-1)
    want = 4000 if after == LOAD else sp.n if after < POOLS else 0
    assert P.pic_num_particles(grid.h, 0) == want
    if after < POOLS:
        for a, b in zip(grid.particles(0), before):
            for u, v in zip(a if isinstance(a, list) else [a], b if isinstance(b, list) else [b]):
                np.testing.assert_array_equal(u, v)
    P.pic_step(grid.h, 12)               # crosses a sort interval, in pairs of steps and alone
    P.pic_step(grid.h, 1)
    d = P.pic_diagnostics(grid.h)
    assert d["n_particles"] == want and d["error_word"] == 0
    grid.load(0, sp.q, sp.m, sp.weight, sp.x, sp.w)
    P.pic_step(grid.h, 2)
    assert P.pic_diagnostics(grid.h)["n_particles"] == sp.n
    grid.close()


@pytest.mark.parametrize("after", list(range(CREATE + 1)))
def test_every_allocation_of_a_creation(P, after):
    wl = W.c0_small2d()
    desc = P.make_desc(wl.dims, wl.n, wl.d, wl.dt, wl.c, P.PIC_FP32, tile=wl.tile, rho_bg=wl.rho_bg)
    P.pic_inject_alloc_failure(after)
    if after < CREATE:
        with pytest.raises(P.PicError) as e:
            P.Grid(desc)
        assert e.value.code == P.PIC_ERR_OOM
    else:
        g = P.Grid(desc)
        P.pic_step(g.h, 1)
        P.pic_sync(g.h)
        g.close()
