"""A particle whose momentum becomes non-finite contributes no current and moves
nowhere, also when the step is taken by its parts: pic_gather_push saves no old
position for it, and pic_deposit_current must not use one.  The others' current is
that of the same plasma without the particle."""
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


@pytest.mark.parametrize("dims,order2", [(2, 3), (3, 3), (2, 4), (3, 4), (3, 5)])
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("beam", [0.0, 3.0])   # c; at 3 the particles leave the staged tiles between the sorts
def test_split_step_with_a_lost_particle(P, dims, order2, prec, beam):
    n = (24, 20, 1) if dims == 2 else (18, 14, 16)
    wl = W.thermal_plasma("lost", dims, n, 3, 0.1, 1, W.SEED_BASE + 87, dt_courant=0.45)
    sp = wl.species[0]
    sp.w[0] += beam * wl.c
    lost = np.array([5, sp.n // 2, sp.n - 1])
    rest = np.setdiff1d(np.arange(sp.n), lost)
    w = sp.w.copy()
    w[0, lost[0]] = np.nan
    w[1, lost[1]] = np.inf
    w[2, lost[2]] = np.nan
    J, cells = [], []
    for x, v in ((sp.x, w), (sp.x[:, rest], sp.w[:, rest])):
        g = P.Grid(P.make_desc(dims, n, wl.d, wl.dt, wl.c, prec, tile=(4, 4, 1) if dims == 2 else (4, 4, 4), halo=0,
                               sort_interval=1000, order2=order2))
        g.load(0, sp.q, sp.m, sp.weight, np.ascontiguousarray(x), np.ascontiguousarray(v))
        at = []
        for _ in range(6):
            P.pic_gather_push(g.h)
            P.pic_deposit_current(g.h)
            at.append(g.get_fields()[2])
        J.append(at)
        cell, _, _, ident = g.particles(0)
        cells.append(dict(zip(ident.tolist(), cell.tolist())))
        if x is sp.x:
            with pytest.raises(P.PicError) as e:
                P.pic_sync(g.h)
            assert e.value.code == P.PIC_ERR_NONFINITE
        else:
            P.pic_sync(g.h)
        g.close()
    c = [np.floor(a).astype(int) for a in sp.x[:dims, lost]]
    start = c[0] + n[0] * (c[1] + (n[1] * c[2] if dims == 3 else 0))
    assert [cells[0][int(q)] for q in lost] == start.tolist()
    # the same sums in another order; the fixed point of the FP32 tiles is exact to 2^-24 of a
    # block's largest sum
    tol = 64 * (2.0 ** -52 if prec == 0 else 2.0 ** -23)
    for a, b in zip(*J):
        for u, v in zip(a, b):
            np.testing.assert_allclose(u, v, rtol=0, atol=tol * float(np.abs(v).max()))
