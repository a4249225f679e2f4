"""The one-pass end of a step (second B half step and E step, into second field
buffers) against the same step by its parts, which updates in place: odd sizes
down to the smallest grid, both precisions, batches of runs of unequal size, an
antenna next to and away from its plane's neighbours, an odd and an even number
of steps, and calls that use the fields between them."""
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


def by_parts(P, h):
    P.pic_yee_update(h, P.PIC_B_HALF)
    P.pic_gather_push(h)
    P.pic_deposit_current(h)
    P.pic_yee_update(h, P.PIC_B_HALF)
    P.pic_yee_update(h, P.PIC_E_FULL)


def equal(a, b, prec):
    """Both sides do the same operations on each cell; they may be contracted to
    fused multiply-adds differently, which moves a sum of six terms by a few ulps
    of the largest."""
    eps = 2.0 ** -52 if prec == 0 else 2.0 ** -23
    scale = max(float(np.abs(b).max()), 1e-300)
    assert float(np.abs(a.astype(np.float64) - b.astype(np.float64)).max()) <= 16 * eps * scale


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("dims,n", [(2, (11, 13, 1)), (2, (64, 9, 1)), (3, (9, 11, 10)), (3, (33, 10, 12))])
@pytest.mark.parametrize("antenna", [None, (1, 1), (2, 4), (1, 8)])
def test_one_pass_equals_the_two_updates(P, prec, dims, n, antenna):
    wl = W.thermal_plasma("fields", dims, n, 1, 0.1, 1, W.SEED_BASE + 80, dt_courant=0.45)
    rng = np.random.Generator(np.random.PCG64(n[0]))
    grids = []
    for _ in range(2):
        g = P.Grid(P.make_desc(dims, wl.n, wl.d, wl.dt, wl.c, prec, tile=(4, 4, 4), halo=0))
        grids.append(g)
    E = [rng.normal(size=grids[0].shape) for _ in range(3)]
    B = [rng.normal(size=grids[0].shape) for _ in range(3)]
    for g in grids:
        g.set_fields(E, B)
        if antenna:
            P.pic_set_antenna(g.h, 0, antenna[0], antenna[1], 0.5, 1.3, 2.0, 7)
    a, b = grids
    for steps in (1, 2, 3):
        P.pic_step(a.h, steps)              # no particles: the field passes alone
        for _ in range(steps):
            by_parts(P, b.h)
        fa, fb = a.get_fields(), b.get_fields()
        for u, v in zip(fa[0] + fa[1], fb[0] + fb[1]):
            equal(u, v, prec)
        for g in grids:                      # both sides go on from the same numbers
            g.set_fields(fb[0], fb[1])
    for g in grids:
        g.close()


def test_a_batch_of_unequal_runs_and_calls_between_the_steps(P):
    import torch
    st = torch.cuda.Stream()
    sizes = [(31, 24, 1), (24, 40, 1), (57, 25, 1)]
    runs = [W.thermal_plasma("run", 2, n, 4, 0.1, 1, W.SEED_BASE + 81 + k, dt_courant=0.45) for k, n in enumerate(sizes)]

    def build():
        b = P.Batch([P.make_desc(2, wl.n, wl.d, wl.dt, wl.c, P.PIC_FP64, tile=(8, 8, 1), rho_bg=wl.rho_bg, sort_interval=2,
                                 stream=st.cuda_stream) for wl in runs])
        for r, wl in enumerate(runs):
            sp = wl.species[0]
            b.load_run(r, 0, sp.q, sp.m, sp.weight, sp.x, sp.w)
        return b

    a, b = build(), build()
    state = np.empty(P.pic_state_bytes(a.h), np.uint8)
    # odd numbers of steps between a graph replay, a snapshot and its restore
    for steps, graph in ((1, 4), (3, 8), (2, 0)):
        P.pic_step(a.h, steps)
        if graph:
            P.pic_step_graph(a.h, graph)
        P.pic_state_save(a.h, state)
        P.pic_step(a.h, 1)
        P.pic_state_restore(a.h, state)
        P.pic_step_persistent(b.h, steps + graph)
    P.pic_sync(a.h)
    P.pic_sync(b.h)
    for r in range(len(runs)):
        fa, fb = a.get_fields_run(r), b.get_fields_run(r)
        for u, v in zip(fa[0] + fa[1], fb[0] + fb[1]):
            np.testing.assert_allclose(u, v, rtol=0, atol=1e-11 * max(np.abs(v).max(), 1e-300))
        for u, v in zip(a.particles_run(r, 0)[2], b.particles_run(r, 0)[2]):
            np.testing.assert_allclose(u, v, rtol=0, atol=1e-11 * np.abs(v).max())
    a.close()
    b.close()
