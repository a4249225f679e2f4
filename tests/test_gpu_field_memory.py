"""The one-pass end of a step takes no memory of its own: E and B go to the unused
particle pool and come back in the next step.  The memory of a grid, and runs
whose sorts, ends and snapshots fall anywhere between the two."""
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


def used():
    import torch
    torch.cuda.synchronize()
    free, total = torch.cuda.mem_get_info()
    return total - free


@pytest.mark.parametrize("prec", [0, 1])
def test_memory_of_a_grid_is_its_fields_and_sums(P, prec):
    n = (256, 256, 256)

    def build():
        return P.Grid(P.make_desc(3, n, (1.0,) * 3, 0.02, 20.0, prec, tile=(8, 4, 4)))

    build().close()                       # the library's own one-time allocations
    before = used()
    g = build()
    P.pic_step(g.h, 3)
    took = used() - before
    g.close()
    cells = n[0] * n[1] * n[2]
    # E, B, J, the charge and the residual's reference; 32 MiB for small buffers and page rounding
    assert took <= cells * (9 * (8 if prec == 0 else 4) + 16) + (32 << 20)


@pytest.mark.parametrize("dims", [2, 3])
@pytest.mark.parametrize("interval", [1, 2, 3, 5, 10])
@pytest.mark.parametrize("ppc", [1, 4])   # 1: in 2D the pool is smaller than the fields
def test_sorts_ends_and_snapshots_between_the_places(P, dims, interval, ppc):
    import torch
    n = (30, 22, 1) if dims == 2 else (17, 12, 14)
    wl = W.thermal_plasma("places", dims, n, ppc, 0.1, 1, W.SEED_BASE + 84, dt_courant=0.45)
    sp = wl.species[0]
    count = sp.n if ppc > 1 else sp.n // 2
    st = torch.cuda.Stream()
    rng = np.random.Generator(np.random.PCG64(85))
    fields = None

    def build():
        nonlocal fields
        g = P.Grid(P.make_desc(dims, n, wl.d, wl.dt, wl.c, P.PIC_FP64, tile=(8, 8, 1) if dims == 2 else (8, 4, 4),
                               rho_bg=wl.rho_bg, sort_interval=interval, stream=st.cuda_stream))
        if fields is None:
            fields = [[rng.normal(size=g.shape) for _ in range(3)] for _ in range(2)]
        g.set_fields(*fields)
        g.load(0, sp.q, sp.m, sp.weight, sp.x[:, :count], sp.w[:, :count])
        return g

    steps = 11
    a, b, c = build(), build(), build()
    P.pic_step(a.h, steps)
    for _ in range(steps):                # one at a time: every field pass in place
        P.pic_step(b.h, 1)
    states = [torch.empty(P.pic_state_bytes(c.h), dtype=torch.uint8, device="cuda") for _ in range(steps)]
    P.pic_step_saving(c.h, states)
    d = build()
    P.pic_state_restore(d.h, states[6])   # the state after six steps, in the middle of the call
    P.pic_step(d.h, steps - 6)
    for g in (a, b, c, d):
        P.pic_sync(g.h)
    fb = b.get_fields()
    for g in (a, c, d):
        f = g.get_fields()
        # the same operations but for the order of the sums of J: a few roundings per
        # step of fields of unit size
        for u, v in zip(f[0] + f[1], fb[0] + fb[1]):
            assert float(np.abs(u - v).max()) <= steps * 64 * 2.0 ** -52 * float(np.abs(v).max())
        order, ob = np.argsort(g.particles(0)[3]), np.argsort(b.particles(0)[3])
        for u, v in zip(g.particles(0)[2], b.particles(0)[2]):
            assert float(np.abs(u[order] - v[ob]).max()) <= steps * 64 * 2.0 ** -52 * float(np.abs(v).max())
    for g in (a, b, c, d):
        g.close()


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("dims", [2, 3])
def test_memory_of_the_particles(P, prec, dims):
    import torch
    n = (256, 256, 1) if dims == 2 else (64, 64, 64)
    count = 6_000_000
    x = [torch.rand(count, dtype=torch.float64, device="cuda") * n[a] for a in range(3)]
    w = [torch.zeros(count, dtype=torch.float64, device="cuda") for _ in range(3)]
    took = None
    for again in range(2):                # the first time brings the library's one-time allocations
        g = P.Grid(P.make_desc(dims, n, (1.0,) * 3, 0.02, 20.0, prec))
        before = used()
        P.pic_load_particles(g.h, 0, -1.0, 1.0, 1.0, x, w)
        took = used() - before
        g.close()
    es = 8 if prec == 0 else 4
    # two pools of cell, id, offsets and momenta; keys and values twice and a class byte
    # for the sort; the old cell and offsets; 20 MiB for the tables and page rounding
    assert took <= count * (2 * (8 + es * (dims + 3)) + 17 + 4 + es * dims) + (20 << 20)
