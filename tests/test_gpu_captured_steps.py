"""Fields stay in the buffers they were created in: a graph that the caller
captured from a step, or from the step by its parts, replays correctly after
steps in any number outside of it, and a run does not depend, to the last bit,
on how its steps are split into calls."""
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


def start(P, prec, dims, particles, stream, more=None):
    """A grid with fields of unit size, and electrons if asked for."""
    n = (40, 26, 1) if dims == 2 else (21, 18, 16)
    wl = W.thermal_plasma("captured", dims, n, 4, 0.1, 1, W.SEED_BASE + 82, dt_courant=0.45)
    g = P.Grid(P.make_desc(dims, n, wl.d, wl.dt, wl.c, prec, tile=(8, 8, 1) if dims == 2 else (8, 4, 4),
                           rho_bg=wl.rho_bg, sort_interval=1000, stream=stream.cuda_stream))
    rng = np.random.Generator(np.random.PCG64(83))
    g.set_fields(*[[rng.normal(size=g.shape) for _ in range(3)] for _ in range(2)])
    if particles:
        sp = wl.species[0]
        g.load(0, sp.q, sp.m, sp.weight, sp.x, sp.w)
    if more:
        more(g)
    return g


@pytest.mark.parametrize("call", ["step", "two steps", "parts"])
@pytest.mark.parametrize("dims,prec", [(2, 0), (3, 1)])
@pytest.mark.parametrize("particles", [False, True])
def test_a_captured_call_replays_between_other_steps(P, call, dims, prec, particles):
    import torch
    one = {"step": lambda h: P.pic_step(h, 1), "two steps": lambda h: P.pic_step(h, 2), "parts": lambda h: by_parts(P, h)}
    st = torch.cuda.Stream()
    a, b = (start(P, prec, dims, particles, st) for _ in range(2))
    done = 0
    P.pic_step(a.h, 1)
    done += 1
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(st):
        graph.capture_begin(capture_error_mode="thread_local")
        one[call](a.h)
        graph.capture_end()
        for outside in (1, 2, 3):
            P.pic_step(a.h, outside)
            graph.replay()
            done += outside + (2 if call == "two steps" else 1)
    P.pic_sync(a.h)
    P.pic_step(b.h, done)
    P.pic_sync(b.h)
    fa, fb = a.get_fields(), b.get_fields()
    # the same operations on both sides, but for the order of J's sums: a rounding
    # of J of 3 ulps a step, carried through the steps without growth
    tol = done * 8 * (2.0 ** -52 if prec == 0 else 2.0 ** -23)
    for u, v in zip(fa[0] + fa[1], fb[0] + fb[1]):
        assert float(np.abs(u.astype(np.float64) - v).max()) <= tol * float(np.abs(v).max())
    del graph
    a.close()
    b.close()


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("dims", [2, 3])
@pytest.mark.parametrize("extra", ["none", "antenna", "vector potential"])
def test_fields_do_not_depend_on_the_split_into_calls(P, prec, dims, extra):
    import torch
    st = torch.cuda.Stream()

    def more(g):
        if extra == "antenna":
            P.pic_set_antenna(g.h, 0, 2, 5, 0.5, 1.3, 2.0, 7)
        if extra == "vector potential":
            dt = np.float64 if prec == 0 else np.float32
            P.pic_set_vector_potential(g.h, [np.full(g.shape, 0.25 * (c + 1), dtype=dt) for c in range(3)], set_B=False)

    def state(g):
        E, B, _ = g.get_fields()
        A = []
        if extra == "vector potential":
            A = [np.empty_like(E[0]) for _ in range(3)]
            P.pic_get_vector_potential(g.h, A)
        return E + B + A

    want = None
    for split in ([7], [1] * 7, [2, 5], [3, 4], [6, 1]):
        g = start(P, prec, dims, False, st, more)
        for k in split:
            P.pic_step(g.h, k)
        P.pic_sync(g.h)
        got = state(g)
        if want is None:
            want = got
        for u, v in zip(got, want):
            np.testing.assert_array_equal(u, v)
        g.close()
